"""The float-float Dslash (two warps per 32 sites) against the FP64 oracle on
ragged site groups and batches and in every operator form.

Tolerance: a multiply-add and an addition err by a few 2^-47 of their operands;
an output is a chain of some 20 of them on partial sums of comparable size, so
2^-42 relative in L2 holds with a wide margin (2e-15 measured) and still tells a
lost low part (2^-24)."""
import numpy as np
import pytest
import torch

from oracle import operator as oop
from paper_1401_6749_gb300 import synth

from .gpu_util import pack, require_gpu, to_dev, unpack

pytestmark = pytest.mark.gpu
KAPPA, MU = 0.16, 0.02


@pytest.mark.parametrize("L,n", [((2, 2, 2, 2), 1), ((6, 4, 2, 10), 3), ((4, 6, 6, 34), 1), ((10, 6, 8, 4), 2),
                                 ((10, 6, 8, 4), 9)])
@pytest.mark.parametrize("kw", [{}, {"dagger": True}, {"mu_zero": True}])
@pytest.mark.parametrize("anti", [True, False])
def test_forms(L, n, kw, anti):
    tl = require_gpu()
    U = synth.gauge_field(L, 5)
    op = tl.Operator(L, KAPPA, MU, to_dev(U), antiperiodic=anti)
    f = pack(tl, L, synth.random_spinor(L, n, 9), tl.FF)
    psi = unpack(tl, L, f, tl.FF, n)
    mu = 0.0 if kw.get("mu_zero") else MU
    ref = oop.apply_M(U, psi, KAPPA, mu, antiperiodic=anti, dagger=bool(kw.get("dagger")))
    out = torch.empty_like(f)
    tl.tm_dslash(op, out, f, n, prec=tl.FF, **kw)
    got = unpack(tl, L, out, tl.FF, n)
    assert np.linalg.norm(got - ref) <= 2.0 ** -42 * np.linalg.norm(ref)
    tl.tm_dslash_g5(op, out, f, n, prec=tl.FF, **kw)
    ref[..., 2:, :] *= -1
    assert np.linalg.norm(unpack(tl, L, out, tl.FF, n) - ref) <= 2.0 ** -42 * np.linalg.norm(ref)


def test_hopping_expansion():
    """No centre term and the inverse twist."""
    tl = require_gpu()
    L, n = (6, 4, 8, 6), 2
    U = synth.gauge_field(L, 6)
    op = tl.Operator(L, KAPPA, MU, to_dev(U))
    psi = synth.random_spinor(L, n, 10)
    out = [tl.empty_field(L, p, n) for p in (tl.FF, tl.F64)]
    for p, o in zip((tl.FF, tl.F64), out):
        tl.tm_hpe_apply(op, o, pack(tl, L, psi, p), n, 3, p)
    a, b = (unpack(tl, L, o, p, n) for p, o in zip((tl.FF, tl.F64), out))
    assert np.linalg.norm(a - b) <= 3 * 2.0 ** -42 * np.linalg.norm(b)
