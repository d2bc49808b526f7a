"""Momentum-projected local loops, all momenta of a pass in one kernel: at the
edges of the momentum groups (4, 8, ..., 32 per pass) and of the site tiles (128)
and chunks (128 to 1024), against the FP64 oracle.

Tolerance: an output sums 4 phased bilinears per site.  In FP32 a bilinear of
three complex products errs by at most 7 u sum_c |L||R|, its phase by 4 u, a sum of
eight sites by 8 u (longer sums are compensated), u = 2^-24: 24 u of
sum |L||R| covers it, and 24 2^-46 the float-float arithmetic, whose steps err by
a few 2^-47."""
import numpy as np
import pytest
import torch

from oracle import loops as olo
from oracle.gamma import gamma_basis
from paper_1401_6749_gb300 import synth

from .gpu_util import from_dev, pack, require_gpu, unpack

pytestmark = pytest.mark.gpu
U = {"f16": 2.0 ** -24, "bf16": 2.0 ** -24, "f32": 2.0 ** -24, "ff": 2.0 ** -46, "f64": 2.0 ** -50}


def _momenta(n):
    rng = np.random.default_rng(n)
    return np.concatenate([[[0, 0, 0]], rng.integers(-9, 10, size=(n - 1, 3))])


def _check(L, n, nmom, prec, mode, mom=None):
    tl = require_gpu()
    p = tl.PREC[prec]
    fl, fr = (pack(tl, L, synth.random_spinor(L, n, s), p) for s in (4, 5))
    left, right = (unpack(tl, L, f, p, n) for f in (fl, fr))  # the stored values
    mom = _momenta(nmom) if mom is None else mom
    out = torch.full((n, nmom, 16, L[3], 2), float("nan"), dtype=torch.float64, device="cuda")
    tl.loop_contract_local_mom(L, fl, fr, p, n, tl.LOOP_MODE[mode], mom, out)
    got = from_dev(out, (n, nmom, 16, L[3]))
    ref = olo.local_loops_mom(left, right, mode, mom)
    size = np.einsum("ntzyxac,ntzyxbc->nt", np.abs(left), np.abs(right))[:, None, None, :]
    assert np.all(np.abs(got - ref) <= 24 * U[prec] * size)


@pytest.mark.parametrize("nmom", [1, 4, 5, 8, 12, 13, 20, 21, 28, 29, 32, 33, 64])
@pytest.mark.parametrize("L", [(6, 4, 8, 4), (4, 4, 4, 40)])  # groups side by side (few blocks), and one after the other
def test_momentum_groups(nmom, L):
    _check(L, 2, nmom, "f32", "vv")


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (8, 8, 4, 2), (10, 6, 10, 4), (16, 12, 12, 2), (16, 16, 10, 4)])
@pytest.mark.parametrize("prec", ["f16", "bf16", "f32", "ff", "f64"])
def test_site_tiles(L, prec):
    _check(L, 1, 7, prec, "std")


@pytest.mark.parametrize("prec", ["ff", "f64"])
def test_wide_full_pass(prec):
    _check((6, 4, 8, 4), 1, 32, prec, "gen")
    _check((4, 4, 4, 40), 2, 32, prec, "gen")


@pytest.mark.parametrize("p", [(0, 0, 0), (3, -1, 2)])
@pytest.mark.parametrize("prec", ["f16", "f32", "ff", "f64"])
def test_single_momentum(p, prec):
    _check((8, 6, 4, 6), 2, 1, prec, "vv", np.array([p]))


@pytest.mark.parametrize("prec", ["f16", "f32", "ff", "f64"])
@pytest.mark.parametrize("L", [(8, 6, 4, 6), (16, 12, 12, 2), (10, 10, 14, 2), (4, 4, 4, 40)])
def test_list_independence(L, prec):
    """A momentum alone and in a list: the same bits."""
    tl = require_gpu()
    p, n = tl.PREC[prec], 2
    fl, fr = (pack(tl, L, synth.random_spinor(L, n, s), p) for s in (4, 5))

    def loops(mom):
        out = torch.full((n, len(mom), 16, L[3], 2), float("nan"), dtype=torch.float64, device="cuda")
        tl.loop_contract_local_mom(L, fl, fr, p, n, tl.LOOP_MODE["vv"], mom, out)
        return out

    mom = _momenta(34)
    many = loops(mom)
    for k in (0, 1, 32, 33):
        assert torch.equal(loops(mom[k:k + 1])[:, 0], many[:, k])
    assert torch.equal(loops(mom[:5]), many[:, :5])


@pytest.mark.parametrize("nmom", [1, 4, 19, 32, 33])
def test_trace_bytes(nmom):
    """The record charges both fields once per pass of at most 32 momenta, and a
    small part more for the phases; not once per momentum."""
    tl = require_gpu()
    L, n = (16, 16, 16, 32), 3  # enough blocks for one group
    fields = 2 * n * 24 * 4 * int(np.prod(L))
    fl, fr = (pack(tl, L, synth.random_spinor(L, n, s), tl.F32) for s in (4, 5))
    out = torch.empty((n, nmom, 16, L[3], 2), dtype=torch.float64, device="cuda")
    tl.tm_trace_reset()
    tl.tm_trace_enable(True)
    try:
        tl.loop_contract_local_mom(L, fl, fr, tl.F32, n, tl.LOOP_MODE["vv"], _momenta(nmom), out)
        launches, _, nbytes = tl.tm_trace_read("localmom.f32")
    finally:
        tl.tm_trace_enable(False)
        tl.tm_trace_reset()
    passes = (nmom + 31) // 32
    assert launches == 1
    assert passes * fields <= nbytes <= 1.2 * passes * fields


def test_float_float_accuracy():
    """The sums over sites add little to the rounding of the bilinears: 3.5e-15 in L2
    (3.0e-15 at zero momentum) against extended precision, where float-float sums
    without compensation of their low parts give 6.6e-15; 2^-47.5 lies between."""
    tl = require_gpu()
    L, n = (8, 8, 8, 16), 2
    fl, fr = (pack(tl, L, synth.random_spinor(L, n, s), tl.FF) for s in (14, 15))
    left, right = (unpack(tl, L, f, tl.FF, n).astype(np.clongdouble) for f in (fl, fr))
    mom = np.array([[0, 0, 0], [1, 0, 0], [1, 2, -1], [2, 1, 1], [0, 1, 2]])
    out = torch.empty((n, len(mom), 16, L[3], 2), dtype=torch.float64, device="cuda")
    tl.loop_contract_local_mom(L, fl, fr, tl.FF, n, tl.LOOP_MODE["std"], mom, out)
    got = from_dev(out, (n, len(mom), 16, L[3]))
    m = np.einsum("ntzyxac,ntzyxbc->ntzyxab", left.conj(), right)
    pi = 4 * np.arctan(np.longdouble(1))
    gammas = gamma_basis().astype(np.clongdouble)
    for q, p in enumerate(mom):
        ph = [np.exp(-2j * pi * ((p[k] * np.arange(L[k])) % L[k]).astype(np.longdouble) / L[k]) for k in range(3)]
        w = ph[2][:, None, None] * ph[1][None, :, None] * ph[0][None, None, :]
        ref = np.einsum("gab,ntab->ngt", gammas, np.einsum("zyx,ntzyxab->ntab", w, m))
        assert np.linalg.norm((got[:, q] - ref).ravel()) <= 2.0 ** -47.5 * np.linalg.norm(ref.ravel())
