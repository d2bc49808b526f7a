"""The FP64 Dslash with the fixed-point hopping sum against the FP64 oracle:
ragged site groups and batches, steep and sparse fields, values out of the
fixed point's range, and links that it does not take.

Tolerance, unless a test states its own: an FP64 evaluation of a real component
rounds some 56 times, by at most 2^-53 of the sum of |terms| behind it; 96 terms of
the stencil's largest component at most, so 2^-46 of that, about 1.4e-14, covers
both sides; typical L2 errors are 1e-16.
"""
import numpy as np
import pytest
import torch

from .gpu_util import pack, require_gpu, site_shape, to_dev, unpack
from oracle import operator as oop
from oracle.gamma import GAMMA, ID4
from oracle.lattice import shift
from paper_1401_6749_gb300 import synth

pytestmark = pytest.mark.gpu
KAPPA, MU = 0.16, 0.01


def _apply(tl, op, L, psi, **kw):
    n = psi.shape[0]
    f = pack(tl, L, psi, tl.F64)
    out = torch.empty_like(f)
    tl.tm_dslash(op, out, f, n, prec=tl.F64, **kw)
    return unpack(tl, L, out, tl.F64, n)


def _local_max(psi):
    """Largest component of each site and its eight neighbours, (n, T, Z, Y, X)."""
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2))
    out = m.copy()
    for ax in range(1, 5):
        for s in (1, -1):
            out = np.maximum(out, np.roll(m, s, axis=ax))
    return out


@pytest.mark.parametrize("L,n", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 5), ((6, 4, 2, 10), 3), ((10, 6, 8, 4), 2),
                                 ((4, 6, 6, 34), 1), ((4, 6, 6, 34), 3), ((10, 6, 8, 4), 9)])
@pytest.mark.parametrize("kw", [{}, {"dagger": True}, {"mu_zero": True}])
def test_ragged(L, n, kw):
    tl = require_gpu()
    U = synth.gauge_field(L, 5)
    op = tl.Operator(L, KAPPA, MU, to_dev(U))
    psi = synth.random_spinor(L, n, 9)
    got = _apply(tl, op, L, psi, **kw)
    ref = oop.apply_M(U, psi, KAPPA, 0.0 if kw.get("mu_zero") else MU, dagger=bool(kw.get("dagger")))
    assert np.linalg.norm(got - ref) <= 4e-16 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [2, 14])  # few sites and many: four and two warps per 32 sites
@pytest.mark.parametrize("decades", [3, 30, 250])
def test_steep_fields(decades, n):
    """Neighbouring sites of very unlike size, in and beyond the fixed point's range
    2^-863 .. 2^878."""
    tl = require_gpu()
    L = (6, 4, 4, 8)
    U = synth.gauge_field(L, 6)
    op = tl.Operator(L, KAPPA, MU, to_dev(U))
    rng = np.random.default_rng(3)
    scale = 10.0 ** rng.uniform(-decades, decades, size=(n,) + site_shape(L))
    scale[:, 1, :2] = 0.0  # zero sites among them
    psi = synth.random_spinor(L, n, 11) * scale[..., None, None]
    got = _apply(tl, op, L, psi)
    ref = oop.apply_M(U, psi, KAPPA, MU)
    err = np.abs(got - ref).max(axis=(-1, -2))
    assert np.all(err <= 1.5e-14 * _local_max(psi))


@pytest.mark.parametrize("n", [3, 24])
def test_special_values(n):
    """Infinities and NaN reach the sites that read them and no others."""
    tl = require_gpu()
    L = (4, 4, 4, 8)
    U = synth.gauge_field(L, 7)
    op = tl.Operator(L, KAPPA, MU, to_dev(U))
    psi = synth.random_spinor(L, n, 12)
    clean = _apply(tl, op, L, psi)
    bad = psi.copy()
    bad[1, 2, 1, 0, 3, 1, 2] = np.inf
    bad[2, 0, 3, 3, 3, 0, 0] = np.nan
    got = _apply(tl, op, L, bad)
    touched = ~np.isfinite(_local_max(np.nan_to_num(bad, nan=np.inf, posinf=np.inf)))
    same = (got == clean).all(axis=(-1, -2))
    assert same[~touched].all()
    assert not np.isfinite(got[touched]).all(axis=(-1, -2)).any()


def test_links_out_of_range():
    """Links beyond the fixed point's range take the FP64 arithmetic."""
    tl = require_gpu()
    L = (4, 4, 4, 4)
    U = synth.gauge_field(L, 8)
    U[2, 1, 1, 1, 1] *= 40.0
    op = tl.Operator(L, KAPPA, MU, to_dev(U), recon=18)
    psi = synth.random_spinor(L, 2, 13)
    ref = oop.apply_M(U, psi, KAPPA, MU)
    assert np.linalg.norm(_apply(tl, op, L, psi) - ref) <= 1e-15 * np.linalg.norm(ref)


@pytest.mark.parametrize("kw", [{}, {"dagger": True}, {"mu_zero": True}])
def test_batch_independence(kw):
    """A system alone (four warps per 32 sites) and among enough others for two:
    the same bits."""
    tl = require_gpu()
    L, n = (8, 8, 8, 16), 5
    op = tl.Operator(L, KAPPA, MU, to_dev(synth.gauge_field(L, 21)))
    psi = synth.random_spinor(L, n, 22)
    psi[3] *= 10.0 ** np.random.default_rng(1).uniform(-3, 3, size=site_shape(L))[..., None, None]
    many = _apply(tl, op, L, psi, **kw)
    for j in (0, 3):
        np.testing.assert_array_equal(_apply(tl, op, L, psi[j:j + 1], **kw)[0], many[j])


@pytest.mark.parametrize("mode", ["plain", "mixed"])
def test_solve_batch_independence(mode):
    """The CG updates, residuals and norms too."""
    tl = require_gpu()
    L, n = (8, 8, 8, 16), 5
    op = tl.Operator(L, KAPPA, MU, to_dev(synth.gauge_field(L, 21)))
    m = tl.CG_PLAIN if mode == "plain" else tl.CG_MIXED
    par = tl.cg_params(1e-10, 500, m, prec=tl.F64, inner_prec=tl.F32, schur=True, true_residual=True)

    def solve(first, k):
        eta, x = tl.empty_field(L, tl.F64, k), tl.empty_field(L, tl.F64, k)
        tl.z4_noise(L, eta, tl.F64, 7, first, k)
        _, stats = tl.tm_cg_solve(op, x, eta, k, par)
        return unpack(tl, L, x, tl.F64, k), stats

    many, stats = solve(0, n)
    for j in (0, 4):
        one, s1 = solve(j, 1)
        np.testing.assert_array_equal(one[0], many[j])
        assert s1[0] == stats[j]


def _bound(U, psi, kappa, nu):
    """(S_re, S_im): the sums of |terms| behind each real and imaginary part of M psi.
    In numbers a + j b with j^2 = 1, |x| = |re| + j |im| multiplies and adds just so, and
    such numbers are pairs (a + b, a - b) that multiply entry by entry."""
    def split(z):
        return np.stack([np.abs(z.real) + np.abs(z.imag), np.abs(z.real) - np.abs(z.imag)])

    u, p, g = split(U), split(psi), split(GAMMA)
    one = split(ID4 + 0j)
    out = p + split(np.array(1j * nu)).reshape(2, *[1] * psi.ndim) * p
    for m in range(4):
        spin = one + g[:, m]
        for step in (1, -1):
            f = np.abs(shift(psi.real, m, step, False)) + 1j * np.abs(shift(psi.imag, m, step, False))
            link = U[m] if step > 0 else np.swapaxes(shift(U[m], m, -1), -1, -2)
            w = np.einsum("k...ab,kn...sb->kn...sa", split(link), split(f))
            out = out + kappa * np.einsum("kst,kn...tc->kn...sc", spin, w)
    return (out[0] + out[1]) / 2, (out[0] - out[1]) / 2


def _diagonal(L, seed):
    """Links that do not mix colours: diagonal phases."""
    ph = np.exp(1j * np.random.default_rng(seed).uniform(0, 2 * np.pi, size=(4,) + site_shape(L) + (3,)))
    U = np.zeros((4,) + site_shape(L) + (3, 3), dtype=np.complex128)
    U[..., range(3), range(3)] = ph
    return U


@pytest.mark.parametrize("n", [1, 24])  # four and two warps per 32 sites
@pytest.mark.parametrize("links", ["unit", "diagonal", "near unit", "random"])
@pytest.mark.parametrize("field", ["gaussian", "colours", "one colour", "spins", "real", "sites", "point"])
def test_componentwise(links, field, n):
    """Every real component has the accuracy of FP64 arithmetic, 56 roundings of
    2^-53 on the terms that it sums (the oracle in extended precision), also where these are far below the largest
    component of the stencil."""
    tl = require_gpu()
    L = (4, 4, 6, 8)
    U = {"unit": synth.unit_gauge, "diagonal": lambda l: _diagonal(l, 4),
         "near unit": lambda l: synth.gauge_field(l, 4, eps=1e-6),
         "random": lambda l: synth.gauge_field(l, 4, eps=2.0)}[links](L)
    op = tl.Operator(L, KAPPA, MU, to_dev(U), recon=18)
    psi = synth.random_spinor(L, n, 5)
    if field == "colours":
        psi *= np.array([1.0, 1e-8, 1e-16])
    elif field == "one colour":
        psi *= np.array([0.0, 1.0, 0.0])
    elif field == "spins":
        psi *= np.array([1.0, 1e-9, 1e-3, 1e-14])[:, None]
    elif field == "real":
        psi = psi.real + 1e-12j * psi.imag
    elif field == "sites":
        psi *= 10.0 ** np.random.default_rng(6).uniform(-20, 20, size=(n,) + site_shape(L))[..., None, None]
    elif field == "point":
        psi = np.zeros_like(psi)
        psi[:, 1, 2, 1, 3, 2, 1] = 1.0
    for kw in ({}, {"dagger": True}):
        got = _apply(tl, op, L, psi, **kw)
        some = [0, n - 1] if n > 1 else [0]
        got = got[some]
        ref = oop.apply_M(U.astype(np.clongdouble), psi[some], KAPPA, MU, dagger=bool(kw))
        sre, sim = _bound(U, psi[some], KAPPA, 2 * KAPPA * MU)
        assert np.all(np.abs(got.real - ref.real) <= 56 * 2.0 ** -53 * sre)
        assert np.all(np.abs(got.imag - ref.imag) <= 56 * 2.0 ** -53 * sim)
