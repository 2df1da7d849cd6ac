"""Fixed-point sums of factors whose sizes differ by many orders of magnitude.

A result is then bounded by what FP64 sums keep, a multiple of u = 2^-53 of the sum of the magnitudes of its own terms, and not
by the product of the largest factors.  The references are sums in the long double of the host.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1612_06424_gb300 import inputs

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


def _lq():
    from paper_1612_06424_gb300 import build, lqcd

    build.build()
    return lqcd


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rng(*seed):
    r = np.random.default_rng(seed)
    return r, lambda *s: r.standard_normal(s) + 1j * r.standard_normal(s)


def _long(a):
    return a.astype(np.clongdouble)


# up to 15 and up to 60 modes (wider limbs), one to three runs of 120
@pytest.mark.parametrize("n", [1, 2, 5, 15, 16, 32, 33, 60, 61, 120, 121, 122, 241])
@pytest.mark.parametrize("scales", ["reciprocal", "columns", "modes", "all", "zeros"])
def test_projected_propagator_keeps_small_terms(n, scales):
    """Two entries, each rounded at 2^-54 of its scale, times the other below twice its scale, and the low parts' product: at
    most 4 u of the product of the scales a term, which may lie four times above the largest term (eight with
    the wider limbs): 16 n u."""
    lqcd = _lq()
    # 192 sums, or (one thread each) more than a wave of blocks
    dims, x = ((4, 2, 2, 2), (0, 1, 0, 1)) if n % 2 else ((4, 12, 12, 12), (0, 1, 0, 1))
    S = 2 * int(np.prod(dims[1:]))
    lat = lqcd.Lattice(dims, "open")
    r, c = _rng(21, n)
    xi, eta = c(n, S, 4, 3), c(n, S, 4, 3)
    if scales in ("reciprocal", "all"):
        f = 10.0 ** r.uniform(-9, 9, (n, 1, 1, 1))
        xi, eta = xi * f, eta / f
    if scales in ("columns", "all"):
        xi, eta = xi * 10.0 ** r.uniform(-8, 8, (1, 1, 4, 3)), eta * 10.0 ** r.uniform(-8, 8, (1, S, 4, 3))
    if scales in ("modes", "all"):
        xi, eta = xi * 10.0 ** r.uniform(-20, 20, (n, 1, 4, 3)), eta * 10.0 ** r.uniform(-20, 20, (n, S, 1, 1))
    if scales == "zeros":
        xi[::2, :, 1], xi[n // 2], eta[:, 3], eta[n // 3, :, :, 2] = 0, 0, 0, 0
        xi[:, :, 3, 1] = 0
    got = lat.projected_propagator(_cuda(xi), _cuda(eta), (0, 1), (2, 3), x).cpu().numpy()[:, S:].reshape(12, S, 12)
    y = slice(None, None, 1 if S < 100 else 31)
    got, e, s = got[:, y], _long(eta.reshape(n, S, 12)[:, y]), _long(xi[:, np.ravel_multi_index(x, dims)].reshape(n, 12))
    ref, M = -np.einsum("nya,nb->bya", e, s.conj()), np.einsum("nya,nb->bya", abs(e), abs(s))
    assert np.all(np.abs(got - ref) <= 16 * n * U64 * M)
    lat.close()


def _nucleon_point(p, T, real):
    """oracle.nucleon_point_correlator in long double, or (real) with every factor of every term replaced by its magnitude."""
    e, cg5 = oracle.EPS3, oracle.charge_conjugation() @ oracle.gamma(4)
    m = oracle.gamma(4) @ (0.5 * (np.eye(4) - oracle.gamma(0)))
    P = _long(p).reshape(4, 3, -1, 4, 3).transpose(2, 3, 4, 0, 1)
    if real:
        e, cg5, m, P = abs(e), abs(cg5), abs(m), abs(P)
    words = ("abc,ABC,mn,MN,gd,ymaNB,ynbMA,ydcgC->", "abc,ABC,mn,MN,gd,ymaNB,ynbgC,ydcMA->")
    return np.array([[np.einsum(w, e, e, cg5, cg5, m, Pt, Pt, Pt, optimize="optimal") for w in words]
                     for Pt in np.split(P, T)])


# slices of 8 (half a stage) and 80 sites
@pytest.mark.parametrize("dims", [(3, 2, 2, 2), (2, 4, 2, 10)])
@pytest.mark.parametrize("scales", ["plain", "colours", "spins", "entries", "sites", "cancelling", "diagonal", "zeros"])
def test_nucleon_point_keeps_small_terms(dims, scales):
    """Sites summed in fixed point have a term of at least 2^-6 of the product of the scales, whose error of 0.7 u is then 45 u of
    that term, with 4 standard deviations 180 u; FP64 sums of a few thousand terms keep less: 256 u of the sum of the terms."""
    lqcd = _lq()
    lat = lqcd.Lattice((4,) + dims[1:], "open")
    r, c = _rng(22, *dims)
    V, T = int(np.prod(dims)), dims[0]
    p = c(12, V, 4, 3)
    ten = lambda w, *s: 10.0 ** r.uniform(-w, w, s)  # noqa: E731
    if scales == "colours":
        p = p * np.tile([1e6, 1, 1e-6], 4).reshape(12, 1, 1, 1) * np.array([1e-5, 1, 1e5]) * ten(30, 1, V, 1, 1)
    if scales == "spins":
        p = p * np.repeat([1e8, 1e-8, 1e8, 1e-8], 3).reshape(12, 1, 1, 1) * np.array([1e-4, 1e4, 1, 1]).reshape(4, 1)
    if scales == "entries":
        p = p * ten(8, 12, V, 4, 3)
    if scales == "sites":
        p = p * ten(90, 1, V, 1, 1)
    if scales == "cancelling":
        p[:, :, 2:] = -p[:, :, :2] * (1 + 1e-9)
    if scales == "diagonal":
        p = p * (1e-12 + ((np.arange(12) % 3)[:, None, None, None] == np.arange(3)))
    if scales == "zeros":
        p[:, 1], p[3], p[:, 2:4, 1] = 0, 0, 0
        p[6:, 4] = 0
        p[np.arange(12) % 3 == 1, 5] = 0
    full = np.zeros((12, lat.V, 4, 3), complex)
    full[:, :V] = p
    got = lat.nucleon_point(_cuda(full), 0, T).cpu().numpy()[0]
    assert np.all(np.abs(got - _nucleon_point(p, T, False)) <= 256 * U64 * _nucleon_point(p, T, True))
    lat.close()


# tiles of 8 columns, runs of 32 coefficients
@pytest.mark.parametrize("n", [1, 8, 9, 33])
def test_orthonormal_columns_keep_small_rows(n):
    """Every row of the result is off by n u times the condition number (below 10) of its own size: 1e-13 sqrt(n) of the row's largest
    entry relative to the columns' norms."""
    lqcd = _lq()
    dims = (4, 4, 6, 6)
    lat = lqcd.Lattice(dims, "open")
    lat.set_gauge(inputs.unit_field(dims), 0.12, 0.0)
    r, c = _rng(23, n)
    S3 = int(np.prod(dims[1:]))
    v = c(n, 3 * S3, 4, 3) * 10.0 ** r.uniform(-4, 4, (n, 1, 1, 1)) * 10.0 ** np.minimum(r.uniform(-12, 8, (3 * S3, 4, 3)), 0)
    v[:, :, 2:] = 0
    phi, _ = lat.boundary_modes(_cuda(v), (0, 2), 1, 0, 0, lqcd.SolverParams(tol=1e-12, precision=64))
    A = _long(v[:, S3:2 * S3, :2].reshape(n, -1).T) / 2  # its negative below
    G = 2 * A.conj().T @ A
    s = np.sqrt(np.diag(G).real)
    L = np.zeros((n, n), np.clongdouble)  # G = L L^dag, W = A L^-dag column by column
    W = np.zeros_like(A)
    for k in range(n):
        L[k, k] = np.sqrt(G[k, k] - (abs(L[k, :k]) ** 2).sum())
        L[k + 1:, k] = (G[k + 1:, k] - L[k + 1:, :k] @ L[k, :k].conj()) / L[k, k]
        W[:, k] = (A[:, k] - W[:, :k] @ L[k, :k].conj()) / L[k, k]
    got = phi.cpu().numpy().reshape(n, S3, 2, 2, 3)
    for sign, half in ((1, got[:, :, 0]), (-1, got[:, :, 1])):
        err = np.abs(sign * half.reshape(n, -1).T - W)
        assert np.all(err.max(1) <= 1e-13 * n ** 0.5 * np.abs(A / s).max(1))
    lat.close()


@pytest.mark.parametrize("csw", [0.0, 1.0])
def test_operator_below_the_normal_range(csw):
    """Inputs of 20 bits, scaled by 2^-1040 without rounding: the result is that of the unscaled input, rounded once more."""
    lqcd = _lq()
    dims = (4, 2, 4, 2)
    lat = lqcd.Lattice(dims, "open")
    lat.set_gauge(inputs.random_su3_field(dims, 0.4, 3), 0.13, csw)
    _, c = _rng(24)
    z = np.round(c(lat.V, 4, 3).view(float) * 2 ** 17) / 2 ** 20
    want = lat.dslash(_cuda(z.view(complex)), 0, None, False, 64).cpu().numpy().view(float)
    got = lat.dslash(_cuda(np.ldexp(z, -1040).view(complex)), 0, None, False, 64).cpu().numpy().view(float)
    assert np.all(np.abs(got - np.ldexp(want, -1040)) <= 2.0 ** -1074) and np.abs(got).max() > 0
    lat.close()


def test_sums_below_the_normal_range():
    """Products near 2^-1050 of numbers of 20 bits: half a unit of the last place for each addition of FP64 numbers there."""
    lqcd = _lq()
    dims, x, n = (4, 2, 2, 2), (0, 1, 0, 1), 5
    lat = lqcd.Lattice(dims, "open")
    _, c = _rng(25)
    xi, eta = (np.round(c(n, 16, 4, 3).view(float) * 2 ** 17).view(complex) / 2 ** 20 for _ in range(2))
    sums = lambda k: lat.projected_propagator(_cuda(xi * 2.0 ** k), _cuda(eta * 2.0 ** k), (0, 1), (2, 3), x)  # noqa: E731
    got, want = (sums(k).cpu().numpy()[:, 16:].copy().view(float) for k in (-525, 0))
    assert np.all(np.abs(got - np.ldexp(want, -1050)) <= 2 * n * 2.0 ** -1074) and np.abs(got).max() > 0
    p = np.round(c(12, lat.V, 4, 3).view(float) * 2 ** 17).view(complex) / 2 ** 20
    got, want = (lat.nucleon_point(_cuda(p * 2.0 ** k)).cpu().numpy().view(float) for k in (-350, 0))
    assert np.all(np.abs(got - np.ldexp(want, -1050)) <= 8 * 4608 * 2.0 ** -1074) and np.abs(got).max() > 2.0 ** -1055
    lat.close()
