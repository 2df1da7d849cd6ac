"""Fixed-point sums of factors whose sizes differ by many orders of magnitude.

A result is then bounded by what FP64 sums keep, a multiple of u = 2^-53 of the sum of the magnitudes of its own terms, and not
by the product of the largest factors.  The references are sums in the long double of the host.
"""
import numpy as np
import pytest
import torch

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


# one run of 32 modes (the wider limbs) and past it, one to three runs of 120
@pytest.mark.parametrize("n", [1, 2, 5, 32, 33, 120, 121, 241])
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
