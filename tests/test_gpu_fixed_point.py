"""The kernels that compute FP64-accurate sums in 64-bit integers, and the tile edges of the contractions.

Bounds, with u = 2^-53 the rounding of FP64 and M the largest magnitude that enters a sum:
  stencil: 8 hops x 3 complex products and 6 of the diagonal block, each entry rounded at 2^-57 M or better and each
    product cut at 2^-57 M, one rounding of a result below 10 M, and as many FP64 roundings in the oracle: 60 x 10 u M,
    taken as 1e-13 M with M the largest component of the site and its neighbours;
  sums of n products: n (2^-53 + 2^-53) M_a M_b for the kernel and the reference, taken as 4 n u M_a M_b x sqrt(2);
  orthonormal columns: the two passes leave n u times the condition number (below 10 for the columns here), 1e-13.
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


BCS = {"open": oracle.BC_OPEN, "periodic": oracle.BC_PERIODIC, "antiperiodic": oracle.BC_ANTIPERIODIC}


# 16 to 160 sites a parity: below, at and past the 64 sites of a block; slabs of one slice to all
@pytest.mark.parametrize("dims,dom", [((2, 2, 2, 4), None), ((4, 4, 4, 2), (3, 3)), ((4, 2, 8, 4), None),
                                      ((10, 2, 4, 4), (1, 8)), ((6, 4, 2, 6), (0, 2))])
@pytest.mark.parametrize("bc,csw,dag", [("open", 1.0, False), ("periodic", 0.0, True), ("antiperiodic", 1.0, True),
                                        ("antiperiodic", 0.0, False)])
def test_stencil_over_a_wide_range(dims, dom, bc, csw, dag):
    """Sites of very different size, and components of very different size within a site."""
    lqcd = _lq()
    U = inputs.random_su3_field(dims, 0.4, 3)
    lat = lqcd.Lattice(dims, bc)
    lat.set_gauge(U, 0.13, csw)
    op = oracle.Operator(dims, U, 0.13, csw, BCS[bc])
    r, c = _rng(5, *dims)
    V, (t0, t1) = int(np.prod(dims)), dom or (0, dims[0] - 1)
    sl = inputs.slab_sites(dims, t0, t1)
    psi = op.masked(c(V, 4, 3) * 10.0 ** r.uniform(-9, 9, (V, 1, 1)) * 10.0 ** r.uniform(-6, 0, (V, 4, 3)), t0, t1)
    got = lat.dslash(_cuda(psi[sl]), 0, dom, dag, 64)
    ref = op.apply(psi, t0, t1, dagger=dag)[sl]
    m = np.abs(psi).max((1, 2)).reshape(dims)
    M = np.max([m] + [np.roll(m, s, a) for a in range(4) for s in (1, -1)], 0).reshape(-1)[sl]
    assert np.all(np.abs(got.cpu().numpy() - ref).max((1, 2)) <= 1e-13 * M)
    # powers of two come out exactly, a zero vector is zero
    for k in (-600, 600):
        assert torch.equal(lat.dslash(_cuda(psi[sl] * 2.0 ** k), 0, dom, dag, 64), got * 2.0 ** k)
    assert not lat.dslash(_cuda(0 * psi[sl]), 0, dom, dag, 64).any()
    # a non-finite component reaches the neighbours and nothing else
    bad = psi[sl].copy()
    site = bad.shape[0] // 2
    bad[site, 1, 2] = np.inf
    out = lat.dslash(_cuda(bad), 0, dom, dag, 64).cpu().numpy()
    probe = np.zeros((V, 4, 3), complex)
    probe[sl][site, 1, 2] = 1
    hit = np.abs(op.apply(probe, t0, t1, dagger=dag)[sl]).max((1, 2)) > 0
    assert hit[site] and not np.isfinite(out[hit]).all((1, 2)).any()
    assert np.array_equal(out[~hit], got.cpu().numpy()[~hit])
    lat.close()


# det(U) - 1 is 3 x of a scaled link and 3 i x of a turned one, U U^dag - 1 2 x and 0: 1e-10 lies between 3e-11 and 4e-11
@pytest.mark.parametrize("change,good", [(lambda u: u * (1 + 3e-11), True), (lambda u: u * (1 - 4e-11), False),
                                         (lambda u: u * np.exp(-3e-11j), True), (lambda u: u * np.exp(4e-11j), False),
                                         (lambda u: u[[1, 0, 2]], False), (lambda u: 2 * u, False),
                                         (lambda u: 1e-200 * u, False), (lambda u: 1e200 * u, False),
                                         (lambda u: u * np.inf, False), (lambda u: u * np.nan, False)])
def test_links_are_checked(change, good):
    lqcd = _lq()
    dims = (2, 2, 2, 4)
    U = inputs.random_su3_field(dims, 0.4, 3).reshape(-1, 4, 3, 3).copy()
    with np.errstate(invalid="ignore"):
        U[17, 2] = change(U[17, 2])
    lat = lqcd.Lattice(dims, "open")
    if good:
        lat.set_gauge(U, 0.13, 1.0)
    else:
        with pytest.raises(lqcd.LQCDError, match="not SU"):
            lat.set_gauge(U, 0.13, 1.0)
    lat.close()


# 16 to 160 sites a parity against blocks of 128, slabs of one slice to all, every warp's slots of the ring
@pytest.mark.parametrize("dims,dom", [((2, 2, 2, 4), None), ((4, 4, 4, 2), (3, 3)), ((4, 4, 4, 4), None),
                                      ((10, 2, 4, 4), (1, 8)), ((6, 4, 2, 6), (0, 2))])
@pytest.mark.parametrize("bc,csw,dag", [("open", 1.0, False), ("periodic", 0.0, True), ("antiperiodic", 1.0, True)])
def test_fp32_stencil_edges(dims, dom, bc, csw, dag):
    """2e-6 of the largest entry: 80 FP32 roundings of 6e-8 of terms below it, as for the larger lattice of the parity
    tests."""
    lqcd = _lq()
    U = inputs.random_su3_field(dims, 0.4, 3)
    lat = lqcd.Lattice(dims, bc)
    lat.set_gauge(U, 0.13, csw)
    op = oracle.Operator(dims, U, 0.13, csw, BCS[bc])
    t0, t1 = dom or (0, dims[0] - 1)
    sl = inputs.slab_sites(dims, t0, t1)
    psi = op.masked(inputs.gaussian_spinor(dims, 4)[0], t0, t1)
    ref = op.apply(psi, t0, t1, dagger=dag)[sl]
    got = lat.dslash(_cuda(psi[sl]), 0, dom, dag, 32).cpu().numpy()
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    lat.close()


@pytest.mark.parametrize("n", [1, 4, 119, 120, 121, 241])
def test_projected_propagator_sums(n):
    """One to three runs of 120 modes, whose sizes differ by twelve orders of magnitude."""
    lqcd = _lq()
    dims, x = (4, 2, 2, 2), (0, 1, 0, 1)
    lat = lqcd.Lattice(dims, "open")
    r, c = _rng(6, n)
    f = 10.0 ** r.uniform(-6, 6, (n, 1, 1, 1))
    xi, eta = c(n, 16, 4, 3) * f, c(n, 16, 4, 3) / f
    got = lat.projected_propagator(_cuda(xi), _cuda(eta), (0, 1), (2, 3), x).cpu().numpy()
    xs = xi[:, 5].reshape(n, 12)
    ref = -np.einsum("nya,nb->bya", eta.reshape(n, 16, 12), xs.conj()).reshape(12, 16, 4, 3)
    M = np.einsum("ya,b->bya", np.abs(eta.reshape(n, 16, 12)).max(0), np.abs(xs).max(0)).reshape(ref.shape)
    assert np.all(np.abs(got[:, 16:] - ref) <= 4 * 2 ** 0.5 * n * U64 * M) and not got[:, :16].any()
    eta[n // 2, 3, 1, 2] = np.nan
    bad = np.isnan(lat.projected_propagator(_cuda(xi), _cuda(eta), (0, 1), (2, 3), x).cpu().numpy())
    assert bad[:, 19, 1, 2].all() and bad.sum() == 12
    lat.close()


@pytest.mark.parametrize("n,dims", [(1, (4, 2, 2, 2)), (7, (4, 2, 2, 2)), (8, (4, 2, 2, 6)), (9, (4, 6, 6, 4)),
                                    (33, (4, 4, 4, 4)), (65, (4, 4, 6, 6))])
def test_orthonormal_columns(n, dims):
    """Column tiles of 8 and runs of 32 coefficients, one row chunk and several; the columns' sizes differ."""
    lqcd = _lq()
    lat = lqcd.Lattice(dims, "open")
    lat.set_gauge(inputs.unit_field(dims), 0.12, 0.0)
    r, c = _rng(7, n)
    S3 = int(np.prod(dims[1:]))
    v = c(n, 3 * S3, 4, 3) * 10.0 ** r.uniform(-4, 4, (n, 1, 1, 1))
    phi, _ = lat.boundary_modes(_cuda(v), (0, 2), 1, 0, 0, lqcd.SolverParams(tol=1e-12, precision=64))
    phi = phi.cpu().numpy().reshape(n, -1)
    s = v[:, S3:2 * S3]
    up = (s[:, :, :2] - s[:, :, 2:]) / 2
    q, R = np.linalg.qr(np.concatenate([up, -up], 2).reshape(n, -1).T)
    q = (q * (np.diag(R) / np.abs(np.diag(R)))).T
    assert np.abs(phi.conj() @ phi.T - np.eye(n)).max() <= 1e-13
    assert np.abs(phi - q).max() <= 1e-13
    lat.close()


@pytest.mark.parametrize("dims,t0,nt,n", [((4, 2, 2, 2), 0, 4, 1), ((2, 2, 2, 6), 1, 1, 3), ((4, 4, 2, 10), 1, 2, 2)])
def test_nucleon_point_sums(dims, t0, nt, n):
    """Slices of 8 to 80 sites, and propagators whose columns, sites and spins differ in size."""
    lqcd = _lq()
    lat = lqcd.Lattice(dims, "open")
    r, c = _rng(8, *dims)
    V = int(np.prod(dims))
    p = c(n, 12, V, 4, 3) * 10.0 ** (r.uniform(-2, 2, (n, 12, 1, 1, 1)) + r.uniform(-2, 2, (n, 1, V, 4, 3)))
    W = lat.nucleon_point(_cuda(p), t0, nt).cpu().numpy()
    for k in range(n):
        ref = oracle.nucleon_point_correlator(p[k], dims[0])[t0:t0 + nt]
        # each term is a product of three entries: 2 x 36 x 64 of them a site
        m = np.abs(p[k]).max((0, 2, 3)).reshape(dims[0], -1)[t0:t0 + nt]
        assert np.all(np.abs(W[k] - ref).max(1) <= 4608 * 8 * U64 * (m ** 3).sum(1))
    p[0, 2, t0 * (V // dims[0]), 3, 1] = np.inf
    W = lat.nucleon_point(_cuda(p), t0, nt).cpu().numpy()
    assert not np.isfinite(W[0, 0]).any() and np.isfinite(W.reshape(n * nt, 2)[1:]).all()
    lat.close()


@pytest.mark.parametrize("n,nx,ny", [(1, 1, 1), (2, 3, 2), (15, 1, 2), (16, 2, 1), (17, 2, 3), (33, 1, 1)])
def test_contraction_tiles(n, nx, ny):
    lqcd = _lq()
    _, c = _rng(9, n)
    bx, by = c(nx, n, n, n, 4), c(ny, n, n, n, 4)
    W = lqcd.nucleon_contract(_cuda(bx), _cuda(by)).cpu().numpy()
    z = np.einsum("gd,yijkd->yijkg", oracle.gamma(4) @ (0.5 * (np.eye(4) - oracle.gamma(0))), by)
    for q, axes in enumerate("jik kij".split()):
        ref = -np.einsum("x%sg,yijkg->xy" % axes, bx, z)
        M = np.einsum("x%sg,yijkg->xy" % axes, np.abs(bx), np.abs(z))
        assert np.all(np.abs(W[:, :, q] - ref) <= 4 * 2 ** 0.5 * 8 * n * U64 * M)


@pytest.mark.parametrize("count", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("n", [1, 3])
def test_level_mean_counts(count, n):
    lqcd = _lq()
    _, c = _rng(10, count)
    b = c(count, 1, n, n, n, 4)
    b[-1, 0, 0, 0, 0, 0] = np.inf
    m = lqcd.level_mean(_cuda(b)).cpu().numpy()
    ok = np.isfinite(b).all(0)
    assert np.abs(m - b.mean(0))[ok].max() <= 2 * (count + 1) * U64 * np.abs(b[np.isfinite(b)]).max()
    assert np.isinf(m[~ok].real).all()


# 8 sites are 2 chunks of the pipeline, 64 one whole group of 16, 72 and 136 one and two groups and two chunks
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 4, 4), (2, 6, 6, 2), (2, 2, 2, 34)])
@pytest.mark.parametrize("n", [3, 33])
def test_tensor_core_block_groups(dims, n, monkeypatch):
    """The tensor-core kernel against the FMA kernel: 6e-5 of the sum of the magnitudes of the terms (as in the
    kernels' other tests), here of M^3 a term, 6 x 4 terms a site."""
    lqcd = _lq()
    lat = lqcd.Lattice(dims, "open")
    _, c = _rng(11, n)
    V = int(np.prod(dims))
    s = _cuda(c(n, V, 4, 3))
    got = []
    for kernel in "10":
        monkeypatch.setenv("LQCD_NUCLEON_TC", kernel)
        got.append(lat.nucleon_blocks(s, (0, 1), 0, 2).cpu().numpy())
    r = np.sqrt((np.abs(s.cpu().numpy()) ** 2).mean((1, 2, 3))).max()
    assert np.abs(got[0] - got[1]).max() <= 6e-5 * 24 * (V // 2) * r ** 3
    assert np.abs(got[1]).max() > 1e-2 * (V // 2) ** 0.5 * r ** 3
    lat.close()


# the force's neighbourhood at the ends of the lattice, across a wrap and on one slice
@pytest.mark.parametrize("dims,bc,dom", [((4, 2, 2, 2), "open", (0, 0)), ((4, 4, 2, 2), "open", (3, 3)),
                                         ((4, 2, 4, 2), "periodic", (3, 3)), ((6, 2, 2, 4), "antiperiodic", (0, 1)),
                                         ((6, 2, 2, 2), "open", (2, 3)), ((2, 2, 2, 2), "periodic", (0, 1))])
@pytest.mark.parametrize("csw", [0.0, 1.0])
def test_force_on_short_slabs(dims, bc, dom, csw):
    """Two solves to 1e-13 each: 1e-9 of the largest entry, as for the force's other tests."""
    lqcd = _lq()
    U = inputs.random_su3_field(dims, 0.4, 13)
    lat = lqcd.Lattice(dims, bc)
    lat.set_gauge(U, 0.12, csw)
    op = oracle.Operator(dims, U, 0.12, csw, BCS[bc])
    phi = op.masked(inputs.gaussian_spinor(dims, 14)[0], *dom)
    ref, S_ref, _, _ = oracle.link_force(op, phi, *dom)
    F, S, _ = lat.link_force(_cuda(phi[inputs.slab_sites(dims, *dom)]), dom, 0,
                             lqcd.SolverParams(tol=1e-13, precision=64))
    assert np.abs(F.cpu().numpy().reshape(ref.shape) - ref).max() <= 1e-9 * np.abs(ref).max()
    assert abs(S - S_ref) <= 1e-9 * abs(S_ref)
    lat.close()


def test_force_in_runs_of_slices():
    """A lattice whose insertions do not fit the scratch at once (8 x 48^3: three runs of slices): shifting the fields in
    time moves every slice to another place in its run and must shift the force.  1e-9: two solves to 1e-12 of an operator
    with a condition number below 100."""
    lqcd = _lq()
    dims = (8, 48, 48, 48)
    S3 = 48 ** 3
    U = inputs.random_su3_field_device(dims, 0.4, 3, rng="device").reshape(8, -1)
    phi = _cuda(inputs.gaussian_spinor(dims, 15)[0])
    F = []
    for k in (0, 1):
        lat = lqcd.Lattice(dims, "periodic")
        lat.set_gauge(U.roll(k, 0).contiguous().reshape(-1, 4, 3, 3), 0.12, 1.0)
        f, _, _ = lat.link_force(phi.roll(k * S3, 0).contiguous(), (0, 7), 0, lqcd.SolverParams(tol=1e-12, precision=32))
        F.append(f.reshape(8, -1).roll(-k, 0).clone())
        lat.close()
    assert (F[0] - F[1]).abs().max().item() <= 1e-9 * F[0].abs().max().item()
