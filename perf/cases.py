"""The measured cases: what a program that uses this framework has it do.

A user of the library loads gauge fields, applies the Dirac operator, solves for
domain propagators and their corrections, evaluates link forces, estimates
disconnected traces, builds projection vectors and contracts nucleons.  Each
kind of case below is one of these calls through the public binding
(``paper_1612_06424_gb300.lqcd``), at the lattices of the bench workloads, of
the tests and at odd ones between them:

  dslash      one application of D or D^dag on a slab (a caller with a solver of its own)
  load        a new gauge field, then one application of D (the start of every step)
  solve       block solves for random sources on several slabs (FP64, FP32 or FP16 inside)
  props       point-source propagators of every slab of a lattice, all in one batch
  fact        the 12-source factorized propagator and its correction (the headline call)
  force       the link force of a domain's pseudofermion action
  disc        stochastic disconnected traces on Gamma, Gamma* and the full lattice
  modes       projection vectors by inverse iteration and orthonormalisation
  blocks      nucleon blocks of N projected factors (the dense contraction)
  multilevel  level-1 averages of nucleon blocks, then their Wick contractions
  projected   the projected case-II propagator from N factors
  npoint      nucleon point correlators of whole propagators

Linear solves ask for 1e-12 (1e-13 for the inverse iterations), as the tests of
the library do: the solutions are then the same to well below 1e-9 whatever
iterates led to them.
"""
import math

import numpy as np
import torch

from paper_1612_06424_gb300 import lqcd

TOL = 1e-12
TOL_MODES = 1e-13


# ------------------------------------------------------------------- the cases
def _case(kind, T, L1, L2, L3, **kw):
    return dict(kind=kind, T=T, L1=L1, L2=L2, L3=L3, **kw)


def listed():
    return [
        # smallest call: one operator application on the 4^4 test lattice; all latency and launches
        dict(_case("dslash", 4, 4, 4, 4, bc="open", kappa=0.12, csw=0.0, t0=0, t1=3, dagger=False), name="dslash_4x4"),
        # a new level-1 field of the force lattice is loaded and D applied once
        dict(_case("load", 48, 24, 24, 24, bc="open", kappa=0.132, csw=1.0), name="load_24x48"),
        # a few block solves on an odd lattice, FP16 inside, antiperiodic in time
        dict(_case("solve", 14, 10, 6, 18, bc="antiperiodic", kappa=0.124, csw=1.0, slabs=2, n=5, precision=16),
             name="solve_fp16_ragged"),
        # the 16^3 x 32 factorized propagator and correction of the bench
        dict(_case("fact", 32, 16, 16, 16, kappa=0.13, csw=1.0, g1=13, d1=17, precision=32), name="factorized_16x32"),
        # domain propagators of the 32^3 workload: 8-slice slabs, 12 sources each
        dict(_case("props", 32, 32, 32, 32, kappa=0.134, csw=1.0, slabs=4, precision=32), name="propagators_32x32"),
        # one molecular-dynamics force on a 12-slice domain: a single right-hand side
        dict(_case("force", 48, 24, 24, 24, kappa=0.132, csw=1.0, t0=12, t1=23, precision=32), name="force_24x48"),
        # Wilson quarks on the paper's lattice: two sources on Gamma, Gamma* and the full lattice
        dict(_case("disc", 64, 24, 24, 24, kappa=0.136, g1=31, n=2, precision=32), name="disconnected_64x24"),
        # one inverse iteration of 24 projection vectors on the 16 slices around the cut
        dict(_case("modes", 16, 24, 24, 24, kappa=0.136, g1=7, n=24, iters=1, precision=32), name="modes_16x24"),
        # nucleon blocks of 120 factors on two slices of 24^3
        dict(_case("blocks", 2, 24, 24, 24, n=120, t0=0, nt=2, conj=False), name="blocks_24_120"),
        # level-1 averages over two fields and all Wick contractions, 120 factors, 8 sink slices
        dict(kind="multilevel", n=120, levels=2, nx=1, ny=8, name="multilevel_120"),
        # the projected propagator from 120 factors on 24 slices of 24^3
        dict(_case("projected", 32, 24, 24, 24, g1=7, n=120), name="projected_32x24"),
        # nucleon point correlator of one propagator on the paper's lattice
        dict(_case("npoint", 64, 24, 24, 24, n=1, t0=0, nt=64), name="npoint_64x24"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    return 2 * max(1, round(_log(rng, lo, hi) / 2))


def _lattice(rng, vmax, lmax=32, tmax=64):
    while True:
        d = (_even(rng, 4, tmax), _even(rng, 4, lmax), _even(rng, 4, lmax), _even(rng, 4, lmax))
        if rng.random() < 0.5:  # cubic space, as most lattices are
            d = (d[0], d[1], d[1], d[1])
        if d[0] * d[1] * d[2] * d[3] <= vmax:
            return d


def draw(rng):
    kind = rng.choice(["dslash", "load", "solve", "props", "fact", "force", "disc", "modes", "blocks", "multilevel",
                       "projected", "npoint"])
    kappa, csw = round(rng.uniform(0.115, 0.132), 5), rng.choice([0.0, 1.0])
    bc = rng.choice(["open", "periodic", "antiperiodic"])
    prec = rng.choice([32, 32, 16])
    if kind == "dslash":
        d = _lattice(rng, 663552)
        t0 = rng.randrange(d[0])
        return _case(kind, *d, bc=bc, kappa=kappa, csw=csw, t0=t0, t1=rng.randrange(t0, d[0]), dagger=rng.random() < 0.5)
    if kind == "load":
        return _case(kind, *_lattice(rng, 663552), bc=bc, kappa=kappa, csw=csw)
    if kind == "solve":
        d = _lattice(rng, 65536)
        return _case(kind, *d, bc=bc, kappa=kappa, csw=csw, slabs=rng.choice([1, 2]), n=rng.randint(1, 13),
                     precision=rng.choice([64, 32, 16]))
    if kind == "props":
        while True:
            d, slabs = _lattice(rng, 524288), rng.choice([1, 2, 3, 4, 8])
            if d[0] >= 2 * slabs:
                return _case(kind, *d, kappa=kappa, csw=csw, slabs=slabs, precision=prec)
    if kind == "fact":
        while True:
            d = _lattice(rng, 131072)
            if d[0] >= 8:
                g1 = rng.randrange(1, d[0] // 2)
                return _case(kind, *d, kappa=kappa, csw=csw, g1=g1, d1=g1 + rng.randint(1, 4) if g1 + 6 < d[0] else g1,
                             precision=prec)
    if kind == "force":
        d = _lattice(rng, 663552, tmax=48)
        t0 = rng.randrange(d[0] - 1)
        return _case(kind, *d, kappa=kappa, csw=csw, t0=t0, t1=min(d[0] - 1, t0 + rng.randint(1, 12)), precision=prec)
    if kind == "disc":
        d = _lattice(rng, 884736)
        return _case(kind, *d, kappa=kappa, g1=rng.randrange(d[0] - 1), n=rng.randint(1, 2), precision=prec)
    if kind == "modes":
        d = _lattice(rng, 131072, lmax=24, tmax=16)
        return _case(kind, *d, kappa=kappa, g1=rng.randrange(d[0]), n=rng.randint(3, 40), iters=1, precision=32)
    if kind == "blocks":
        d = _lattice(rng, 2 * 13824, lmax=24, tmax=8)
        t0 = rng.randrange(d[0])
        n = max(3, round(_log(rng, 3, 120)))
        return _case(kind, *d, n=n, t0=t0, nt=rng.randint(1, min(2, d[0] - t0)), conj=rng.random() < 0.5)
    if kind == "multilevel":
        return dict(kind=kind, n=max(3, round(_log(rng, 3, 120))), levels=rng.randint(1, 2), nx=rng.randint(1, 2),
                    ny=rng.randint(1, 4))
    if kind == "projected":
        d = _lattice(rng, 442368, lmax=24, tmax=32)
        return _case(kind, *d, g1=rng.randrange(d[0] // 2), n=max(1, round(_log(rng, 1, 120))))
    d = _lattice(rng, 442368)
    t0 = rng.randrange(d[0])
    return _case("npoint", *d, n=rng.randint(1, 2), t0=t0, nt=rng.randint(1, d[0] - t0))


# ------------------------------------------------------------------ the inputs
def _dims(c):
    return (c["T"], c["L1"], c["L2"], c["L3"])


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + stream)
    return g


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _gauge(dims, seed, eps=0.4):
    """Links exp(i eps H), H = sum_a h_a lambda_a / 2 with normal h_a, re-unitarised: [V, 4, 3, 3] complex128."""
    n = int(np.prod(dims)) * 4
    lam = torch.from_numpy(_gell_mann() / 2).to("cuda")
    gen = _gen(seed, 1)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    for lo in range(0, n, 1 << 20):
        m = min(n, lo + (1 << 20)) - lo
        h = torch.randn((m, 8), dtype=torch.float64, device="cuda", generator=gen)
        x = (1j * eps) * (h.to(torch.complex128) @ lam.reshape(8, 9)).reshape(m, 3, 3)
        u = torch.eye(3, dtype=torch.complex128, device="cuda").expand(m, 3, 3)
        for k in range(12, 0, -1):
            u = torch.eye(3, dtype=torch.complex128, device="cuda") + _mm(x, u) / k
        r0 = u[:, 0] / torch.linalg.vector_norm(u[:, 0], dim=-1, keepdim=True)
        r1 = u[:, 1] - (r0.conj() * u[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        out[lo:lo + m] = torch.stack([r0, r1, torch.linalg.cross(r0, r1, dim=-1).conj()], dim=1)
    return out.reshape(-1, 4, 3, 3)


def _gell_mann():
    m = np.zeros((8, 3, 3), dtype=np.complex128)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        m[a, i, j] = m[a, j, i] = 1
        m[a + 1, i, j], m[a + 1, j, i] = -1j, 1j
    m[7] = np.diag([1, 1, -2]) / np.sqrt(3)
    m[2] = np.diag([1, -1, 0])
    return m


def _normal(shape, seed, stream, scale=1.0):
    """Complex normal numbers (Re, Im ~ N(0, scale^2 / 2))."""
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=_gen(seed, stream)) * scale


def _slabs(T, n):
    return [(k * T // n, (k + 1) * T // n - 1) for k in range(n)]


def _x_src(c, seed, t):
    r = np.random.RandomState(seed % (1 << 31))
    return (t, int(r.randint(c["L1"])), int(r.randint(c["L2"])), int(r.randint(c["L3"])))


def _inputs(c, seed):
    """What a case's inputs are made of, from the seed alone."""
    k = c["kind"]
    if k == "multilevel":
        n = c["n"]
        return {"bx": _normal((c["levels"], c["nx"], n, n, n, 4), seed, 2),
                "be": _normal((c["levels"], c["ny"], n, n, n, 4), seed, 3)}
    dims = _dims(c)
    S3 = dims[1] * dims[2] * dims[3]
    V = dims[0] * S3
    d = {}
    if k in ("dslash", "load", "solve", "props", "fact", "force", "disc", "modes"):
        d["U"] = _gauge(dims, seed)
    if k == "dslash":
        d["psi"] = _normal(((c["t1"] - c["t0"] + 1) * S3, 4, 3), seed, 2)
    elif k == "load":
        d["psi"] = _normal((V, 4, 3), seed, 2)
    elif k == "solve":
        sl = _slabs(c["T"], c["slabs"])
        d["doms"] = [sl[i % len(sl)] for i in range(c["n"])]
        d["src"] = _normal((sum(b - a + 1 for a, b in d["doms"]) * S3, 4, 3), seed, 2)
    elif k == "props":
        d["doms"] = _slabs(c["T"], c["slabs"])
        d["x"] = [_x_src(c, seed + i, (a + b + 1) // 2) for i, (a, b) in enumerate(d["doms"])]
    elif k == "fact":
        d["x"] = _x_src(c, seed, min(2, c["g1"]))
    elif k == "force":
        d["phi"] = _normal(((c["t1"] - c["t0"] + 1) * S3, 4, 3), seed, 2)
    elif k == "disc":
        d["doms"] = [(0, c["g1"]), (c["g1"] + 1, c["T"] - 1), (0, c["T"] - 1)]
        d["eta"] = _normal((c["n"], V, 4, 3), seed, 2)
    elif k == "modes":
        d["v0"] = _normal((c["n"], V, 4, 3), seed, 2)
    elif k == "blocks":
        d["s"] = _normal((c["n"], V, 4, 3), seed, 2, 0.1)
    elif k == "projected":
        d["xi"] = _normal((c["n"], (c["g1"] + 1) * S3, 4, 3), seed, 2, 0.1)
        d["eta"] = _normal((c["n"], V - (c["g1"] + 1) * S3, 4, 3), seed, 3, 0.1)
        d["x"] = _x_src(c, seed, c["g1"] // 2)
    elif k == "npoint":
        d["prop"] = _normal((c["n"], 12, V, 4, 3), seed, 2, 0.1)
    return d


def prepare(case, seed):
    c, k = dict(case), case["kind"]
    s = {"c": c, "in": _inputs(c, seed)}
    if k == "multilevel":
        return s
    lat = lqcd.Lattice(_dims(c), c.get("bc", "open"))
    s["lat"] = lat
    if "U" in s["in"]:
        if k == "load":
            s["U"] = s["in"]["U"].unsqueeze(0).contiguous()
        else:
            lat.set_gauge(s["in"].pop("U"), c["kappa"], c.get("csw", 0.0))
    if "precision" in c:
        s["prm"] = lqcd.SolverParams(tol=TOL_MODES if k == "modes" else TOL, precision=c["precision"])
    return s


def run(state):
    c, d, k = state["c"], state["in"], state["c"]["kind"]
    if k == "multilevel":
        return lqcd.multilevel_nucleon(d["bx"], d["be"])
    lat, prm = state["lat"], state.get("prm")
    if k == "dslash":
        return lat.dslash(d["psi"], dom=(c["t0"], c["t1"]), dagger=c["dagger"])
    if k == "load":
        lat.set_gauge(state["U"], c["kappa"], c["csw"])
        return lat.dslash(d["psi"])
    if k == "solve":
        return lat.solve_block(d["src"], d["doms"], [0] * c["n"], prm)[0]
    if k == "props":
        doms = [m for m in d["doms"] for _ in range(12)]
        xs = [x for x in d["x"] for _ in range(12)]
        return lat.point_propagators(doms, [0] * len(doms), xs, list(range(12)) * len(d["doms"]), prm)[0]
    if k == "fact":
        delta = (c["g1"] + 1, c["d1"]) if c["d1"] > c["g1"] else None
        fact, corr, _ = lat.factorized_propagator((0, c["g1"]), (c["g1"] + 1, c["T"] - 1), d["x"], delta=delta, params=prm)
        corr += fact  # the full propagator, which the correction completes
        return fact, corr
    if k == "force":
        F, S, _ = lat.link_force(d["phi"], (c["t0"], c["t1"]), 0, prm)
        return F, S
    if k == "disc":
        return lat.disconnected_trace(d["eta"], d["doms"], 0, prm)[:2]
    if k == "modes":
        return lat.boundary_modes(d["v0"], (0, c["T"] - 1), c["g1"], 0, c["iters"], prm)[0]
    if k == "blocks":
        return lat.nucleon_blocks(d["s"], (0, c["T"] - 1), c["t0"], c["nt"], conj=c["conj"])
    if k == "projected":
        return lat.projected_propagator(d["xi"], d["eta"], (0, c["g1"]), (c["g1"] + 1, c["T"] - 1), d["x"])
    return lat.nucleon_point(d["prop"], c["t0"], c["nt"])


# -------------------------------------------------------------------- the work
# Operator applications of an even-odd BiCGStab to the tolerances above are counted as SOLVE
# per system: a typical number on these fields (100 iterations of two applications), since no
# formula gives what a Krylov solve needs.
SOLVE = 200


def work(case):
    c, k = case, case["kind"]
    z = 16  # bytes of a complex128
    if k == "multilevel":
        n3 = 4 * c["n"] ** 3
        return {"bytes": z * n3 * c["levels"] * (c["nx"] + c["ny"]),
                "flops": n3 * (2 * c["levels"] * (c["nx"] + c["ny"]) + 2 * 8 * c["nx"] * c["ny"])}
    T, S3 = c["T"], c["L1"] * c["L2"] * c["L3"]
    V = T * S3
    app = 1368 + (504 if c.get("csw") else 0)  # flop of D per site
    fld, spn = z * 36, z * 12  # bytes per site
    if k == "dslash":
        n = (c["t1"] - c["t0"] + 1) * S3
        return {"bytes": n * (fld + 2 * spn), "flops": n * app}
    if k == "load":
        clover = 6 * 4 * 3 * 198 + 2 * 1000 if c["csw"] else 0  # leaves, then two 6x6 inverses on half the sites
        return {"bytes": V * (fld + 2 * spn), "flops": V * (app + clover)}
    if k == "solve":
        sl = _slabs(T, c["slabs"])
        n = sum((sl[i % len(sl)][1] - sl[i % len(sl)][0] + 1) for i in range(c["n"])) * S3
        return {"bytes": V * fld + 2 * n * spn, "flops": n * app * SOLVE}
    if k == "props":
        return {"bytes": V * (fld + 12 * spn), "flops": 12 * V * app * SOLVE}
    if k == "fact":
        n = 12 * S3 * (c["g1"] + 1 + max(c["d1"], c["g1"]) + 1 + T - c["g1"] - 1 + T)
        return {"bytes": V * (fld + 24 * spn), "flops": n * app * SOLVE}
    if k == "force":
        n = (c["t1"] - c["t0"] + 1) * S3
        return {"bytes": V * fld + n * spn + V * 32 * 8, "flops": n * (2 * app * SOLVE + 4 * 20000)}
    if k == "disc":
        return {"bytes": V * (fld + c["n"] * spn), "flops": 2 * c["n"] * V * app * (SOLVE + 8)}
    if k == "modes":
        n = c["n"] * V
        return {"bytes": V * fld + n * spn, "flops": n * (app * SOLVE * c["iters"] + 2 * 8 * 12 * c["n"])}
    if k == "blocks":
        n, m = c["n"], c["nt"] * S3
        return {"bytes": n * m * spn + z * 4 * c["nt"] * n ** 3, "flops": m * (8 * 12 * n ** 3 + 8 * 24 * n * n)}
    if k == "projected":
        m = (T - c["g1"] - 1) * S3
        return {"bytes": c["n"] * m * spn + 12 * V * spn, "flops": 8 * 144 * c["n"] * m}
    m = c["n"] * c["nt"] * S3
    return {"bytes": 12 * m * spn, "flops": m * 8 * (2 * 81 * 16 + 36 * 16 * 3)}


# ------------------------------------------------------- the same in plain torch
def _gammas():
    s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    g = [np.block([[np.zeros((2, 2)), -np.eye(2)], [-np.eye(2), np.zeros((2, 2))]])]
    g += [np.block([[np.zeros((2, 2)), -1j * p], [1j * p, np.zeros((2, 2))]]) for p in s]
    return g


class _Dirac:
    """D = 1/(2 kappa) - D_hop / 2 + clover in plain torch; vectors [T, L1, L2, L3, colour, spin, column].
    Time hops between slices t and t + 1 are dropped for t in `cuts` (t = T - 1: the wrapping hop)."""

    def __init__(self, U, dims, kappa, csw, bc, cuts, dev="cuda"):
        self.kappa, self.csw, self.dims, self.dev = kappa, csw, dims, dev
        T = dims[0]
        U = U.reshape(*dims, 4, 3, 3)
        w = torch.ones(T, dtype=torch.complex128, device=dev)
        w[T - 1] = {"open": 0.0, "periodic": 1.0, "antiperiodic": -1.0}[bc]
        for t in cuts:
            w[t] = 0.0
        self.u = [U[..., m, :, :] for m in range(4)]
        gate = torch.ones(T, dtype=torch.complex128, device=dev)
        if bc == "open":
            gate[T - 1] = 0.0
        self.clover = self._clover([self.u[0] * gate.reshape(T, 1, 1, 1, 1, 1)] + self.u[1:]) if csw else None
        self.u[0] = self.u[0] * w.reshape(T, 1, 1, 1, 1, 1)
        # a row of gamma_mu has one entry: (gamma psi)_s = phase_s psi_perm(s)
        self.perm = [torch.from_numpy(np.abs(g).argmax(1)).to(dev) for g in _gammas()]
        self.phase = [torch.from_numpy(g[np.arange(4), np.abs(g).argmax(1)].reshape(4, 1).astype(np.complex128)).to(dev)
                      for g in _gammas()]

    def _clover(self, u):
        g = _gammas()
        dag = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
        out = 0
        for m in range(4):
            for n in range(m + 1, 4):
                a, b = u[m], u[n]
                up = lambda x, d: torch.roll(x, -1, d)  # noqa: E731
                dn = lambda x, d: torch.roll(x, 1, d)  # noqa: E731
                q = _mm(_mm(a, up(b, m)), _mm(dag(up(a, n)), dag(b)))
                q = q + _mm(_mm(b, dag(up(dn(a, m), n))), _mm(dag(dn(b, m)), dn(a, m)))
                q = q + _mm(_mm(dag(dn(a, m)), dag(dn(dn(b, m), n))), _mm(dn(dn(a, m), n), dn(b, n)))
                q = q + _mm(_mm(dag(dn(b, n)), dn(a, n)), _mm(up(dn(b, n), m), dag(a)))
                sig = torch.from_numpy(0.5j * (g[m] @ g[n] - g[n] @ g[m])).to(self.dev)
                f = (q - dag(q)) / 8
                # [.., colour, spin, colour', spin']
                out = out + f[..., :, None, :, None] * sig[:, None, :]
        return (0.5j * self.csw * out).reshape(*self.dims, 12, 12)

    def apply(self, psi, dagger=False):
        sh = psi.shape
        out = psi / (2 * self.kappa)
        if self.clover is not None:
            out = out + torch.matmul(self.clover, psi.reshape(*self.dims, 12, -1)).reshape(sh)
        flat = sh[:-3] + (3, sh[-2] * sh[-1])
        for m in range(4):
            g = psi.index_select(-2, self.perm[m]) * (-0.5 * self.phase[m] if dagger else 0.5 * self.phase[m])
            h = torch.matmul(self.u[m], torch.roll(0.5 * psi - g, -1, m).reshape(flat))
            out -= h.reshape(sh)
            h = torch.matmul(self.u[m].conj().transpose(-1, -2), (0.5 * psi + g).reshape(flat))
            out -= torch.roll(h.reshape(sh), 1, m)
        return out

    def solve(self, b, dagger=False, tol=2e-14):
        """BiCGStab per column, restarted from the true residual until that is below tol or stops falling."""
        dot = lambda x, y: (x.conj() * y).sum(dim=tuple(range(6)))  # noqa: E731
        safe = lambda x: torch.where(x == 0, torch.ones_like(x), x)  # noqa: E731
        nb = dot(b, b).real
        x, last = torch.zeros_like(b), None
        for _ in range(6):
            r = b - self.apply(x, dagger)
            rr = dot(r, r).real
            if bool((rr <= tol * tol * nb).all()) or (last is not None and bool((rr > 0.1 * last).any())):
                break
            last = rr
            r0, p = r.clone(), r.clone()
            rho = dot(r0, r)
            goal = torch.maximum(1e-24 * rr, 0.1 * tol * tol * nb)
            e = torch.zeros_like(b)
            for it in range(3000):
                live = (rr > goal).to(b.dtype)
                if it % 10 == 0 and not bool(live.abs().any()):
                    break
                v = self.apply(p, dagger)
                al = live * rho / safe(dot(r0, v))
                s = r - al * v
                t = self.apply(s, dagger)
                om = live * dot(t, s) / safe(dot(t, t))
                e += al * p + om * s
                r = s - om * t
                new = dot(r0, r)
                be = live * new / safe(rho) * al / safe(om)
                p = r + be * (p - om * v)
                rho, rr = torch.where(live == 0, rho, new), dot(r, r).real
            x = x + e
        return x


def _in(v, dims):
    """[n, sites, 4, 3] -> [T, L1, L2, L3, 3, 4, n]."""
    return v.reshape(-1, *dims, 4, 3).permute(1, 2, 3, 4, 6, 5, 0).contiguous()


def _out(v):
    n = v.shape[-1]
    return v.permute(6, 0, 1, 2, 3, 5, 4).reshape(n, -1, 4, 3)


def _points(dims, xs):
    v = torch.zeros((12, *dims, 4, 3), dtype=torch.complex128, device="cuda")
    for x in xs:
        for col in range(12):
            v[(col, *x, col // 3, col % 3)] = 1
    return _in(v, dims)


def _slab_view(v, dims, a, b):
    S3 = dims[1] * dims[2] * dims[3]
    return v[:, a * S3:(b + 1) * S3]


def _qr(w):
    q, r = torch.linalg.qr(w)
    d = torch.diagonal(r)
    return q * (d / d.abs())


def _dslash_exact(c, d, dims, t0, t1, dagger):
    whole = t0 == 0 and t1 == dims[0] - 1
    cuts = [] if whole else [t for t in (t0 - 1, t1) if t >= 0]
    D = _Dirac(d["U"], dims, c["kappa"], c["csw"], c["bc"], cuts + ([] if whole else [dims[0] - 1]))
    S3 = dims[1] * dims[2] * dims[3]
    full = torch.zeros((1, dims[0] * S3, 4, 3), dtype=torch.complex128, device="cuda")
    full[0, t0 * S3:(t1 + 1) * S3] = d["psi"]
    return _out(D.apply(_in(full, dims), dagger))[0, t0 * S3:(t1 + 1) * S3].contiguous()


def _solve_exact(c, d, dims):
    S3 = dims[1] * dims[2] * dims[3]
    sl = _slabs(dims[0], c["slabs"])
    cuts = [] if c["slabs"] == 1 else [b for _, b in sl]
    D = _Dirac(d["U"], dims, c["kappa"], c["csw"], c["bc"], cuts)
    full = torch.zeros((c["n"], dims[0] * S3, 4, 3), dtype=torch.complex128, device="cuda")
    at = 0
    for i, (a, b) in enumerate(d["doms"]):
        m = (b - a + 1) * S3
        full[i, a * S3:(b + 1) * S3] = d["src"][at:at + m]
        at += m
    x = _out(D.solve(_in(full, dims)))
    return torch.cat([x[i, a * S3:(b + 1) * S3] for i, (a, b) in enumerate(d["doms"])])


def _props_exact(c, d, dims):
    D = _Dirac(d["U"], dims, c["kappa"], c["csw"], "open", [b for _, b in d["doms"]])
    x = _out(D.solve(_points(dims, d["x"])))
    return torch.cat([_slab_view(x, dims, a, b).reshape(-1, 4, 3) for a, b in d["doms"]])


def _fact_exact(c, d, dims):
    g1, d1, T = c["g1"], max(c["d1"], c["g1"]), c["T"]
    op = lambda cuts: _Dirac(d["U"], dims, c["kappa"], c["csw"], "open", cuts)  # noqa: E731
    eta = _points(dims, [d["x"]])
    D, Dg = op([]), op([g1])
    full = D.solve(eta)
    psi = op([d1]).solve(eta) if d1 > g1 else Dg.solve(eta)
    psi[g1 + 1:] = 0
    chi = D.apply(psi)
    chi[:g1 + 1] = 0
    eta2 = eta - chi  # Gamma and Gamma* decouple in Dg: both parts of fact in one solve
    return _out(Dg.solve(eta2)), _out(full)


def _force_exact(c, d, dims):
    t0, t1, T = c["t0"], c["t1"], c["T"]
    S3 = dims[1] * dims[2] * dims[3]
    cuts = [t for t in (t0 - 1, t1) if 0 <= t < T]
    U = d["U"].reshape(*dims, 4, 3, 3).clone().requires_grad_(True)
    phi = torch.zeros((1, T * S3, 4, 3), dtype=torch.complex128, device="cuda")
    phi[0, t0 * S3:(t1 + 1) * S3] = d["phi"]
    with torch.no_grad():
        D = _Dirac(U, dims, c["kappa"], c["csw"], "open", cuts)
        Y = D.solve(_in(phi, dims), dagger=True)
        X = D.solve(Y)
        S = float((Y.abs() ** 2).sum())
    lo, hi = max(0, t0 - 1), min(T, t1 + 2)
    part = _Dirac(U, dims, c["kappa"], c["csw"], "open", cuts)
    z = -2 * (Y.conj() * part.apply(X)).sum().real
    (g,) = torch.autograd.grad(z, U)
    U = U.detach()
    F = torch.zeros((T * S3, 4, 8), dtype=torch.float64, device="cuda")
    lam = torch.from_numpy(_gell_mann() / 2).to("cuda")
    for a in range(8):
        du = 1j * torch.matmul(lam[a], U)
        F[..., a] = (g.conj() * du).sum(dim=(-1, -2)).real.reshape(T * S3, 4)
    F.reshape(T, S3, 4, 8)[:lo] = 0
    F.reshape(T, S3, 4, 8)[hi:] = 0
    return F, S


def _disc_exact(c, d, dims):
    T, g1 = c["T"], c["g1"]
    eta = _in(d["eta"], dims)
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.complex128, device="cuda").reshape(4, 1)
    out = torch.zeros((c["n"], 3, T), dtype=torch.complex128, device="cuda")
    for cuts, where in (([g1], (0, 1)), ([], (2,))):
        D = _Dirac(d["U"], dims, c["kappa"], 0.0, "open", cuts)
        y = D.solve(g5 * eta)
        for _ in range(8):
            y = y - 2 * c["kappa"] * D.apply(y)
        tr = (eta.conj() * y).sum(dim=(1, 2, 3, 4, 5)).transpose(0, 1)  # [n, T]
        for k in where:
            a, b = d["doms"][k]
            out[:, k, a:b + 1] = tr[:, a:b + 1]
    return out, out.mean(0)


def _modes_exact(c, d, dims):
    S3, n = dims[1] * dims[2] * dims[3], c["n"]
    D = _Dirac(d["U"], dims, c["kappa"], c["csw"] if "csw" in c else 0.0, "open", [])
    v = _in(d["v0"], dims)
    for _ in range(c["iters"]):
        v = _in(_qr(_out(D.solve(v)).reshape(n, -1).transpose(0, 1)).transpose(0, 1).reshape(n, -1, 4, 3), dims)
    s = _out(v)[:, c["g1"] * S3:(c["g1"] + 1) * S3]
    u = 0.5 * (s[:, :, :2] - s[:, :, 2:])
    phi = torch.cat([u, -u], dim=2).reshape(n, -1)
    return _qr(phi.transpose(0, 1)).transpose(0, 1).reshape(n, S3, 4, 3).contiguous()


_EVEN = [(0, 1, 2, 1.0), (1, 2, 0, 1.0), (2, 0, 1, 1.0), (0, 2, 1, -1.0), (2, 1, 0, -1.0), (1, 0, 2, -1.0)]


def _spin_forms():
    g = _gammas()
    g5 = np.diag([1.0, 1.0, -1.0, -1.0])
    to = lambda m: torch.from_numpy(np.ascontiguousarray(m.astype(np.complex128))).to("cuda")  # noqa: E731
    return to(g[0] @ g[2] @ g5), to(g5 @ (0.5 * (np.eye(4) - g[0])))


def _blocks_exact(c, d, dims):
    S3, n = dims[1] * dims[2] * dims[3], c["n"]
    cg5, _ = _spin_forms()
    s = d["s"].conj().resolve_conj() if c["conj"] else d["s"]
    B = torch.zeros((c["nt"], n, n, n, 4), dtype=torch.complex128, device="cuda")
    for t in range(c["nt"]):
        for lo in range(0, S3, 1024):
            f = s[:, (c["t0"] + t) * S3 + lo:(c["t0"] + t) * S3 + min(S3, lo + 1024)]  # [n, x, 4, 3]
            w = torch.einsum("mn,jxnb->jxmb", cg5, f)
            dq = torch.stack([sum(sg * torch.einsum("ixm,jxm->ijx", f[..., a], w[..., b])
                                  for a, b, cc, sg in _EVEN if cc == col) for col in range(3)], dim=-1)
            B[t] += (dq.reshape(n * n, -1) @ f.permute(1, 3, 0, 2).reshape(-1, 4 * n)).reshape(n, n, n, 4)
    return B


def _multilevel_exact(c, d):
    _, g5pm = _spin_forms()
    bx, be = d["bx"].mean(0), d["be"].mean(0)
    be = torch.einsum("gd,yijkd->yijkg", g5pm, be).reshape(c["ny"], -1)
    w1 = -bx.permute(0, 2, 1, 3, 4).reshape(c["nx"], -1) @ be.T  # B_xi[j, i, k]
    w2 = -bx.permute(0, 2, 3, 1, 4).reshape(c["nx"], -1) @ be.T  # B_xi[k, i, j]
    return torch.stack([w1, w2], dim=-1)


def _projected_exact(c, d, dims):
    S3 = dims[1] * dims[2] * dims[3]
    V, y0, x = dims[0] * S3, (c["g1"] + 1) * S3, d["x"]
    at = ((x[0] * dims[1] + x[1]) * dims[2] + x[2]) * dims[3] + x[3]
    q = d["xi"][:, at].reshape(c["n"], 12)
    out = torch.zeros((12, V, 4, 3), dtype=torch.complex128, device="cuda")
    out[:, y0:] = -(q.conj().T @ d["eta"].reshape(c["n"], -1)).reshape(12, V - y0, 4, 3)
    return out


def _npoint_exact(c, d, dims):
    S3 = dims[1] * dims[2] * dims[3]
    cg5, g5pm = _spin_forms()
    W = torch.zeros((c["n"], c["nt"], 2), dtype=torch.complex128, device="cuda")
    for p in range(c["n"]):
        for t in range(c["nt"]):
            for lo in range((c["t0"] + t) * S3, (c["t0"] + t + 1) * S3, 4096):
                hi = min((c["t0"] + t + 1) * S3, lo + 4096)
                P = d["prop"][p, :, lo:hi].reshape(4, 3, hi - lo, 4, 3).permute(2, 3, 4, 0, 1)  # y, mu, a, nu, b
                X = torch.einsum("mn,ymaNB->ynaNB", cg5, P)
                Y = torch.einsum("MN,ynbMA->ynbNA", cg5, P)
                Z = torch.einsum("ynaNB,ynbNA->yaBbA", X, Y)
                R = torch.einsum("gd,ydcgC->ycC", g5pm, P)
                Q = torch.einsum("gd,ydcNA->ygcNA", g5pm, Y)
                w1 = w2 = 0
                for a, b, cc, s in _EVEN:
                    for A, Bb, C, S in _EVEN:
                        w1 = w1 + s * S * (Z[:, a, Bb, b, A] * R[:, cc, C]).sum()
                        # sum over n, N, gamma of X[n, a, N, B] P[n, b, gamma, C] Q[gamma, c, N, A]
                        u = torch.einsum("ynN,yng->yNg", X[:, :, a, :, Bb], P[:, :, b, :, C])
                        w2 = w2 + s * S * (u * Q[:, :, cc, :, A].transpose(1, 2)).sum()
                W[p, t, 0] += w1
                W[p, t, 1] += w2
    return W


def exact(case, seed):
    c, k = dict(case), case["kind"]
    # plain torch applies D in about 1e-8 s per site and (column + 2.3); applications of a case's solves:
    applied = {"solve": 500, "props": 400, "fact": 1250, "force": 830, "disc": 1100, "modes": 500}.get(k)
    if applied:
        columns = 12 if k in ("props", "fact") else c.get("n", 1)
        if applied * 1e-8 * c["T"] * c["L1"] * c["L2"] * c["L3"] * (columns + 2.3) > 18:
            return None  # about 20 s or more
    if k == "npoint" and c["n"] * c["nt"] * c["L1"] * c["L2"] * c["L3"] > 450000:
        return None
    d = _inputs(c, seed)
    if k == "multilevel":
        return _multilevel_exact(c, d)
    dims = _dims(c)
    if k == "dslash":
        return _dslash_exact(c, d, dims, c["t0"], c["t1"], c["dagger"])
    if k == "load":
        return _dslash_exact(c, d, dims, 0, dims[0] - 1, False)
    return {"solve": _solve_exact, "props": _props_exact, "fact": _fact_exact, "force": _force_exact,
            "disc": _disc_exact, "modes": _modes_exact, "blocks": _blocks_exact, "projected": _projected_exact,
            "npoint": _npoint_exact}[k](c, d, dims)
