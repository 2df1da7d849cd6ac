"""What the FP64 operator takes of the device's memory, the form that takes none, and the timing hook."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1612_06424_gb300 import inputs

pytestmark = pytest.mark.gpu


def _lq():
    from paper_1612_06424_gb300 import build, lqcd

    build.build()
    return lqcd


class _Pool:
    """The default stream-ordered memory pool's mark of the most memory in use (CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH)."""

    def __init__(self):
        self.cu, self.h = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.h), torch.cuda.current_device()) == 0

    def used(self, attr):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.h, attr, ctypes.byref(v)) == 0
        return v.value

    def trim(self):
        torch.cuda.synchronize()
        assert self.cu.cuMemPoolTrimTo(self.h, ctypes.c_size_t(0)) == 0

    def peak_of(self, call):
        torch.cuda.synchronize()
        zero, before = ctypes.c_uint64(0), self.used(7)
        assert self.cu.cuMemPoolSetAttribute(self.h, 8, ctypes.byref(zero)) == 0
        call()
        return self.used(8) - before


@pytest.mark.parametrize("dom", [None, (2, 5)])
def test_dslash_takes_four_vectors_of_a_parity(dom):
    lqcd = _lq()
    dims = (8, 12, 8, 12)
    lat = lqcd.Lattice(dims, "periodic")
    lat.set_gauge(inputs.unit_field(dims), 0.13, 0.0)
    n = lat.slab_len(*(dom or (0, 7)))
    psi = torch.randn((n, 4, 3), dtype=torch.complex128, device="cuda")
    peak = _Pool().peak_of(lambda: lat.dslash(psi, 0, dom, False, 64))
    assert 0 < peak <= 4 * 192 * (n // 2) + 8 * (n // 2) + 4096
    lat.close()


# 2 x 21840 sites are four sites a parity below the limit of the scratch
@pytest.mark.parametrize("dims,dom,bc", [((2, 2, 2, 4), None, "periodic"), ((6, 4, 2, 10), (1, 4), "open"),
                                         ((4, 2, 2, 2730), None, "antiperiodic"), ((4, 8, 8, 4), None, "open")])
@pytest.mark.parametrize("csw,dag", [(0.0, 0), (1.0, 1)])
def test_noalloc_dslash_is_dslash(dims, dom, bc, csw, dag):
    """The same kernels in the same order, also replayed from a captured graph."""
    lqcd = _lq()
    lat = lqcd.Lattice(dims, bc)
    lat.set_gauge(inputs.random_su3_field(dims, 0.4, 91), 0.13, csw)
    n = lat.slab_len(*(dom or (0, dims[0] - 1)))
    psi = torch.from_numpy(inputs.gaussian_spinor(dims, 92)[0][:n] * 10.0 ** np.arange(-6, 6).reshape(4, 3)).cuda()
    out = torch.full_like(psi, float("nan"))
    L = lqcd.lib()
    L.lqcd_dslash_noalloc.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.POINTER(lqcd.Slab), ctypes.c_int,
                                      ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]

    def call():
        rc = L.lqcd_dslash_noalloc(lat._h, 0, ctypes.byref(lqcd.Slab(*dom)) if dom else None, dag, psi.data_ptr(),
                                   out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0, L.lqcd_last_error()

    peak = _Pool().peak_of(call)
    assert peak == 0
    assert torch.equal(out, lat.dslash(psi, 0, dom, bool(dag), 64))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    psi.mul_(0.5)
    graph.replay()
    assert torch.equal(out, lat.dslash(psi, 0, dom, bool(dag), 64))
    lat.close()


def test_stencil_bench_knows_its_kernels():
    """Six kernels, each under one number: an iteration's sum over all numbers counts none twice."""
    lqcd = _lq()
    lat = lqcd.Lattice((4, 4, 4, 4), "open")
    lat.set_gauge(inputs.unit_field((4, 4, 4, 4)), 0.13, 1.0)
    for kernel in range(6):
        for precision in (64, 32, 16):
            assert lat.stencil_bench([(0, 3)] * 2, [0] * 2, precision, kernel, 1)[0] > 0
    for kernel in (-1, 6):
        with pytest.raises(lqcd.LQCDError, match="bad arguments"):
            lat.stencil_bench([(0, 3)], [0], 32, kernel, 1)
    lat.close()


def test_set_gauge_on_a_nearly_full_device():
    """A field is loaded again (its storage stays) with 200 MB left, half of what runs of 2^19 sites take for the clover planes."""
    lqcd = _lq()
    dims = (24, 24, 24, 80)
    lat = lqcd.Lattice(dims, "open")
    U = inputs.random_su3_field_device(dims, 0.4, 3, rng="device").contiguous()
    psi = torch.randn((lat.V, 4, 3), dtype=torch.complex128, device="cuda")
    lat.set_gauge(U, 0.13, 1.0)
    want = lat.dslash(psi, 0, None, False, 64)
    lat.set_gauge(U, 0.13, 0.0)
    torch.cuda.empty_cache()
    pool = _Pool()
    pool.trim()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (200 << 20), dtype=torch.uint8, device="cuda")
    lat.set_gauge(U, 0.13, 1.0)
    del fill
    torch.cuda.empty_cache()
    assert torch.equal(lat.dslash(psi, 0, None, False, 64), want)
    lat.close()


@pytest.mark.parametrize("nx,ny", [(608, 1), (304, 5), (607, 1)])
def test_contraction_without_parts(nx, ny):
    """As many pairs as fill the GPU take one part each and no scratch: summed in place.  16 products a sum."""
    lqcd = _lq()
    r = np.random.default_rng(94)
    c = lambda *s: r.standard_normal(s) + 1j * r.standard_normal(s)  # noqa: E731
    bx, by = c(nx, 2, 2, 2, 4), c(ny, 2, 2, 2, 4)
    gx, gy = torch.from_numpy(bx).cuda(), torch.from_numpy(by).cuda()
    W = []
    peak = _Pool().peak_of(lambda: W.append(lqcd.nucleon_contract(gx, gy).cpu().numpy()))
    assert (peak == 0) == (nx != 607)
    z = np.einsum("gd,yijkd->yijkg", oracle.gamma(4) @ (0.5 * (np.eye(4) - oracle.gamma(0))), by)
    for q, axes in enumerate("jik kij".split()):
        ref = -np.einsum("x%sg,yijkg->xy" % axes, bx, z)
        M = np.einsum("x%sg,yijkg->xy" % axes, np.abs(bx), np.abs(z))
        assert np.all(np.abs(W[0][:, :, q] - ref) <= 4 * 2 ** 0.5 * 16 * 2.0 ** -53 * M)
