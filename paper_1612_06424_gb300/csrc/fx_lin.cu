// Instantiations of the fixed-point FP64 stencil (k_fx_lin) and its conversion.
#include "fx.cuh"

namespace lq {

// FP64 vectors of a batch to limbs and exponents, one site per thread.
__global__ void __launch_bounds__(128) k_to_fx(int nsys, const SysDesc* sys, const int* active, const double2* in,
                                               int4* out, int* oute) {
  int s, by;
  grid_pos(nsys, s, by);
  if (active && !active[s]) return;
  const SysDesc sd = sys[s];
  const int j = by * blockDim.x + threadIdx.x;
  if (j >= sd.n) return;
  cx<double> v[12];
  Prec<64>::load(v, in + sd.off * 12, nullptr, sd.n, j);
  const int e = fx_max_exponent<12>(v);
  oute[sd.off + j] = e;
  int4* o = out + sd.off * 12 + j;
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const cl q = fx_limbs(v[k], e == FX_NAN ? 2047 : e);
    o[k * sd.n] = make_int4(q.r1, q.r0, q.i1, q.i0);
  }
}

void to_fx_launch(dim3 gr, int nsys, const SysDesc* sys, const int* active, const double2* in, int4* out, int* oute,
                  cudaStream_t st) {
  k_to_fx<<<gr, 128, 0, st>>>(nsys, sys, active, in, out, oute);
}

// lqcd_dslash's input: natural slab vector to even / odd FP64 vectors and limbs, one site of parity blockIdx.y
// per thread; the descriptor and the output pointer, which later kernels read, to the device.
__global__ void __launch_bounds__(128) k_dslash_in(Geom g, SysDesc sd, const double2* in, void* out, SysDesc* d_sys,
                                                   void** d_ptr, double2* ve, double2* vo, int4* le, int4* lo, int* ee,
                                                   int* eo) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, p = blockIdx.y;
  if (j == 0 && p == 0) {
    *d_sys = sd;
    d_ptr[0] = out;
  }
  if (j >= sd.n) return;
  int x[4];
  eo_coords(g, sd.cb0 + j, p, x);
  const long long loc = (((long long)(x[0] - sd.t0) * g.L[1] + x[1]) * g.L[2] + x[2]) * g.L[3] + x[3];
  cx<double> v[12];
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const double2 w = __ldg(in + loc * 12 + k);
    v[k] = {w.x, w.y};
  }
  Prec<64>::store(p ? vo : ve, nullptr, sd.n, j, v);
  const int e = fx_max_exponent<12>(v);
  (p ? eo : ee)[j] = e;
  int4* o = (p ? lo : le) + j;
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const cl q = fx_limbs(v[k], e == FX_NAN ? 2047 : e);
    o[k * sd.n] = make_int4(q.r1, q.r0, q.i1, q.i0);
  }
}
void dslash_in_launch(const Geom& g, const SysDesc& s, const double2* in, void* out, SysDesc* d_sys, void** d_ptr,
                      double2* ve, double2* vo, int4* le, int4* lo, int* ee, int* eo, cudaStream_t st) {
  k_dslash_in<<<dim3((unsigned)((s.n + 127) / 128), 2), 128, 0, st>>>(g, s, in, out, d_sys, d_ptr, ve, vo, le, lo, ee, eo);
}

template <bool DAG, bool CLOV>
static int pick(int red, int epi, dim3 gr, const FxArgs& m, cudaStream_t st) {
  constexpr int XY = EPI_X | EPI_Y, XZ = EPI_X | EPI_Z, XYZ = EPI_X | EPI_Y | EPI_Z;
  if (red == RED_NONE && epi == XY) k_fx_lin<DAG, CLOV, RED_NONE, XY><<<gr, 128, 0, st>>>(m);
  else if (red == RED_NONE && epi == XZ) k_fx_lin<DAG, CLOV, RED_NONE, XZ><<<gr, 128, 0, st>>>(m);
  else if (red == RED_DOT_W && epi == XY) k_fx_lin<DAG, CLOV, RED_DOT_W, XY><<<gr, 128, 0, st>>>(m);
  else if (red == RED_TS && epi == XY) k_fx_lin<DAG, CLOV, RED_TS, XY><<<gr, 128, 0, st>>>(m);
  else if (red == RED_NORM && epi == XYZ) k_fx_lin<DAG, CLOV, RED_NORM, XYZ><<<gr, 128, 0, st>>>(m);
  else return -1;
  return 0;
}

int fx_lin_launch(bool dag, bool clov, int red, int epi, dim3 gr, const FxArgs& m, cudaStream_t st) {
  if (dag) return clov ? pick<true, true>(red, epi, gr, m, st) : pick<true, false>(red, epi, gr, m, st);
  return clov ? pick<false, true>(red, epi, gr, m, st) : pick<false, false>(red, epi, gr, m, st);
}

}  // namespace lq
