// Reductions of the batched Krylov kernels and the per-system scalars they feed.
//
// A kernel with a fused inner product stores one FP64 partial per block (block_reduce_store).  The
// solver's kernels then finish the sum themselves (finish_last): the last block of a system to
// arrive, by a counter, adds the system's partials in a fixed order and updates the system's
// scalars and its activity flag.  Nothing waits for another block.  An iteration so needs no
// kernel of its own for each inner product: with k_finalize behind each of the three, launches
// of 5 to 10 us each were 7% of a 16^3 x 32 propagator and a quarter of a solve on a small lattice.
// k_finalize (blas.cuh) does the same in a kernel of its own, for the sums outside the iteration.
#pragma once

#include "common.cuh"

namespace lq {

// Block reduction of NQ per-thread partial sums of type A (the kernel's own
// precision: FP32 for the FP32 / FP16 solver, whose FP64 rate on this GPU is a
// small fraction of its FP32 rate) through a warp-shuffle tree; the per-warp
// sums are widened to FP64 and combined in FP64, one thread per sum in warp order (a shuffle tree
// of FP64 sums held a block back by about 1400 clocks: 35 FP64 steps for 7 sums), and one
// partial per block is stored.  The order is fixed, so results are deterministic.
constexpr int RED_WARPS = 4;  // warps of a block (k_finalize has more)
constexpr int red_smem(int nq) { return 2 * RED_WARPS * nq * 8 + 16; }  // block_reduce_store and finish_last

template <int NQ, typename A>
LQ_DI void block_reduce_store(A v[NQ], double* dst) {
  __shared__ double sh[RED_WARPS][NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NQ; q++) sh[wid][q] = (double)v[q];
  __syncthreads();
  if (threadIdx.x < NQ) {
    double t = sh[0][threadIdx.x];
    for (int w = 1; w < RED_WARPS; w++) t += sh[w][threadIdx.x];
    dst[threadIdx.x] = t;
  }
}

// Sum of nb block partials of NQ values (PW doubles apart), in a fixed order: each thread of the block
// sums a strided subset, the warps reduce by shuffles and thread 0 adds the warp sums in warp order
// and receives the result.  Partials are read past L1 (other blocks of this launch wrote them).
template <int NQ, int PW, int WARPS = RED_WARPS>
LQ_DI void block_sum_partials(const double* partial, int nb, double* out) {
  __shared__ double sh[WARPS][NQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) v[q] = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const double* p = partial + (long long)b * PW;
#pragma unroll
    for (int q = 0; q < NQ; q++) v[q] += __ldcg(p + q);
  }
#pragma unroll
  for (int q = 0; q < NQ; q++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  }
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < NQ; q++) sh[wid][q] = v[q];
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NQ; q++) {
      double t = 0.0;
      for (int w = 0; w < WARPS; w++) t += sh[w][q];
      out[q] = t;
    }
  }
}

LQ_DI double2 cdiv(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
LQ_DI double2 cmul2(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
LQ_DI bool finite2(double2 a) { return isfinite(a.x) && isfinite(a.y); }

// Folds the sums v[7] of a system into its iteration scalars c; a system that stops has *active cleared.
//  FIN_INIT : v[2] = |r|^2: rr = rho = |r|^2, rr0 = rr, iters = 0, target2 = max(tau2*rr, floor2)
//  FIN_ALPHA: v[0..1] = <r0, v>: alpha = rho / <r0, v>
//  FIN_OMEGA_BETA: v[0..1] = <t, s>, v[2] = |t|^2, v[3..4] = <r0, t>, v[5..6] = <r0, s>:
//             omega = <t, s> / |t|^2, rho' = <r0, r> = <r0, s> - omega <r0, t> for the coming
//             r = s - omega t, beta = (rho'/rho)(alpha/omega)
//  FIN_OMEGA: v[0..1] = <t, s>, v[2] = |t|^2: omega
//  FIN_BETA : v[0..1] = <r0, r>, v[2] = |r|^2: beta from omega and rho' = <r0, r>, and FIN_STOP
//  FIN_STOP : v[2] = |r|^2: stop the system when rr <= target2, on breakdown, NaN or divergence (rr > 1e8 rr0)
//  FIN_NORM : rr = v[2] only
//  FIN_BB, FIN_BB_ADD: bb = v[2], bb += v[2]
//  CG on the normal equations (real scalars in .x), the sum in v[2]:
//  FIN_CG_RHO  : rho = |z|^2 (z = D^dag r), beta = 0 (the first direction is z)
//  FIN_CG_ALPHA: alpha = rho / |v|^2 (v = D^ p); breakdown if |v|^2 is not positive
//  FIN_CG_R    : rr = |r|^2; stop the system when rr <= target2, on NaN or divergence
//  FIN_CG_BETA : beta = |z|^2 / rho, rho = |z|^2
// status: 1 breakdown, 2 NaN or divergence.
LQ_DI void next_direction(SolverScal& c, double2 rho) {  // rho' = <r0, r> and beta = (rho'/rho)(alpha/omega)
  if (!finite2(rho)) {
    c.status = 2;
  } else if ((rho.x == 0.0 && rho.y == 0.0) || (c.omega.x == 0.0 && c.omega.y == 0.0)) {
    c.status = 1;
  } else {
    c.beta = cmul2(cdiv(rho, c.rho), cdiv(c.alpha, c.omega));
    c.rho = rho;
  }
}
LQ_DI void fin_update(int mode, const double* v, SolverScal& c, int* active, double tau2, double floor_rel2) {
  const double2 d = make_double2(v[0], v[1]);
  switch (mode) {
    case FIN_INIT:
      c.rr = c.rr0 = v[2];
      c.rho = make_double2(v[2], 0.0);
      c.iters = 0;
      c.status = 0;
      c.target2 = fmax(tau2 * v[2], floor_rel2 * c.bb);
      if (!(v[2] > c.target2)) *active = 0;
      if (!isfinite(v[2])) {
        c.status = 2;
        *active = 0;
      }
      break;
    case FIN_ALPHA:
      if (!finite2(d) || (d.x == 0.0 && d.y == 0.0)) {
        c.status = 1;
        *active = 0;
      } else {
        c.alpha = cdiv(c.rho, d);
      }
      break;
    case FIN_OMEGA:
    case FIN_OMEGA_BETA:
      c.beta = make_double2(0.0, 0.0);
      if (!(v[2] > 0.0) || !isfinite(v[2])) {
        c.omega = make_double2(0.0, 0.0);
        c.status = 1;
        break;
      }
      c.omega = make_double2(d.x / v[2], d.y / v[2]);
      if (mode == FIN_OMEGA_BETA) {
        const double2 w = cmul2(c.omega, make_double2(v[3], v[4]));
        next_direction(c, make_double2(v[5] - w.x, v[6] - w.y));
      }
      break;
    case FIN_BETA:
      if (c.status == 0) next_direction(c, d);
      // fall through
    case FIN_STOP:
      c.iters += 1;
      c.rr = v[2];
      if (!isfinite(v[2]) || c.status == 2 || v[2] > 1e8 * c.rr0) {
        c.status = 2;
        *active = 0;
      } else if (v[2] <= c.target2 || c.status == 1) {
        *active = 0;
      }
      break;
    case FIN_NORM:
      c.rr = v[2];
      break;
    case FIN_BB:
      c.bb = v[2];
      break;
    case FIN_BB_ADD:
      c.bb += v[2];
      break;
    case FIN_CG_RHO:
      c.rho = make_double2(v[2], 0.0);
      c.beta = make_double2(0.0, 0.0);
      break;
    case FIN_CG_ALPHA:
      if (!(v[2] > 0.0) || !isfinite(v[2]) || !(c.rho.x > 0.0)) {
        c.status = 1;
        *active = 0;
      } else {
        c.alpha = make_double2(c.rho.x / v[2], 0.0);
      }
      break;
    case FIN_CG_R:
      c.iters += 1;
      c.rr = v[2];
      if (!isfinite(v[2]) || v[2] > 1e8 * c.rr0) {
        c.status = 2;
        *active = 0;
      } else if (v[2] <= c.target2) {
        *active = 0;
      }
      break;
    case FIN_CG_BETA:
      if (!(c.rho.x > 0.0) || !isfinite(v[2])) {
        c.status = 1;
        *active = 0;
      } else {
        c.beta = make_double2(v[2] / c.rho.x, 0.0);
        c.rho = make_double2(v[2], 0.0);
      }
      break;
  }
}

// Arguments of finish_last: mode FIN_NONE leaves the partials to the caller.
struct FinArgs {
  int mode;
  int* active;
  SolverScal* sc;
  unsigned* count;  // one per system, zero between launches
};

// Called by every thread of each of the nb blocks of system s once its partial is stored by warp 0:
// the last block to arrive adds the partials (NQ values from slot Q0, PW doubles apart) and updates the
// system's scalars.
template <int NQ, int Q0, int PW>
LQ_DI void finish_last(const FinArgs& f, const double* partial, int nb, int s) {
  __shared__ int last;
  if (threadIdx.x < 32) {
    __threadfence();
    __syncwarp();
  }
  if (threadIdx.x == 0) {
    last = atomicAdd(f.count + s, 1u) == (unsigned)(nb - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v[7] = {0.0};
  block_sum_partials<NQ, PW>(partial + Q0, nb, v + Q0);
  if (threadIdx.x != 0) return;
  f.count[s] = 0;
  SolverScal c = f.sc[s];
  fin_update(f.mode, v, c, f.active + s, 0.0, 0.0);
  f.sc[s] = c;
}

}  // namespace lq
