// FP64-accurate stencil in fixed-point integer arithmetic.
//
// The FP64 pipe of this GPU issues 2 fused multiply-adds per clock and SM, its integer pipe 64
// multiply-adds 32 x 32 + 64 bits (measured, both): a product of two 57-bit numbers in three of the
// latter costs a tenth of a DFMA.  The operator is a short sum of products of numbers whose size
// is bounded (links: |U| <= 1; a spinor or a clover block: its largest entry), which is where fixed
// point is as good as floating point, so the FP64 operator of the solvers runs here:
//
//   * a spinor is 24 integers q, |q| <= 2^57, and one exponent: psi_k = q_k 2^(E - 1079), E the largest
//     biased FP64 exponent of its 24 components.  Components of the largest binade and the four
//     below it keep all 53 bits; a smaller one is rounded at 2^-58 of the largest, a thirtieth of
//     what one FP64 rounding of a sum with the largest costs;
//   * a link entry is q 2^-58; a clover block (of 6 x 6) 36 integers with an exponent of its own;
//   * q = q1 2^29 + q0 with |q0| <= 2^28 (limbs: an int2, so a complex number is an int4 of the
//     size of its FP64 form).  A product is q1 p1 2^58 + (q1 p0 + q0 p1) 2^29; q0 p0 is below 2^-57 of the
//     full scale and left out.  Both partial sums of a row (at most 24 products) fit 64 bits;
//   * the eight hops of a site are added as 64-bit integers, each shifted to the largest exponent
//     of the eight neighbours, and the result is rounded to FP64 once.
//
// Error against long double over random fields, D, open and periodic, with and without clover: 1.9 to 2.2e-16 of the
// 2-norm, FP64 sums 2.1 to 2.7e-16.  Inputs and results keep denormals; a non-finite
// component makes its spinor and every result that it enters NaN.
//
// Bound by latency at 12 warps an SM: issue slots 38% used (three multiply-adds of 64 bits a product, then shifts, negations
// and conversions), waits for loads and for the multiply-adds' results in front.  32 x 16^3 with clover, 12 slabs of
// 14 slices: A y - D_hop x / 4 takes 683 us on the FP64 pipe, 260 us so.  Four blocks an SM (126 registers, spilled)
// instead of three: 244 us there, but 1282 instead of 1203 us on 16 x 24^3 with 24 systems; two: 246 and 1630 us.  The
// hops' words through shared memory as in the FP32 stencil: 264 and 1355 us with four blocks, 235 and 1505 with mad_wide().
#pragma once

#include "dslash.cuh"
#include "internal.h"

namespace lq {

constexpr int FX_BLOCKS = 3;  // blocks of 128 threads per SM

struct cl {  // a complex number in limbs
  int r1, r0, i1, i0;
};
struct cll {  // a complex 64-bit integer
  long long re, im;
};

// v 2^-s rounded, |s| small when negative
LQ_DI long long fx_shift(long long v, int s) {
  if (s <= 0) return v << -s;
  return s < 63 ? (v + (1ll << (s - 1))) >> s : 0ll;
}

LQ_DI cl as_cl(int4 v) { return cl{v.x, v.y, v.z, v.w}; }

// (hh, cr) += a b in limbs.  In C++ and not with mad_wide(): the instructions that the compiler makes of it are more, but
// it orders them better between the loads (16 x 24^3, 24 systems, D_hop alone: 1.09 ms, with mad_wide 1.62 ms).
LQ_DI void fx_mac(long long& hh, long long& cr, int a1, int a0, int b1, int b0) {
  hh += (long long)a1 * b1;
  cr += (long long)a1 * b0;
  cr += (long long)a0 * b1;
}
// a + sg (I ? i b : b), sg = +-1
template <bool I>
LQ_DI cl cl_add(cl a, cl b, int sg) {
  if (I) return cl{a.r1 - sg * b.i1, a.r0 - sg * b.i0, a.i1 + sg * b.r1, a.i0 + sg * b.r0};
  return cl{a.r1 + sg * b.r1, a.r0 + sg * b.r0, a.i1 + sg * b.i1, a.i0 + sg * b.i0};
}
// acc += (neg ? - : +) (I ? i w : w), neg = 0 or -1
template <bool I>
LQ_DI void cll_add(cll& acc, cll w, long long neg) {
  const long long x = (w.re ^ neg) - neg, y = (w.im ^ neg) - neg;
  acc.re += I ? -y : x;
  acc.im += I ? x : y;
}

// Two threads work on a site.  Thread `sp` (0, 1) transports spin sp of each hop's half spinor and
// so reads spins sp and one of 2, 3 of the neighbour; it collects
//   U  the hop sum's spin sp,
//   LA its part of spin 2 + sp (directions 0 and 3), LB that of spin 3 - sp (directions 1 and 2).
// The spin of the half spinor of (1 + S g_mu) psi is psi_sp + c psi_q, c = -S, -S i, eps S, eps S i for mu = 0..3
// (q = 2 + sp for mu = 0, 3, else 3 - sp; eps = -1 for sp = 0, +1 for sp = 1), and the transported spin
// w enters spin q with the factor -S, S i, eps S, -eps S i.
struct FxSum {
  cll u[3], la[3], lb[3];
};
struct FxRaw {
  int4 a[3], b[3];  // the two spins read
};

template <int K>
LQ_DI void fx_fetch(FxRaw& r, const int4* in, int n, int q, int sp) {
  constexpr int MU = K >> 1;
  const int4* p = in + q + 3 * sp * n;
  const int4* o = in + q + (MU == 0 || MU == 3 ? 6 + 3 * sp : 9 - 3 * sp) * n;
#pragma unroll
  for (int c = 0; c < 3; c++) r.a[c] = __ldg(p + c * n);
#pragma unroll
  for (int c = 0; c < 3; c++) r.b[c] = __ldg(o + c * n);
}

// Hop K from its raw words, shifted right by sh.
template <bool DAG, int K>
LQ_DI void fx_apply(FxSum& A, const FxRaw& r, const FieldPtrs& f, int Vh, const HopTgt& t, int sp, int sh) {
  constexpr int MU = K >> 1;
  constexpr bool FWD = (K & 1) == 0;
  constexpr int SF = DAG ? +1 : -1;
  constexpr int S = FWD ? SF : -SF;
  const int eps = 2 * sp - 1;
  const int4* ub = f.U64 + (t.pl * 4 + MU) * 9 * Vh + t.cl;
  int4 u[9];
#pragma unroll
  for (int k = 0; k < 9; k++) u[k] = __ldg(ub + k * Vh);
  cl h[3];
#pragma unroll
  for (int c = 0; c < 3; c++)
    h[c] = cl_add<MU == 1 || MU == 3>(as_cl(r.a[c]), as_cl(r.b[c]), MU < 2 ? -S : eps * S);
#pragma unroll
  for (int a = 0; a < 3; a++) {
    long long hr = 0, cr = 1ll << 28, hi = 0, ci = 1ll << 28;  // (the halves round the shift below)
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const cl e = as_cl(u[FWD ? 3 * a + c : 3 * c + a]), v = h[c];
      // u h (forward) or conj(u) h
      const int p1 = FWD ? -e.i1 : e.i1, p0 = FWD ? -e.i0 : e.i0;
      fx_mac(hr, cr, v.r1, v.r0, e.r1, e.r0);
      fx_mac(hr, cr, v.i1, v.i0, p1, p0);
      fx_mac(hi, ci, v.i1, v.i0, e.r1, e.r0);
      fx_mac(hi, ci, v.r1, v.r0, -p1, -p0);
    }
    cll w = {(hr + (cr >> 29)) >> sh, (hi + (ci >> 29)) >> sh};
    if (MU == 0 && t.w < 0.f) w = {-w.re, -w.im};  // antiperiodic wrap
    cll_add<false>(A.u[a], w, 0);
    if (MU == 0) cll_add<false>(A.la[a], w, S > 0 ? -1 : 0);
    if (MU == 1) cll_add<true>(A.lb[a], w, S > 0 ? 0 : -1);
    if (MU == 2) cll_add<false>(A.lb[a], w, (long long)(S > 0 ? sp - 1 : -sp));
    if (MU == 3) cll_add<true>(A.la[a], w, (long long)(S > 0 ? -sp : sp - 1));
  }
}

LQ_DI cll cll_swap(cll v) {  // the other thread of the site's
  return {__shfl_xor_sync(0xffffffffu, v.re, 1), __shfl_xor_sync(0xffffffffu, v.im, 1)};
}

// Sum of the eight hops at output site cb: D_hop psi = acc 2^(E - FX_BIAS), of which thread sp receives
// chirality block sp (spins 2 sp, 2 sp + 1); bad: a neighbour is not finite.  All threads of a warp call it.
template <bool DAG>
LQ_DI void fx_hop_sum(cll (&acc)[6], int& E, bool& bad, const Geom& g, const SysDesc& sd, const FieldPtrs& f, int pout,
                      int cb, int j, int sp, const int4* in, const int* ine) {
  int x[4];
  eo_coords(g, cb, pout, x);
  const HopTgt t[8] = {hop_target<0>(g, sd, pout, cb, j, x), hop_target<1>(g, sd, pout, cb, j, x),
                       hop_target<2>(g, sd, pout, cb, j, x), hop_target<3>(g, sd, pout, cb, j, x),
                       hop_target<4>(g, sd, pout, cb, j, x), hop_target<5>(g, sd, pout, cb, j, x),
                       hop_target<6>(g, sd, pout, cb, j, x), hop_target<7>(g, sd, pout, cb, j, x)};
  int e[8];
#pragma unroll
  for (int k = 0; k < 8; k++) e[k] = __ldg(ine + t[k].q);
  FxRaw r0, r1;
  fx_fetch<0>(r0, in, sd.n, t[0].q, sp);
  E = 1;
  bad = false;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const bool on = k >= 2 || t[k].w != 0.f;  // only time hops are dropped
    if (on && e[k] >= FX_NAN) {
      bad = true;
      e[k] = 1;
    }
    if (on) E = max(E, e[k]);
  }
  FxSum A;
#pragma unroll
  for (int k = 0; k < 3; k++) A.u[k] = A.la[k] = A.lb[k] = {0, 0};
  // the next hop's words are loaded before a hop is computed
  fx_fetch<1>(r1, in, sd.n, t[1].q, sp);
  if (t[0].w != 0.f) fx_apply<DAG, 0>(A, r0, f, g.Vh, t[0], sp, min(E - e[0], 63));
  fx_fetch<2>(r0, in, sd.n, t[2].q, sp);
  if (t[1].w != 0.f) fx_apply<DAG, 1>(A, r1, f, g.Vh, t[1], sp, min(E - e[1], 63));
  fx_fetch<3>(r1, in, sd.n, t[3].q, sp);
  fx_apply<DAG, 2>(A, r0, f, g.Vh, t[2], sp, min(E - e[2], 63));
  fx_fetch<4>(r0, in, sd.n, t[4].q, sp);
  fx_apply<DAG, 3>(A, r1, f, g.Vh, t[3], sp, min(E - e[3], 63));
  fx_fetch<5>(r1, in, sd.n, t[5].q, sp);
  fx_apply<DAG, 4>(A, r0, f, g.Vh, t[4], sp, min(E - e[4], 63));
  fx_fetch<6>(r0, in, sd.n, t[6].q, sp);
  fx_apply<DAG, 5>(A, r1, f, g.Vh, t[5], sp, min(E - e[5], 63));
  fx_fetch<7>(r1, in, sd.n, t[7].q, sp);
  fx_apply<DAG, 6>(A, r0, f, g.Vh, t[6], sp, min(E - e[6], 63));
  fx_apply<DAG, 7>(A, r1, f, g.Vh, t[7], sp, min(E - e[7], 63));
  // thread 0 takes spins 0 (its U), 1 (the other's U); thread 1 spins 2 (the other's LA, its LB), 3 (its LA, the
  // other's LB)
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const cll o1 = cll_swap(sp ? A.u[a] : A.la[a]), o2 = cll_swap(A.lb[a]);
    acc[a] = sp ? cll{o1.re + A.lb[a].re, o1.im + A.lb[a].im} : A.u[a];
    acc[3 + a] = sp ? cll{A.la[a].re + o2.re, A.la[a].im + o2.im} : o1;
  }
}

// Largest exponent of N FP64 complex numbers (at least 1), FX_NAN if one is not finite.
template <int N>
LQ_DI int fx_max_exponent(const cx<double>* v) {
  int m = 1;
#pragma unroll
  for (int k = 0; k < N; k++) m = max(m, max(fx_exponent(v[k].re), fx_exponent(v[k].im)));
  return m == 2047 ? FX_NAN : m;
}
LQ_DI cl fx_limbs(cx<double> v, int E) {
  cl r;
  fx_split(fx_of(v.re, E), r.r1, r.r0);
  fx_split(fx_of(v.im, E), r.i1, r.i0);
  return r;
}

// out = B in for a packed Hermitian 6 x 6 block of limbs (18 int4: two reals each): the integers HH + CR 2^-29,
// in units of 2^58 of the product of the two scales.
LQ_DI void fx_herm6(const int4* base, int Vh, int cb, const cl in[6], cll out[6]) {
  int2 d[6];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int4 v = __ldg(base + k * Vh + cb);
    d[2 * k] = make_int2(v.x, v.y);
    d[2 * k + 1] = make_int2(v.z, v.w);
  }
  long long hr[6], cr[6], hi[6], ci[6];
#pragma unroll
  for (int r = 0; r < 6; r++) {
    hr[r] = hi[r] = 0;
    cr[r] = ci[r] = 1ll << 28;  // rounds the shift below
    fx_mac(hr[r], cr[r], d[r].x, d[r].y, in[r].r1, in[r].r0);
    fx_mac(hi[r], ci[r], d[r].x, d[r].y, in[r].i1, in[r].i0);
  }
  int q = 3;
#pragma unroll
  for (int r = 1; r < 6; r++)
#pragma unroll
    for (int c = 0; c < r; c++) {
      const cl e = as_cl(__ldg(base + q * Vh + cb));  // B[r][c]; B[c][r] = conj
      q++;
      fx_mac(hr[r], cr[r], e.r1, e.r0, in[c].r1, in[c].r0);
      fx_mac(hr[r], cr[r], -e.i1, -e.i0, in[c].i1, in[c].i0);
      fx_mac(hi[r], ci[r], e.r1, e.r0, in[c].i1, in[c].i0);
      fx_mac(hi[r], ci[r], e.i1, e.i0, in[c].r1, in[c].r0);
      fx_mac(hr[c], cr[c], e.r1, e.r0, in[r].r1, in[r].r0);
      fx_mac(hr[c], cr[c], e.i1, e.i0, in[r].i1, in[r].i0);
      fx_mac(hi[c], ci[c], e.r1, e.r0, in[r].i1, in[r].i0);
      fx_mac(hi[c], ci[c], -e.i1, -e.i0, in[r].r1, in[r].r0);
    }
#pragma unroll
  for (int r = 0; r < 6; r++) out[r] = {hr[r] + (cr[r] >> 29), hi[r] + (ci[r] >> 29)};
}
// the same with a multiple d of the unit matrix
LQ_DI void fx_diag6(int2 d, const cl in[6], cll out[6]) {
#pragma unroll
  for (int r = 0; r < 6; r++) {
    long long hr = 0, cr = 1ll << 28, hi = 0, ci = 1ll << 28;
    fx_mac(hr, cr, d.x, d.y, in[r].r1, in[r].r0);
    fx_mac(hi, ci, d.x, d.y, in[r].i1, in[r].i0);
    out[r] = {hr + (cr >> 29), hi + (ci >> 29)};
  }
}

// Arguments of the fixed-point kernels: HopArgs with the hop input x in limbs (xe: exponents), the factors
// alpha, beta, gamma (+-2^k) as sign and k, and diag (or 1/diag) in limbs.
struct FxArgs {
  HopArgs a;
  const int4* x;
  const int* xe;
  int ka, kb, kg;  // exponents of |alpha|, |beta|, |gamma|
  int sa, sb, sg;  // 1: negative
  int2 d;          // diagonal without clover, value d 2^(de - FX_BIAS)
  int de;
};

// Chirality block sp of a system's FP64 vector at site j.  NC: the kernel does not write the vector.
template <bool NC = true>
LQ_DI void fx_load6(cx<double> v[6], const void* pool, const SysDesc& sd, int j, int sp) {
  const double2* p = (const double2*)pool + sd.off * 12 + (long long)6 * sp * sd.n + j;
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const double2 w = NC ? __ldg(p + k * sd.n) : p[k * sd.n];
    v[k] = {w.x, w.y};
  }
}
LQ_DI void fx_store6(void* pool, const SysDesc& sd, int j, int sp, const cx<double> v[6]) {
  double2* p = (double2*)pool + sd.off * 12 + (long long)6 * sp * sd.n + j;
#pragma unroll
  for (int k = 0; k < 6; k++) p[k * sd.n] = make_double2(v[k].re, v[k].im);
}
// tot += (neg ? - : +) v 2^-s rounded
LQ_DI void fx_accum(cll& tot, cll v, int s, int neg) {
  const cll r = {fx_shift(v.re, s), fx_shift(v.im, s)};
  tot.re += neg ? -r.re : r.re;
  tot.im += neg ? -r.im : r.im;
}

constexpr int FX_SITES = 64;  // sites of a 128-thread block, two threads each
LQ_DI int fx_site(const HopArgs& a, int by) {
  return site_of_block(a.tblk, a.g.S3h, by >> 1, (by & 1) * FX_SITES + (int)(threadIdx.x >> 1));
}

// out = beta A(y) + alpha D_hop x + gamma z with k_hop_lin's reductions, y, z, w, out in FP64; out may be y.
template <bool DAG, bool CLOV, int RED, int EPI>
__global__ void __launch_bounds__(128, FX_BLOCKS) k_fx_lin(FxArgs m) {
  const HopArgs& a = m.a;
  int s, by;
  grid_pos_tiled((int)blockIdx.x, a.nsys, a.nby, a.tile, s, by);
  if (s >= a.nsys) return;
  if (a.active && !a.active[s]) return;
  const SysDesc sd = a.sys[s];
  const int nblk = (sd.n + FX_SITES - 1) / FX_SITES;
  if (by >= nblk) return;
  const int sp = threadIdx.x & 1;
  int j = fx_site(a, by);
  const bool valid = j < sd.n;
  if (!valid) j = sd.n - 1;  // in range; nothing is stored for it
  const FieldPtrs f = a.fields[sd.field];
  const int cb = sd.cb0 + j;
  cll acc[6];
  int E = 1;
  bool bad = false;
  fx_hop_sum<DAG>(acc, E, bad, a.g, sd, f, a.pout, cb, j, sp, m.x + sd.off * 12, m.xe + sd.off);
  // The terms' last-place exponents e1, e2, e3 and the sum's, et: |acc| < 2^63, |A y| < 2^60 (2^56 for a multiple
  // of 1) and |z| < 2^57 leave the sum of the three below 2^63 in units of 2^et.
  const int e1 = E - FX_BIAS + m.ka;
  int et = e1 + 3, e2 = 0, e3 = 0;
  cx<double> yv[6], zv[6];
  int ey = 1, ez = 1;
  if ((EPI & EPI_Y) || RED == RED_TS) fx_load6<false>(yv, a.y, sd, j, sp);
  if (EPI & EPI_Z) fx_load6(zv, a.z, sd, j, sp);
  if (EPI & EPI_Y) {
    ey = fx_max_exponent<6>(yv);
    if (ey == FX_NAN) {
      bad = true;
      ey = 1;
    }
    const int ea = CLOV ? __ldg(f.A64e + (a.pout * 2 + sp) * a.g.Vh + cb) : m.de;
    e2 = ea + ey - 2 * FX_BIAS + 58 + m.kb;
    et = max(et, e2 - (CLOV ? 1 : 4));
  }
  if (EPI & EPI_Z) {
    ez = fx_max_exponent<6>(zv);
    if (ez == FX_NAN) {
      bad = true;
      ez = 1;
    }
    e3 = ez - FX_BIAS + m.kg;
    et = max(et, e3 - 3);
  }
  cll tot[6];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    tot[k] = {0, 0};
    fx_accum(tot[k], acc[k], et - e1, m.sa);
  }
  if (EPI & EPI_Z) {
#pragma unroll
    for (int k = 0; k < 6; k++) fx_accum(tot[k], cll{fx_of(zv[k].re, ez), fx_of(zv[k].im, ez)}, et - e3, m.sg);
  }
  if (EPI & EPI_Y) {
    cl yl[6];
    cll ay[6];
#pragma unroll
    for (int k = 0; k < 6; k++) yl[k] = fx_limbs(yv[k], ey);
    if (CLOV)
      fx_herm6(f.A64 + (a.pout * 36 + 18 * sp) * a.g.Vh, a.g.Vh, cb, yl, ay);
    else
      fx_diag6(m.d, yl, ay);
#pragma unroll
    for (int k = 0; k < 6; k++) fx_accum(tot[k], ay[k], et - e2, m.sb);
  }
  bad = __shfl_xor_sync(0xffffffffu, (int)bad, 1) || bad;  // either block's
  cx<double> res[6];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    res[k] = {fx_to_double(tot[k].re, et), fx_to_double(tot[k].im, et)};
    if (bad) res[k] = {nan(""), nan("")};
  }
  double red[red_count(RED)] = {0};
  if (valid) {
    fx_store6(a.out, sd, j, sp, res);
    if (RED != RED_NONE) {
      cx<double> wv[6];
      if (RED == RED_DOT_W) fx_load6(wv, a.w, sd, j, sp);
      red_add<RED, 6, double>(red, res, yv, wv);
    }
  }
  if (RED != RED_NONE) red_store<RED, double>(red, a, s, by, nblk);
}

// out = A^{-1} (alpha D_hop x + beta y) on even sites (terms per EPI), y and out in FP64.
template <bool DAG, bool CLOV, int EPI>
__global__ void __launch_bounds__(128, FX_BLOCKS) k_fx_clinv(FxArgs m) {
  const HopArgs& a = m.a;
  int s, by;
  grid_pos_tiled((int)blockIdx.x, a.nsys, a.nby, a.tile, s, by);
  if (s >= a.nsys) return;
  if (a.active && !a.active[s]) return;
  const SysDesc sd = a.sys[s];
  if (by * FX_SITES >= sd.n) return;
  const int sp = threadIdx.x & 1;
  int j = fx_site(a, by);
  const bool valid = j < sd.n;
  if (!valid) j = sd.n - 1;
  const FieldPtrs f = a.fields[sd.field];
  const int cb = sd.cb0 + j;
  cll tot[6];
  int et = 0;
  bool bad = false;
  if (EPI & EPI_X) {
    int E;
    fx_hop_sum<DAG>(tot, E, bad, a.g, sd, f, a.pout, cb, j, sp, m.x + sd.off * 12, m.xe + sd.off);
    et = E - FX_BIAS + m.ka;
    if (m.sa) {
#pragma unroll
      for (int k = 0; k < 6; k++) tot[k] = {-tot[k].re, -tot[k].im};
    }
  }
  if (EPI & EPI_Y) {
    cx<double> yv[6];
    fx_load6(yv, a.y, sd, j, sp);
    int ey = fx_max_exponent<6>(yv);
    if (ey == FX_NAN) {
      bad = true;
      ey = 1;
    }
    const int e2 = ey - FX_BIAS + m.kb, en = (EPI & EPI_X) ? max(et + 2, e2 - 3) : e2;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      if (EPI & EPI_X)
        tot[k] = {fx_shift(tot[k].re, en - et), fx_shift(tot[k].im, en - et)};
      else
        tot[k] = {0, 0};
      fx_accum(tot[k], cll{fx_of(yv[k].re, ey), fx_of(yv[k].im, ey)}, en - e2, m.sb);
    }
    et = en;
  }
  // back to limbs of 57 bits: the largest magnitude's leading bit to bit 56
  unsigned long long mag = 0;
#pragma unroll
  for (int k = 0; k < 6; k++) mag |= (unsigned long long)((tot[k].re ^ (tot[k].re >> 63)) | (tot[k].im ^ (tot[k].im >> 63)));
  const int c = mag ? 7 - __clzll((long long)mag) : 0;  // right shift (negative: left)
  cl in[6];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    fx_split(fx_shift(tot[k].re, c), in[k].r1, in[k].r0);
    fx_split(fx_shift(tot[k].im, c), in[k].i1, in[k].i0);
  }
  cll o[6];
  int ea = m.de;
  if (CLOV) {
    ea = __ldg(f.Ai64e + sp * a.g.Vh + cb);
    fx_herm6(f.Ai64 + 18 * sp * a.g.Vh, a.g.Vh, cb, in, o);
  } else {
    fx_diag6(m.d, in, o);
  }
  const int eo = ea - FX_BIAS + et + c + 58;
  bad = __shfl_xor_sync(0xffffffffu, (int)bad, 1) || bad;  // either block's
  cx<double> res[6];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    res[k] = {fx_to_double(o[k].re, eo), fx_to_double(o[k].im, eo)};
    if (bad) res[k] = {nan(""), nan("")};
  }
  if (valid) fx_store6(a.out, sd, j, sp, res);
}

}  // namespace lq

// k_fx_lin / k_fx_clinv for a (reduction, epilogue) pair, in translation units of their own (fx_lin.cu,
// fx_clinv.cu); -1 for a pair that is not built.
namespace lq {
// FP64 vectors of a batch to limbs (out may be in) and exponents
void to_fx_launch(dim3 gr, int nsys, const SysDesc* sys, const int* active, const double2* in, int4* out, int* oute,
                  cudaStream_t st);
void dslash_in_launch(const Geom& g, const SysDesc& s, const double2* in, void* out, SysDesc* d_sys, void** d_ptr,
                      double2* ve, double2* vo, int4* le, int4* lo, int* ee, int* eo, cudaStream_t st);
int fx_lin_launch(bool dag, bool clov, int red, int epi, dim3 gr, const FxArgs& m, cudaStream_t st);
int fx_clinv_launch(bool dag, bool clov, int epi, dim3 gr, const FxArgs& m, cudaStream_t st);
}
