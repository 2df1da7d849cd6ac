// Quark-line projection (Sec. 3.3 eqs. projection, quark_prop_II_proj) and
// the inverse-iteration projection vectors of Sec. 6:
//   * orthonormalisation of N FP64 complex columns by Cholesky QR, twice
//     (Gram matrix G = V^dag V, G = L L^dag, W = V L^{-dag}; the second pass
//     restores orthogonality lost to cond(V)^2 in the first);
//   * slice extraction with P_+ = (1 + gamma_0)/2 and slice sources;
//   * the projected case-II propagator  -sum_i eta_i(y) xi_i(x)^dag.
#include "internal.h"

using namespace lq;

#define RC(call)            \
  do {                      \
    int r_ = (call);        \
    if (r_ != 0) return r_; \
  } while (0)

namespace {

constexpr int GT = 8;    // Gram / apply column tile
constexpr int GR = 32;   // rows per shared-memory stage of the Gram kernel

int launched_here() {
  lq_count_launch();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    lq_set_error(std::string("kernel launch: ") + cudaGetErrorString(e));
    return LQCD_ECUDA;
  }
  return 0;
}

LQ_DI double2 cmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

// Element (row r, column k) of a column matrix; r runs over the segments.
LQ_DI double2 cm_get(const ColMat& m, long long r, int k) {
  if (k >= m.ncol) return make_double2(0.0, 0.0);
  if (r < m.rows[0]) return m.p[0][(long long)k * m.ld[0] + r];
  r -= m.rows[0];
  if (m.nseg > 1 && r < m.rows[1]) return m.p[1][(long long)k * m.ld[1] + r];
  return make_double2(0.0, 0.0);
}

// Dot products of FP64 numbers in 64-bit integers (fxnum.cuh; the integer pipe does 32 times the FP64
// pipe's multiply-adds).  A vector's entries are q 2^(E - px_bias<X>), |q| < 2^(55 + X), E their largest exponent, in
// limbs q = q1 2^28 + q0; the sums of q1 p1 and of q1 p0 + q0 p1 over px_modes<X> complex products fit 64 bits.  The
// propagator takes X = 0, whose 120 modes need one sum, or more for fewer modes.  The orthonormalisation takes X = 1: its second
// pass multiplies by nearly 1, where FP64 hardly rounds (error of 24 columns against long double: 1.5e-16 with
// FP64 sums, 1.4e-16 with X = 1, 2.6e-16 with X = 0).
template <int X>
constexpr int px_bias = 1077 + X;
template <int X>
constexpr int px_modes = X ? 32 : 120;
template <int X>
LQ_DI void px_split(double x, int E, int& q1, int& q0) {
  const long long q = fx_of(x, E + 2 - X);
  q0 = (int)((unsigned)q << 4) >> 4;
  q1 = (int)((q - q0) >> 28);
}
LQ_DI void px_mac(long long& hh, long long& cr, int a1, int a0, int b1, int b0) {
  mad_wide(hh, a1, b1);
  mad_wide(cr, a1, b0);
  mad_wide(cr, a0, b1);
}

// (hr, cr, hi, ci) += conj(a) b
LQ_DI void px_conj_mac(long long (&t)[4], int4 a, int4 b) {
  px_mac(t[0], t[1], a.x, a.y, b.x, b.y);
  px_mac(t[0], t[1], a.z, a.w, b.z, b.w);
  px_mac(t[2], t[3], a.x, a.y, b.z, b.w);
  px_mac(t[2], t[3], -a.z, -a.w, b.x, b.y);
}
template <bool DEN>
LQ_DI double2 px_value(const long long (&t)[4], int e) {
  return make_double2(fx_sum<28, DEN>(t[0], t[1], e), fx_sum<28, DEN>(t[2], t[3], e));
}
template <int X>
LQ_DI int4 px_limbs(double2 v, int E) {
  int4 q;
  px_split<X>(v.x, E, q.x, q.y);
  px_split<X>(v.y, E, q.z, q.w);
  return q;
}

// Partial Gram matrices: block (tile pair (ta <= tb), split z) sums
// conj(V[r][a]) V[r][b] over its row chunk into part[z][a][b].
//
// Fixed-point products (px_*), GF rows at a time: a first look at the rows' 2 x 8 columns gives each its
// exponent, then the four groups of 64 threads, one thread a pair (a, b), sum every fourth row and the sums of
// GS stages are added up in FP64.  8 x 8 pairs a tile waste little of the triangle (24 columns: 300 of 384 pairs used, 16 x 16
// tiles 300 of 768).  24 columns of 2.65 M rows: 13.6 ms with FP64 sums in 16 x 16 tiles, 3.7 ms so.
constexpr int GS = 4 * px_modes<1> / GR;
constexpr int GF = 4 * GS * GR;
__global__ void __launch_bounds__(256) k_gram(ColMat m, long long chunk, int npad, const int2* pairs, double2* part) {
  __shared__ int4 sa[GR][GT], sb[GR][GT];
  __shared__ int ex[2 * GT];
  __shared__ double2 red[3][GT * GT];
  const int2 tp = pairs[blockIdx.x];
  const int a0 = tp.x * GT, b0 = tp.y * GT;
  const int g = threadIdx.x >> 6, pr = threadIdx.x & 63, ty = pr >> 3, tx = pr & 7;
  const long long R = m.rows[0] + (m.nseg > 1 ? m.rows[1] : 0);
  const long long r_lo = (long long)blockIdx.y * chunk;
  const long long r_hi = r_lo + chunk < R ? r_lo + chunk : R;
  auto column = [&](int c) { return c < GT ? a0 + c : b0 + c - GT; };
  double2 acc = make_double2(0.0, 0.0);
  for (long long rf = r_lo; rf < r_hi; rf += GF) {
    __syncthreads();
    if (threadIdx.x < 2 * GT) ex[threadIdx.x] = 1;
    __syncthreads();
    for (int e = threadIdx.x; e < GF * 2 * GT; e += 256) {  // GF % 32 == 0: a warp reads one column
      const int c = e / GF;
      const long long r = rf + e - c * GF;
      int x = 1;
      if (r < r_hi) {
        const double2 v = cm_get(m, r, column(c));
        x = max(fx_exponent(v.x), fx_exponent(v.y));
      }
      x = __reduce_max_sync(0xffffffffu, x);
      if ((threadIdx.x & 31) == 0) atomicMax(&ex[c], x);
    }
    long long t[4] = {0, 0, 0, 0};
    auto flush = [&]() {
      const double2 v = px_value<false>(t, ex[ty] + ex[GT + tx] - 2 * px_bias<1> + 56);
      acc.x += v.x;
      acc.y += v.y;
      t[0] = t[1] = t[2] = t[3] = 0;
    };
    int stage = 0;
    for (long long r0 = rf; r0 < rf + GF && r0 < r_hi; r0 += GR) {
      if (stage++ == GS) {
        flush();
        stage = 1;
      }
      __syncthreads();
      for (int e = threadIdx.x; e < GR * 2 * GT; e += 256) {
        const int rr = e % GR, c = e / GR;
        const long long r = r0 + rr;
        const int4 q = px_limbs<1>(r < r_hi ? cm_get(m, r, column(c)) : make_double2(0.0, 0.0), ex[c]);
        if (c < GT) sa[rr][c] = q;
        else sb[rr][c - GT] = q;
      }
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < GR / 4; rr++) px_conj_mac(t, sa[4 * rr + g][ty], sb[4 * rr + g][tx]);
    }
    flush();
    if (ex[ty] == 2047 || ex[GT + tx] == 2047) acc = make_double2(nan(""), nan(""));
  }
  if (g) red[g - 1][pr] = acc;
  __syncthreads();
  if (g) return;
  for (int k = 0; k < 3; k++) {
    acc.x += red[k][pr].x;
    acc.y += red[k][pr].y;
  }
  part[((long long)blockIdx.y * npad + a0 + ty) * npad + b0 + tx] = acc;
}

// G[a][b] = sum over splits, mirrored from the computed upper tiles.
__global__ void k_gram_reduce(const double2* part, int nsplit, int npad, int n, double2* G) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int a = t / n, b = t % n;
  const bool up = a / GT <= b / GT;
  const int i = up ? a : b, j = up ? b : a;
  double2 s = make_double2(0.0, 0.0);
  for (int z = 0; z < nsplit; z++) {
    const double2 v = part[((long long)z * npad + i) * npad + j];
    s.x += v.x;
    s.y += v.y;
  }
  G[(long long)a * n + b] = up ? s : make_double2(s.x, -s.y);
}

// One block: G = L L^dag in place (lower triangle), then Linv = L^{-1}.
// status = 1 when a pivot falls below 1e-14 of its column's squared norm
// (the column's part orthogonal to the previous ones is below 1e-7 of its
// norm: linearly dependent at FP64 precision for Cholesky QR).  cexp: the exponents of the columns' norms.  n <= 1024.
__global__ void __launch_bounds__(1024) k_chol_inv(double2* G, int n, double2* Linv, int* cexp, int* status) {
  __shared__ int bad;
  __shared__ double diag0[1024];
  if (threadIdx.x == 0) bad = 0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    diag0[k] = G[(long long)k * n + k].x;
    cexp[k] = fx_exponent(sqrt(diag0[k]));
  }
  __syncthreads();
  for (int k = 0; k < n; k++) {
    if (threadIdx.x == 0) {
      const double d = G[(long long)k * n + k].x;
      if (!(d > 1e-14 * diag0[k]) || !isfinite(d)) bad = 1;
      G[(long long)k * n + k] = make_double2(bad ? 1.0 : sqrt(d), 0.0);
    }
    __syncthreads();
    if (bad) break;
    const double piv = G[(long long)k * n + k].x;
    for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) {
      double2 v = G[(long long)i * n + k];
      G[(long long)i * n + k] = make_double2(v.x / piv, v.y / piv);
    }
    __syncthreads();
    const int m = n - k - 1;  // trailing block (i, j), k < j <= i < n
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      if (j > i) continue;
      const double2 li = G[(long long)i * n + k], lj = G[(long long)j * n + k];
      double2 g = G[(long long)i * n + j];
      // g -= li * conj(lj)
      g.x -= li.x * lj.x + li.y * lj.y;
      g.y -= li.y * lj.x - li.x * lj.y;
      G[(long long)i * n + j] = g;
    }
    __syncthreads();
  }
  if (bad) {
    if (threadIdx.x == 0) *status = 1;
    return;
  }
  // forward substitution, one column c of L^{-1} per thread
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    for (int i = 0; i < c; i++) Linv[(long long)i * n + c] = make_double2(0.0, 0.0);
    for (int i = c; i < n; i++) {
      double2 s = make_double2(i == c ? 1.0 : 0.0, 0.0);
      for (int j = c; j < i; j++) {
        const double2 t = cmul(G[(long long)i * n + j], Linv[(long long)j * n + c]);
        s.x -= t.x;
        s.y -= t.y;
      }
      const double d = G[(long long)i * n + i].x;
      Linv[(long long)i * n + c] = make_double2(s.x / d, s.y / d);
    }
  }
}

// W[r][k] = sum_{j <= k} V[r][j] conj(Linv[k][j])   (W = V L^{-dag}), a thread a row and GT columns k.
//
// Fixed-point products (px_*): column j of V has the exponent cx[j] of its norm, which the coefficients take off again, so
// that a sum over j has one scale, ek[k]; the row has the exponent er of its largest entry relative to the columns', so a small
// row keeps as many digits as a large one.  (A single W[r][k] far below its row's others does not: the coefficients'
// own errors, 2^-53 of the norms, are worth as much in it.)  24 columns of 2.65 M rows: 10.9
// ms with FP64 sums and 16 columns a thread, 4.1 ms so.
constexpr int AJ = px_modes<1>;
__global__ void __launch_bounds__(128) k_apply_rinv(ColMat in, ColMat out, const double2* Linv, const int* cexp, int n) {
  __shared__ int4 cf[AJ][GT];
  __shared__ int cx[1024], ek[GT];
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int k0 = blockIdx.y * GT;
  const long long R = in.rows[0] + (in.nseg > 1 ? in.rows[1] : 0);
  const int jend = min(n, k0 + GT);
  for (int j = threadIdx.x; j < jend; j += blockDim.x) cx[j] = cexp[j];
  if (threadIdx.x < GT) ek[threadIdx.x] = -10000;
  __syncthreads();
  int er = -10000;
  bool bad = false;
  if (r < R) {
#pragma unroll 4
    for (int j = 0; j < jend; j++) {
      const double2 v = cm_get(in, r, j);
      const int x = max(max(fx_exponent(v.x), fx_exponent(v.y)), 1);
      er = max(er, x - cx[j]);
      bad = bad || x == 2047;
    }
  }
  auto coefficient = [&](int j, int q) {  // conj(Linv[k0 + q][j])
    const int k = k0 + q;
    double2 c = make_double2(0.0, 0.0);
    if (k < n && j <= k) {
      const double2 l = Linv[(long long)k * n + j];
      c = make_double2(l.x, -l.y);
    }
    return c;
  };
  for (int e = threadIdx.x; e < jend * GT; e += blockDim.x) {
    const int j = e / GT, q = e % GT;
    const double2 c = coefficient(j, q);
    if (c.x != 0.0 || c.y != 0.0) atomicMax(&ek[q], max(fx_exponent(c.x), fx_exponent(c.y)) + cx[j]);
  }
  __syncthreads();
  double2 sum[GT];
  long long t[GT][4];
#pragma unroll
  for (int q = 0; q < GT; q++) {
    sum[q] = make_double2(0.0, 0.0);
    t[q][0] = t[q][1] = t[q][2] = t[q][3] = 0;
  }
  auto flush = [&]() {
#pragma unroll
    for (int q = 0; q < GT; q++) {
      const double2 v = px_value<true>(t[q], ek[q] + er - 2 * px_bias<1> + 56);
      sum[q].x += v.x;
      sum[q].y += v.y;
      t[q][0] = t[q][1] = t[q][2] = t[q][3] = 0;
    }
  };
  for (int j0 = 0; j0 < jend; j0 += AJ) {
    if (j0) {
      flush();
      __syncthreads();
    }
    for (int e = threadIdx.x; e < AJ * GT; e += blockDim.x) {
      const int jj = e / GT, q = e % GT;
      if (j0 + jj < jend) cf[jj][q] = px_limbs<1>(coefficient(j0 + jj, q), ek[q] - cx[j0 + jj]);
    }
    __syncthreads();
    if (r < R) {
      const int jn = min(AJ, jend - j0);
#pragma unroll 2
      for (int jj = 0; jj < jn; jj++) {
        const int4 v = px_limbs<1>(cm_get(in, r, j0 + jj), er + cx[j0 + jj]);
#pragma unroll
        for (int q = 0; q < GT; q++) {
          const int4 c = cf[jj][q];
          px_mac(t[q][0], t[q][1], v.x, v.y, c.x, c.y);
          px_mac(t[q][0], t[q][1], -v.z, -v.w, c.z, c.w);
          px_mac(t[q][2], t[q][3], v.x, v.y, c.z, c.w);
          px_mac(t[q][2], t[q][3], v.z, v.w, c.x, c.y);
        }
      }
    }
  }
  if (r >= R) return;
  flush();
  int sg = 0;
  long long rr = r;
  if (rr >= out.rows[0]) {
    rr -= out.rows[0];
    sg = 1;
  }
#pragma unroll
  for (int q = 0; q < GT; q++) {
    const int k = k0 + q;
    if (k < n) out.p[sg][(long long)k * out.ld[sg] + rr] = bad ? make_double2(nan(""), nan("")) : sum[q];
  }
}

// phi[s][site of slice g1][12] = P_+ v_s(x), x on slice g1 of system s
// (P_+ = (1 + gamma_0)/2: upper = (u - l)/2, lower = -upper in the chiral basis).
__global__ void __launch_bounds__(128) k_slice_plus(Geom g, int nsys, const SysDesc* sys, int g1, const double2* ve,
                                                    const double2* vo, double2* phi) {
  int s, by;
  grid_pos(nsys, s, by);
  const SysDesc sd = sys[s];
  const int S3 = 2 * g.S3h;
  const int i = by * blockDim.x + threadIdx.x;
  if (i >= S3) return;
  const int x3 = i % g.L[3], x2 = (i / g.L[3]) % g.L[2], x1 = i / (g.L[3] * g.L[2]);
  const int p = (g1 + x1 + x2 + x3) & 1;
  const long long nat = (long long)g1 * S3 + i;
  const int j = (int)(nat >> 1) - sd.cb0;
  const double2* v = (p == 0 ? ve : vo) + sd.off * 12 + j;
  double2* o = phi + ((long long)s * S3 + i) * 12;
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const double2 u = v[(long long)k * sd.n], l = v[(long long)(k + 6) * sd.n];
    const double2 h = make_double2(0.5 * (u.x - l.x), 0.5 * (u.y - l.y));
    o[k] = h;
    o[k + 6] = make_double2(-h.x, -h.y);
  }
}

// Source of system s: phi[ids[s]] on slice g1, zero elsewhere in its slab.
__global__ void __launch_bounds__(128) k_slice_source(Geom g, int nsys, const SysDesc* sys, const int* ids, int g1,
                                                      const double2* phi, double2* ve, double2* vo) {
  int s, by;
  grid_pos(nsys, s, by);
  const SysDesc sd = sys[s];
  const int j = by * blockDim.x + threadIdx.x;
  if (j >= sd.n) return;
  const int p = blockIdx.z;
  int x[4];
  eo_coords(g, sd.cb0 + j, p, x);
  const int S3 = 2 * g.S3h;
  double2* out = (p == 0 ? ve : vo) + sd.off * 12;
  if (x[0] == g1) {
    const int i = (x[1] * g.L[2] + x[2]) * g.L[3] + x[3];
    const double2* f = phi + ((long long)ids[s] * S3 + i) * 12;
#pragma unroll
    for (int k = 0; k < 12; k++) out[k * sd.n + j] = f[k];
  } else {
#pragma unroll
    for (int k = 0; k < 12; k++) out[k * sd.n + j] = make_double2(0.0, 0.0);
  }
}

// What k_proj_prop needs of a mode besides its limbs: the exponent r of its largest |xi_i(x)[b]|, and those of the twelve
// entries relative to r and to the columns' scales.
struct __align__(16) ProjMode {
  int r, pad;
  short d[12];
};
constexpr int PJ_NONE = -10000;  // exponent of a zero (two of them and an exponent of FP64 fit 16 bits)
template <int X>
constexpr int PJ_LOSS = 2 + X;
template <int X>
constexpr int PJ_MODES = X == 2 ? 15 : X == 1 ? 60 : 120;  // products whose 64-bit sums fit (below 16, 64 and 128)

LQ_DI int px_exponent(double2 v) { return max(max(fx_exponent(v.x), fx_exponent(v.y)), 1); }

// The scales of a thread's sums: E, the largest exponent(eta_i) + md[i].r, and the columns that need one of their own (bit b; also
// where the result may be a denormal number; bit 12: an eta_i is not finite), as E 2^13 + bits.
template <int X>
LQ_DI int pj_scan(int n, long long ld, const double2* col, const ProjMode* md, const int* xe) {
  int E = PJ_NONE, emax = 1;
  unsigned T[6];  // the largest exponent(eta_i) + exponent(xi_i[b]), relative to the columns' scales
#pragma unroll
  for (int k = 0; k < 6; k++) T[k] = 0x80008000u;
  auto add = [&](double2 v, int i) {
    const int e = px_exponent(v);
    const int4* m = reinterpret_cast<const int4*>(md + i);
    const int4 m0 = __ldg(m), m1 = __ldg(m + 1);
    const int s = e + m0.x;
    emax = max(emax, e);
    E = max(E, s);
    const unsigned ss = __byte_perm((unsigned)s, 0, 0x1010);
    const unsigned d[6] = {(unsigned)m0.z, (unsigned)m0.w, (unsigned)m1.x, (unsigned)m1.y, (unsigned)m1.z, (unsigned)m1.w};
#pragma unroll
    for (int q = 0; q < 6; q++) T[q] = __viaddmax_s16x2(d[q], ss, T[q]);
  };
  int i0 = 0;
  for (; i0 + 8 <= n; i0 += 8) {
    double2 v[8];  // eight loads in flight
#pragma unroll
    for (int k = 0; k < 8; k++) v[k] = __ldg(col + (i0 + k) * ld);
#pragma unroll
    for (int k = 0; k < 8; k++) add(v[k], i0 + k);
  }
  for (; i0 < n; i0 += 2) {  // the last one of an odd number twice
    const int i1 = min(i0 + 1, n - 1);
    const double2 u = __ldg(col + i0 * ld), v = __ldg(col + i1 * ld);
    add(u, i0);
    add(v, i1);
  }
  int w = E * 8192 + (emax == 2047 ? 4096 : 0);
#pragma unroll
  for (int b = 0; b < 12; b++)
    if (E - (short)(T[b >> 1] >> (16 * (b & 1))) > PJ_LOSS<X> || E + __ldg(xe + b) < 2 * 1023 - 900) w |= 1 << b;
  return w;
}
template <int X>
__global__ void __launch_bounds__(128) k_proj_scan(int n, long long ld, const double2* eta, const ProjMode* md,
                                                   const int* xe, int* word) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < ld) word[t] = pj_scan<X>(n, ld, eta + t, md, xe);
}

// sum_i eta_i conj(xi_i[b]) by a warp, a lane a mode, every term relative to 2^T, T the largest exponent(eta_i) + exponent(xi_i[b]).
// (By one thread the loads' latency in a row, 0.6 us a mode, set the time of small calls.)
template <int X>
LQ_DI double2 px_column(int n, long long ld, const double2* col, const double2* xb) {
  const int lane = threadIdx.x & 31;
  int T = 2;
#pragma unroll 1
  for (int i = lane; i < n; i += 32) {
    const double2 x = __ldg(xb + 12 * i);
    if (x.x != 0.0 || x.y != 0.0) T = max(T, px_exponent(x) + px_exponent(__ldg(col + i * ld)));
  }
  T = __reduce_max_sync(0xffffffffu, T);
  double2 sum = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += PJ_MODES<X>) {
    const int i1 = min(n, i0 + PJ_MODES<X>);
    long long t[4] = {0, 0, 0, 0};
#pragma unroll 1
    for (int i = i0 + lane; i < i1; i += 32) {
      const double2 x = __ldg(xb + 12 * i);
      if (x.x == 0.0 && x.y == 0.0) continue;
      const int e = px_exponent(x);
      px_conj_mac(t, px_limbs<X>(x, e), px_limbs<X>(__ldg(col + i * ld), T - e));
    }
#pragma unroll 1
    for (int o = 16; o; o >>= 1) {
#pragma unroll
      for (int k = 0; k < 4; k++) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
    }
    const double2 v = px_value<true>(t, T - 2 * px_bias<X> + 56);
    sum.x += v.x;
    sum.y += v.y;
  }
  return sum;
}

// fact[b][y][a] = -sum_i eta_i(y)[a] conj(xi_i(x)[b]) for y in Gamma*; one thread per (site of Gamma*, a).
//
// Scales.  Modes may differ in size by any factor that their partners take off again, so mode i has an exponent, md[i].r, and
// column b one, xe[b], of what is left of its entries; the limbs of xi_i(x)[b], staged in shared memory (n * 12 entries),
// are relative to both, those of eta_i(y)[a] to E - r_i, E the largest exponent(eta_i) + r_i.  A sum is then off by a few
// 2^-55 2^(E + xe[b]), which is what FP64 sums do as long as one of the terms of column b is not far below 2^(E + xe[b]).
// pj_scan looks for such a term of each column, and where there is none within a factor of 2^PJ_LOSS the column is summed
// again on a scale of its own (px_column).  Columns of modes of similar sizes seldom come there: of 120 normal modes 1e-6, of
// 2 2e-5.
//
// Bound by the integer pipe: 144 multiply-adds (32 x 32 + 64) per complex number read.  For many modes (X = 0) the scan is a
// kernel of its own, bound by HBM, whose results are in word; next to the sums it cost them 4 to 20% by the order of
// registers and instructions alone.  For fewer a kernel more is what costs.
// 120 modes on 24 slices of 24^3: 37.0 ms with FP64 sums (at the FP64 pipe's peak), 12.7 ms so; 24 modes 3.2 ms.
template <int X>
__global__ void __launch_bounds__(128, 2) k_proj_prop(int n, long long nsite, long long y0, long long V,
                                                   const double2* eta, const int4* xi_l, const double2* xi_x,
                                                   const ProjMode* md, const int4* r4, const int* xe, const int* word,
                                                   double2* fact) {
  extern __shared__ int4 xs[];
  for (int e = threadIdx.x; e < n * 12; e += blockDim.x) xs[e] = xi_l[e];
  __syncthreads();
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, ld = nsite * 12;
  const bool valid = t0 < ld;
  const long long t = valid ? t0 : ld - 1;  // in range; nothing is stored for it
  const double2* col = eta + t;
  const int w = X == 0 ? __ldg(word + t) : pj_scan<X>(n, ld, col, md, xe);
  const int E = w >> 13;
  const long long y = y0 + t / 12;
  const int a = (int)(t % 12);
  double2 sum[12];
#pragma unroll
  for (int b = 0; b < 12; b++) sum[b] = make_double2(0.0, 0.0);
  for (int i0 = 0; i0 < n; i0 += PJ_MODES<X>) {
    const int i1 = min(n, i0 + PJ_MODES<X>);
    long long hr[12], cr[12], hi[12], ci[12];
#pragma unroll
    for (int b = 0; b < 12; b++) hr[b] = cr[b] = hi[b] = ci[b] = 0;
    double2 next[4];  // loads four modes ahead
    int4 rn = __ldg(r4 + i0 / 4);
#pragma unroll
    for (int k = 0; k < 4; k++) next[k] = __ldg(col + min(i0 + k, i1 - 1) * ld);
    const double2* ahead = col + (i0 + 4) * ld;
#pragma unroll 1
    for (int i = i0; i < i1; i += 4) {
      const int r[4] = {rn.x, rn.y, rn.z, rn.w};
      rn = __ldg(r4 + min(i + 4, i1 - 1) / 4);
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const double2 e = next[k];
        if (i + 4 + k < i1) next[k] = __ldg(ahead);
        ahead += ld;
        if (i + k >= i1) continue;
        int r1, r0, m1, m0;
        px_split<X>(e.x, E - r[k], r1, r0);
        px_split<X>(e.y, E - r[k], m1, m0);
#pragma unroll
        for (int b = 0; b < 12; b++) {
          const int4 c = xs[(i + k) * 12 + b];  // e conj(c)
          px_mac(hr[b], cr[b], r1, r0, c.x, c.y);
          px_mac(hr[b], cr[b], m1, m0, c.z, c.w);
          px_mac(hi[b], ci[b], m1, m0, c.x, c.y);
          px_mac(hi[b], ci[b], -r1, -r0, c.z, c.w);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < 12; b++) {
      const int s = E + __ldg(xe + b) - 2 * px_bias<X> + 56;
      const double re = fx_sum<28, false>(hr[b], cr[b], s), im = fx_sum<28, false>(hi[b], ci[b], s);
      sum[b] = i0 ? make_double2(sum[b].x + re, sum[b].y + im) : make_double2(re, im);
    }
  }
  int redo = valid ? w & 4095 : 0;
#pragma unroll
  for (int b = 0; b < 12; b++) {
    const bool bad = (w & 4096) || __ldg(xe + b) == 2047;
    if (bad) redo &= ~(1 << b);
    if (valid)
      fact[((long long)b * V + y) * 12 + a] = bad ? make_double2(nan(""), nan("")) : make_double2(-sum[b].x, -sum[b].y);
  }
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (unsigned lanes = __ballot_sync(0xffffffffu, redo != 0); lanes; lanes &= lanes - 1) {
    const int l = __ffs(lanes) - 1;
#pragma unroll 1
    for (int cols = __shfl_sync(0xffffffffu, redo, l); cols; cols &= cols - 1) {
      const int b = __ffs(cols) - 1;
      const double2 v = px_column<X>(n, ld, eta + (t0 - lane + l), xi_x + b);
      if (lane == l) fact[((long long)b * V + y) * 12 + a] = make_double2(-v.x, -v.y);
    }
  }
}

// xi_x[i][b] = xi_i(x)[b], the modes' and columns' exponents (xe[b] = 2047: column b has an entry that is not finite) and the
// limbs: one block, a thread an entry.
template <int X>
__global__ void __launch_bounds__(1024) k_gather_site(int n, long long nsite_gb, long long xloc, const double2* xi,
                                                      int4* xi_l, double2* xi_x, ProjMode* md, int* r4, int* xe) {
  __shared__ int r[1024], ce[12], bad[12];
  for (int i = threadIdx.x; i < n; i += blockDim.x) r[i] = PJ_NONE;
  if (threadIdx.x < 12) {
    ce[threadIdx.x] = PJ_NONE;
    bad[threadIdx.x] = 0;
  }
  __syncthreads();
  auto entry = [&](int t) { return __ldg(xi + ((long long)(t / 12) * nsite_gb + xloc) * 12 + t % 12); };
  auto exponent = [](double2 v) {  // of a number that counts: neither zero nor without a size
    const int e = px_exponent(v);
    return (v.x == 0.0 && v.y == 0.0) || e == 2047 ? PJ_NONE : e;
  };
  for (int t = threadIdx.x; t < n * 12; t += blockDim.x) atomicMax(&r[t / 12], exponent(entry(t)));
  __syncthreads();
  for (int t = threadIdx.x; t < n * 12; t += blockDim.x) {
    const double2 v = entry(t);
    const int e = exponent(v);
    if (e != PJ_NONE) atomicMax(&ce[t % 12], e - r[t / 12]);
    if (px_exponent(v) == 2047) bad[t % 12] = 1;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n * 12; t += blockDim.x) {
    const int i = t / 12, b = t % 12;
    const double2 v = entry(t);
    const int e = exponent(v);
    xi_x[t] = v;
    xi_l[t] = px_limbs<X>(e == PJ_NONE ? make_double2(0.0, 0.0) : v, max(r[i] + ce[b], 1));
    md[i].d[b] = (short)((e == PJ_NONE ? PJ_NONE : e - r[i]) - ce[b]);
    if (b == 0) md[i].r = r4[i] = r[i];
  }
  if (threadIdx.x < 12) xe[threadIdx.x] = bad[threadIdx.x] ? 2047 : ce[threadIdx.x];
}

struct Scratch {
  void* p = nullptr;
  cudaStream_t st = nullptr;
  ~Scratch() {
    if (p) cudaFreeAsync(p, st);
  }
  int alloc(size_t bytes, cudaStream_t s) {
    st = s;
    if (cudaMallocAsync(&p, bytes ? bytes : 16, s) != cudaSuccess) {
      cudaGetLastError();
      lq_set_error("device allocation failed (orthonormalisation scratch)");
      return LQCD_ENOMEM;
    }
    return 0;
  }
};

// One Cholesky-QR pass: out = in R^{-1}, in = out R.
int chol_qr(const ColMat& in, const ColMat& out, double2* G, double2* Linv, int* cexp, int2* d_pairs, int npairs,
            double2* part, int nsplit, long long chunk, int npad, int* d_status, cudaStream_t st) {
  const int n = in.ncol;
  k_gram<<<dim3((unsigned)npairs, (unsigned)nsplit), 256, 0, st>>>(in, chunk, npad, d_pairs, part);
  RC(launched_here());
  k_gram_reduce<<<(unsigned)((n * n + 255) / 256), 256, 0, st>>>(part, nsplit, npad, n, G);
  RC(launched_here());
  k_chol_inv<<<1, 1024, 0, st>>>(G, n, Linv, cexp, d_status);
  RC(launched_here());
  const long long R = in.rows[0] + (in.nseg > 1 ? in.rows[1] : 0);
  k_apply_rinv<<<dim3((unsigned)((R + 127) / 128), (unsigned)((n + GT - 1) / GT)), 128, 0, st>>>(in, out, Linv, cexp, n);
  return launched_here();
}

}  // namespace

int lq_orthonormalize(ColMat v, ColMat tmp, cudaStream_t st) {
  const int n = v.ncol;
  if (n < 1 || n > 1024) {
    lq_set_error("orthonormalisation: 1..1024 columns");
    return LQCD_EBADARG;
  }
  const long long R = v.rows[0] + (v.nseg > 1 ? v.rows[1] : 0);
  if (R < n) {
    lq_set_error("orthonormalisation: fewer rows than columns");
    return LQCD_ERANK;
  }
  const int nt = (n + GT - 1) / GT, npad = nt * GT;
  std::vector<int2> pairs;
  for (int a = 0; a < nt; a++)
    for (int b = a; b < nt; b++) pairs.push_back(make_int2(a, b));
  const int npairs = (int)pairs.size();
  int nsplit = (152 * 8 + npairs - 1) / npairs;
  long long chunk = (R + nsplit - 1) / nsplit;
  chunk = (chunk + GF - 1) / GF * GF;
  nsplit = (int)((R + chunk - 1) / chunk);
  const size_t b_pairs = sizeof(int2) * npairs, b_part = sizeof(double2) * (size_t)nsplit * npad * npad,
               b_g = sizeof(double2) * (size_t)n * n;
  Scratch s;
  RC(s.alloc(b_pairs + b_part + 2 * b_g + 256 + 64 + sizeof(int) * n, st));
  char* base = (char*)s.p;
  int2* d_pairs = (int2*)base;
  double2* part = (double2*)(base + ((b_pairs + 255) / 256) * 256);
  double2* G = (double2*)((char*)part + b_part);
  double2* Linv = (double2*)((char*)G + b_g);
  int* d_status = (int*)((char*)Linv + b_g);
  int* cexp = d_status + 16;
  if (cudaMemcpyAsync(d_pairs, pairs.data(), b_pairs, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(d_status, 0, sizeof(int), st) != cudaSuccess) {
    lq_set_error("orthonormalisation: copy failed");
    return LQCD_ECUDA;
  }
  RC(chol_qr(v, tmp, G, Linv, cexp, d_pairs, npairs, part, nsplit, chunk, npad, d_status, st));
  RC(chol_qr(tmp, v, G, Linv, cexp, d_pairs, npairs, part, nsplit, chunk, npad, d_status, st));
  int h_status = 0;
  if (cudaMemcpyAsync(&h_status, d_status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    lq_set_error("orthonormalisation: synchronisation failed");
    return LQCD_ECUDA;
  }
  if (h_status) {
    lq_set_error("orthonormalisation: the vectors are linearly dependent");
    return LQCD_ERANK;
  }
  return 0;
}

int lq_slice_plus(const lqcd_lattice* L, const Batch& b, int g1, const double2* ve, const double2* vo, double2* phi,
                  cudaStream_t st) {
  const int S3 = 2 * L->g.S3h;
  k_slice_plus<<<(unsigned)(b.nsys * ((S3 + 127) / 128)), 128, 0, st>>>(L->g, b.nsys, b.sys, g1, ve, vo, phi);
  return launched_here();
}

int lq_slice_source(const lqcd_lattice* L, const Batch& b, const int* d_ids, int g1, const double2* phi, double2* ve,
                    double2* vo, cudaStream_t st) {
  k_slice_source<<<dim3((unsigned)(b.nsys * b.nby), 1, 2), 128, 0, st>>>(L->g, b.nsys, b.sys, d_ids, g1, phi, ve, vo);
  return launched_here();
}

template <int X>
static int proj_prop(const lqcd_lattice* L, int n, long long nsite_gb, long long xloc, const double2* xi,
                     long long nsite_gs, long long y0, const double2* eta, double2* fact, cudaStream_t st) {
  Scratch s;
  const size_t n4 = ((size_t)n + 3) / 4 * 4;
  const long long nt = nsite_gs * 12;
  RC(s.alloc((sizeof(int4) + sizeof(double2)) * 12 * n + (sizeof(ProjMode) + sizeof(int)) * n4 + sizeof(int) * 12 +
                 (X == 0 ? sizeof(int) * (size_t)nt : 0),
             st));
  int4* xi_l = (int4*)s.p;
  double2* xi_x = (double2*)(xi_l + 12 * (size_t)n);
  ProjMode* md = (ProjMode*)(xi_x + 12 * (size_t)n);
  int* r4 = (int*)(md + n4);
  int* xe = r4 + n4;
  int* word = xe + 12;
  k_gather_site<X><<<1, 1024, 0, st>>>(n, nsite_gb, xloc, xi, xi_l, xi_x, md, r4, xe);
  RC(launched_here());
  const size_t sm = sizeof(int4) * 12 * (size_t)n;
  if (sm > 48 * 1024) {
    if (cudaFuncSetAttribute(k_proj_prop<X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess) {
      cudaGetLastError();
      lq_set_error("projected propagator: too many modes for shared memory");
      return LQCD_EBADARG;
    }
  }
  const unsigned blocks = (unsigned)((nt + 127) / 128);
  if (X == 0) {
    k_proj_scan<X><<<blocks, 128, 0, st>>>(n, nt, eta, md, xe, word);
    RC(launched_here());
  }
  k_proj_prop<X><<<blocks, 128, sm, st>>>(n, nsite_gs, y0, L->V, eta, xi_l, xi_x, md, (const int4*)r4, xe, word, fact);
  return launched_here();
}

// The widest limbs whose sums hold all modes: the more bits, the seldomer a column needs a second sum.  Above 60 modes
// the scan's words take 4 bytes a component of eta; without room for them, and where all blocks run at a time and another kernel
// is the larger cost (120 modes on three slices of 4 x 4 x 8: 158 us, 143 in runs), runs of 60.
int lq_proj_prop(const lqcd_lattice* L, int n, long long nsite_gb, long long xloc, const double2* xi, long long nsite_gs,
                 long long y0, const double2* eta, double2* fact, cudaStream_t st) {
  if (n <= PJ_MODES<2>) return proj_prop<2>(L, n, nsite_gb, xloc, xi, nsite_gs, y0, eta, fact, st);
  if (n > PJ_MODES<1> && nsite_gs * 12 > 152 * 2 * 128) {
    const int rc = proj_prop<0>(L, n, nsite_gb, xloc, xi, nsite_gs, y0, eta, fact, st);
    if (rc != LQCD_ENOMEM) return rc;
  }
  return proj_prop<1>(L, n, nsite_gb, xloc, xi, nsite_gs, y0, eta, fact, st);
}
