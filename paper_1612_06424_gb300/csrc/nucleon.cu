// Nucleon blocks on projected quark lines (Sec. 4.2 eq. nucleon_prop_factorized):
//   B[i][j][k][alpha](t) = sum_{x in slice t} eps^{abc} {[s_i^T]^a(x) C g5 [s_j]^b(x)} [s_k]^c_alpha(x)
// as a contraction over (x, c) of the diquark D[(i,j)][(x,c)] with
// S[(x,c)][(k,alpha)] = s_k(x)[alpha][c]: a dense O(N^3 L^3) product, run on
// the FP32 pipes (the GB300's FP64 rate is 1/62 of FP32): per-thread FP32
// partial sums over 64 sites are added into FP32 running sums (two-level
// summation); the diquark tiles are generated in shared memory and never stored.  Then the two Wick contractions
//   W1 = -sum_ijk B_xi[j,i,k]^T g5 P_- B_eta[i,j,k],  W2 = -sum_ijk B_xi[k,i,j]^T g5 P_- B_eta[i,j,k].
#include <algorithm>
#include <mutex>
#include <vector>

#include "internal.h"

using namespace lq;

namespace {

constexpr int TI = 8, TJ = 8;  // (i, j) pair tile: 64 rows
constexpr int TK = 16;         // k tile: 64 (k, alpha) columns
constexpr int XS = 8;          // sites per shared-memory stage
constexpr int FLUSH = 8;       // stages per first-level partial sum (64 sites)
constexpr int TOT_BYTES = 16 * 256 * 8;  // dynamic shared memory of the second-level sums

#define RC_LAUNCH()                     \
  do {                                  \
    const int r_ = launched_here();     \
    if (r_ != 0) return r_;             \
  } while (0)

int launched_here() {
  lq_count_launch();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    lq_set_error(std::string("kernel launch: ") + cudaGetErrorString(e));
    return LQCD_ECUDA;
  }
  return 0;
}

// C g5 with C = g0 g2 in the chiral basis of lqcd.h (g0 = [[0,-1],[-1,0]],
// g2 = [[0,-i s2],[i s2,0]], g5 = diag(1,1,-1,-1)): its non-zero entries are
// (0,1) = -1, (1,0) = +1, (2,3) = -1, (3,2) = +1, so
// s^T C g5 t = -s0 t1 + s1 t0 - s2 t3 + s3 t2   (spin indices).
LQ_DI float2 cg5_pair(const float2* si, const float2* tj, int a, int b) {
  // si, tj: 12 complex [spin*3 + colour]; colour a of s, colour b of t
  float2 r = make_float2(0.f, 0.f);
  const int sp[4][2] = {{0, 1}, {1, 0}, {2, 3}, {3, 2}};
  const float sg[4] = {-1.f, 1.f, -1.f, 1.f};
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const float2 u = si[sp[q][0] * 3 + a], v = tj[sp[q][1] * 3 + b];
    r.x += sg[q] * (u.x * v.x - u.y * v.y);
    r.y += sg[q] * (u.x * v.y + u.y * v.x);
  }
  return r;
}

// One block: a 64 x 64 tile of B[(i,j)][(k,alpha)] of one time slice.
// s: n slab vectors (FP64, [n][nsite][12]); slice blockIdx.z covers the
// slab-local sites lo0 + z * t_stride_sites .. + S3.
__global__ void __launch_bounds__(256, 2) k_nucleon_block(int n, long long nsite, const double2* s, int conj,
                                                       int S3, long long lo0, int t_stride_sites, double2* B) {
  __shared__ float2 fi[XS][TI][13], fj[XS][TJ][13];  // 13: rows on distinct banks
  __shared__ __align__(16) float2 Ds[XS * 3][TI * TJ], Ss[XS * 3][TK * 4];
  extern __shared__ float2 tot[];  // [16][256]: second-level sums of each thread's 4 x 4 tile
  const int nti = (n + TI - 1) / TI, ntj = (n + TJ - 1) / TJ;
  const int tile = blockIdx.x;
  const int i0 = (tile % nti) * TI, j0 = ((tile / nti) % ntj) * TJ;
  const int k0 = blockIdx.y * TK;
  const int t = blockIdx.z;
  const long long lo = lo0 + (long long)t * t_stride_sites;
  // thread tile: rows tr*4 .. tr*4+3 and columns 2tc, 2tc+1, 32+2tc, 32+2tc+1 (so that the
  // 16 threads of a row read 256 contiguous bytes of S per 16-byte load)
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;
  float2 acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; p++)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      acc[p][q] = make_float2(0.f, 0.f);
      tot[(p * 4 + q) * 256 + threadIdx.x] = make_float2(0.f, 0.f);
    }
  const float cs = conj ? -1.f : 1.f;
  int stage = 0;
  for (int x0 = 0; x0 < S3; x0 += XS, stage++) {
    // the i and j fields of the stage's sites, FP64 -> FP32 (conjugated for the xi side)
    for (int e = threadIdx.x; e < XS * (TI + TJ) * 12; e += blockDim.x) {
      const int comp = e % 12, r = e / 12;
      const int x = r % XS, w = r / XS;  // w: 0..TI+TJ-1
      const int f = w < TI ? i0 + w : j0 + w - TI;
      float2 v = make_float2(0.f, 0.f);
      if (f < n && x0 + x < S3) {
        const double2 d = s[((long long)f * nsite + lo + x0 + x) * 12 + comp];
        v = make_float2((float)d.x, cs * (float)d.y);
      }
      if (w < TI) fi[x][w][comp] = v;
      else fj[x][w - TI][comp] = v;
    }
    // S[(x, c)][(k, alpha)] = s_k(x)[alpha][c]; consecutive threads read one site's 12 components
    for (int e = threadIdx.x; e < XS * TK * 12; e += blockDim.x) {
      const int comp = e % 12, r = e / 12;
      const int x = r % XS, kk = r / XS;
      const int al = comp / 3, c = comp % 3;
      const int k = k0 + kk;
      float2 v = make_float2(0.f, 0.f);
      if (k < n && x0 + x < S3) {
        const double2 d = s[((long long)k * nsite + lo + x0 + x) * 12 + comp];
        v = make_float2((float)d.x, cs * (float)d.y);
      }
      Ss[x * 3 + c][kk * 4 + al] = v;
    }
    __syncthreads();
    // diquark D[(x, c)][(i, j)], the three colours c of one (x, i, j) from one read of s_i(x), s_j(x)
    for (int e = threadIdx.x; e < XS * TI * TJ; e += blockDim.x) {
      const int pr = e % (TI * TJ), x = e / (TI * TJ);
      const int ii = pr / TJ, jj = pr % TJ;
      float2 u[12], v[12];
#pragma unroll
      for (int q = 0; q < 12; q++) {
        u[q] = fi[x][ii][q];
        v[q] = fj[x][jj][q];
      }
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const int a = (c + 1) % 3, b = (c + 2) % 3;  // eps^{abc} = +1 for (a, b) and -1 for (b, a)
        const float2 p = cg5_pair(u, v, a, b), m = cg5_pair(u, v, b, a);
        Ds[x * 3 + c][pr] = make_float2(p.x - m.x, p.y - m.y);
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int r = 0; r < XS * 3; r++) {
      float2 av[4], bv[4];
      {
        const float4* pa = reinterpret_cast<const float4*>(&Ds[r][tr * 4]);
        const float4 a0 = pa[0], a1 = pa[1];
        const float4 b0 = *reinterpret_cast<const float4*>(&Ss[r][2 * tc]);
        const float4 b1 = *reinterpret_cast<const float4*>(&Ss[r][32 + 2 * tc]);
        av[0] = make_float2(a0.x, a0.y);
        av[1] = make_float2(a0.z, a0.w);
        av[2] = make_float2(a1.x, a1.y);
        av[3] = make_float2(a1.z, a1.w);
        bv[0] = make_float2(b0.x, b0.y);
        bv[1] = make_float2(b0.z, b0.w);
        bv[2] = make_float2(b1.x, b1.y);
        bv[3] = make_float2(b1.z, b1.w);
      }
#pragma unroll
      for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) {
          acc[p][q].x = fmaf(av[p].x, bv[q].x, fmaf(-av[p].y, bv[q].y, acc[p][q].x));
          acc[p][q].y = fmaf(av[p].x, bv[q].y, fmaf(av[p].y, bv[q].x, acc[p][q].y));
        }
    }
    __syncthreads();
    if ((stage + 1) % FLUSH == 0) {
#pragma unroll
      for (int p = 0; p < 4; p++)
#pragma unroll
        for (int q = 0; q < 4; q++) {
          float2& t2 = tot[(p * 4 + q) * 256 + threadIdx.x];
          t2.x += acc[p][q].x;
          t2.y += acc[p][q].y;
          acc[p][q] = make_float2(0.f, 0.f);
        }
    }
  }
#pragma unroll
  for (int p = 0; p < 4; p++) {
    const int pr = tr * 4 + p;
    const int i = i0 + pr / TJ, j = j0 + pr % TJ;
    if (i >= n || j >= n) continue;
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int col = q < 2 ? 2 * tc + q : 32 + 2 * tc + q - 2;
      const int k = k0 + col / 4, al = col % 4;
      if (k >= n) continue;
      const float2 t2 = tot[(p * 4 + q) * 256 + threadIdx.x];
      const double2 v = make_double2((double)t2.x + acc[p][q].x, (double)t2.y + acc[p][q].y);
      B[((((long long)t * n + i) * n + j) * n + k) * 4 + al] = v;
    }
  }
}

// Wick contractions of every pair (ix of B_xi, iy of B_eta), FP64.  g5 P_- = g5 (1 - g0)/2 in the
// chiral basis is (1/2)[[1,0,1,0],[0,1,0,1],[-1,0,-1,0],[0,-1,0,-1]], so with
// u_h = B_eta_h + B_eta_{h+2} and d_h = B_xi_h - B_xi_{h+2} (h = 0, 1)
//   W1 = -(1/2) sum_ijk sum_h d_h[j][i][k] u_h[i][j][k],
//   W2 = -(1/2) sum_ijk sum_h d_h[k][i][j] u_h[i][j][k].
//
// Bound by the FP64 pipe (20 instructions per (i,j,k) and pair of slices, the GB300 issues about 2
// per clock and SM) just above the read of the blocks.  The sum over (i,j,k) is therefore cut into
// enough parts for every SM: a block takes 16 x 16 (j, k) tiles of one i (one thread an element, so
// that the transposed rows B_xi[k][i][j0..] are read as runs of 1 KB too), and one read of B_xi serves
// CT_NY sink slices.  Part p of pair (ix, iy) goes to part[((ix ny + iy) nsplit + p) 4]; k_contract_sum
// adds the parts in a fixed order.  120 factors, 8 sink slices: 38.7 ms with one block per pair of
// slices, 0.6 ms so.
constexpr int CT = 16;     // edge of a (j, k) tile
constexpr int CT_NY = 4;   // sink slices per block

__global__ void __launch_bounds__(CT * CT) k_nucleon_contract(int n, int ny, int nsplit, const double2* Bx,
                                                              const double2* By, double* part) {
  // grid: ((ix, group of sink slices), part), the part fastest
  const int sp = (int)(blockIdx.x % (unsigned)nsplit), pr = (int)(blockIdx.x / (unsigned)nsplit);
  const int ngy = (ny + CT_NY - 1) / CT_NY;
  const int ix = pr / ngy, iy0 = (pr - ix * ngy) * CT_NY;
  const long long n3 = (long long)n * n * n;
  const double2* bx = Bx + (long long)ix * n3 * 4;
  const int nt = (n + CT - 1) / CT;
  const int tj = threadIdx.x / CT, tk = threadIdx.x % CT;
  double acc[CT_NY][4];
#pragma unroll
  for (int y = 0; y < CT_NY; y++)
#pragma unroll
    for (int q = 0; q < 4; q++) acc[y][q] = 0.0;
  const long long tiles = (long long)n * nt * nt;
  for (long long tile = sp; tile < tiles; tile += nsplit) {
    const int i = (int)(tile / (nt * nt)), r = (int)(tile - (long long)i * nt * nt);
    const int j = (r / nt) * CT + tj, k = (r % nt) * CT + tk;
    if (j >= n || k >= n) continue;
    const double2* x1 = bx + ((((long long)j * n + i) * n) + k) * 4;  // B_xi[j][i][k]
    const double2* x2 = bx + ((((long long)k * n + i) * n) + j) * 4;  // B_xi[k][i][j]
    double2 d1[2], d2[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const double2 a = __ldg(x1 + h), b = __ldg(x1 + h + 2), c = __ldg(x2 + h), e = __ldg(x2 + h + 2);
      d1[h] = make_double2(a.x - b.x, a.y - b.y);
      d2[h] = make_double2(c.x - e.x, c.y - e.y);
    }
    const double2* yv = By + ((long long)iy0 * n3 + (((long long)i * n + j) * n) + k) * 4;  // B_eta[i][j][k]
#pragma unroll
    for (int y = 0; y < CT_NY; y++) {
      if (iy0 + y >= ny) break;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const double2 a = __ldg(yv + (long long)y * n3 * 4 + h), b = __ldg(yv + (long long)y * n3 * 4 + h + 2);
        const double2 u = make_double2(a.x + b.x, a.y + b.y);
        acc[y][0] = fma(d1[h].x, u.x, fma(-d1[h].y, u.y, acc[y][0]));
        acc[y][1] = fma(d1[h].x, u.y, fma(d1[h].y, u.x, acc[y][1]));
        acc[y][2] = fma(d2[h].x, u.x, fma(-d2[h].y, u.y, acc[y][2]));
        acc[y][3] = fma(d2[h].x, u.y, fma(d2[h].y, u.x, acc[y][3]));
      }
    }
  }
  __shared__ double sh[CT_NY * 4][CT * CT / 32];
#pragma unroll
  for (int y = 0; y < CT_NY; y++)
#pragma unroll
    for (int q = 0; q < 4; q++) {
      double v = acc[y][q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((threadIdx.x & 31) == 0) sh[y * 4 + q][threadIdx.x >> 5] = v;
    }
  __syncthreads();
  if (threadIdx.x < CT_NY * 4) {
    const int iy = iy0 + threadIdx.x / 4;
    if (iy < ny) {
      double r = 0.0;
      for (int w = 0; w < CT * CT / 32; w++) r += sh[threadIdx.x][w];
      part[(((long long)ix * ny + iy) * nsplit + sp) * 4 + threadIdx.x % 4] = r;
    }
  }
}

// W[pair] = -(1/2) sum of the pair's nsplit parts, one warp per value, lanes then shuffles in a fixed
// order.  part may be W itself when nsplit is 1.
__global__ void __launch_bounds__(128) k_contract_sum(int nsplit, const double* part, double* W) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* p = part + (long long)blockIdx.x * nsplit * 4 + q;
  double r = 0.0;
  for (int k = lane; k < nsplit; k += 32) r += p[4LL * k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if (lane == 0) W[(long long)blockIdx.x * 4 + q] = -0.5 * r;
}

// out[e] = (1/count) sum_j in[j * size + e], summed in j order (FP64).  inv = 1/count: a power of two is
// divided by exactly with one product; else one Newton correction rounds the quotient as a division
// does, at three FP64 instructions (a division takes about ten, which held the kernel at 1.2 TB/s).  Two
// elements a thread keep more loads in flight.  120^3 x 4 x 9 from two levels: 2.47 ms with divisions, 0.50 ms so.
LQ_DI double quotient(double s, double n, double inv, bool pow2) {
  const double q = s * inv;
  return pow2 || !isfinite(q) ? q : fma(fma(-q, n, s), inv, q);
}
__global__ void __launch_bounds__(256) k_level_mean(long long size, int count, double inv, int pow2, const double2* in,
                                                    double2* out) {
  const double n = count;
  for (long long e0 = ((long long)blockIdx.x * blockDim.x) * 2 + threadIdx.x; e0 < size;
       e0 += (long long)gridDim.x * blockDim.x * 2) {
    const long long e1 = e0 + blockDim.x;
    const bool two = e1 < size;
    double2 a = __ldg(in + e0), b = two ? __ldg(in + e1) : make_double2(0.0, 0.0);
#pragma unroll 4
    for (int j = 1; j < count; j++) {
      const double2* p = in + (long long)j * size;
      const double2 v = __ldg(p + e0), w = two ? __ldg(p + e1) : make_double2(0.0, 0.0);
      a.x += v.x;
      a.y += v.y;
      b.x += w.x;
      b.y += w.y;
    }
    out[e0] = make_double2(quotient(a.x, n, inv, pow2), quotient(a.y, n, inv, pow2));
    if (two) out[e1] = make_double2(quotient(b.x, n, inv, pow2), quotient(b.y, n, inv, pow2));
  }
}

// The two nucleon Wick contractions from a point source to every sink y of a
// time slice (the contractions behind eq. nucleon_prop_factorized), FP64.
// S(y) = the 12 x 12 propagator matrix at y, S_{(mu a),(nu b)} =
// prop[3 nu + b][y][mu][a]; with nu(mu), cg(mu) the non-zero entries of C g5
// and M = g5 P_-, whose rows gam and gam + 2 differ by the sign:
//   V^c_{g,X}    = S_{(g c),X} + S_{(g+2 c),X},   Z_{R,(g c')} = S_{R,(g c')} - S_{R,(g+2 c')}   (g = 0, 1),
//   H^{c g c'}_{mu a} = sum_{mu' a'b'} eps_{a'b'c'} cg(mu') S_{(mu a),(nu(mu') b')} V^c_{g,(mu' a')},
//   W2 = (1/2) sum_{c g c'} sum_{mu ab} eps_{abc} cg(mu) H^{c g c'}_{mu a} Z_{(nu(mu) b),(g c')};
//   W1 = sum_{cc'} sum_mu cg(mu) T^{cc'}_mu sum_g (V^c_{g,(g c')} - V^c_{g,(g+2 c')}),
//   T^{cc'}_mu = sum_{mu' a'b'} eps_{a'b'c'} cg(mu') S_{(mu a0),(nu(mu') b')} S_{(nu(mu) b0),(mu' a')},
// (a0, b0, c) cyclic: the terms with a, b and both mu -> nu(mu), a' <-> b' exchanged are equal in
// pairs, which removes the factor 1/2 of M and half of the products.
//
// The products run in fixed point on the integer pipe (fxnum.cuh, 32 times the FP64 pipe's rate): a
// site's 144 entries become 57-bit integers, H and T are 64-bit sums, and each H Z and T U
// is rounded to FP64 once and summed there.  1620 complex multiply-adds a site in the factored form, where the
// plain sums over all terms take 17000.  A block stages 16 sites of one slice in shared memory and
// spreads their 16 x 144 elements H and 16 x 36 elements T over its 128 threads (consecutive threads
// take the 8 rows (mu, a) of one (c, g, c'), so their reads of V and Z are broadcasts and those of S nearly
// free of conflicts); three blocks an SM overlap one another's loads.  Up to four stages of a block share its
// final sums.
//
// Scales.  Every term has each sink colour and each source colour once, so each of these has an exponent of its own (rho_a,
// kappa_b; S_{(mu a),(nu b)} is stored relative to 2^(rho_a + kappa_b)) and all terms share their sum.  What is left can differ
// by spins or by pairs of colours.  The error of a site, 0.7 2^-53 of the product of the scales, is then one of its terms only
// if one of them is about that large: np_large_terms looks for a term of W1 and one of W2 whose three entries all lie
// within a factor of four of their scales, and a site without them is summed in FP64 (6600 multiply-adds on a pipe a 32nd as
// fast: 64 x 24^3 takes 13.7 ms if all sites do, as with entries spread over 16 decades).
//
// Propagator of 64 x 24^3: 114.8 ms with the plain FP64 sums, one warp a site; 11.4 ms factored in
// FP64; 5.7 ms so, 0.1 of them for the scales (error against long double over six propagators 2.3e-16 rms, of the FP64 sums 4.1e-16).
constexpr int NP_T = 128;        // threads
constexpr int NP_SITES = 16;     // sites staged at a time
constexpr int NP_GROUPS = 4;     // most stages per block
constexpr int NP_WORDS = 144 + 72 + 72;  // S, V and Z of a site
constexpr int NP_SMEM = NP_SITES * NP_WORDS * 16;

struct np_acc {  // sum of products of limbs: hh 2^58 + cr 2^29
  long long hr, cr, hi, ci;
};
// t += (NEG ? - : +) a b
template <bool NEG>
LQ_DI void np_mac(np_acc& t, int4 a, int4 b) {
  const int r1 = NEG ? -a.x : a.x, r0 = NEG ? -a.y : a.y, i1 = NEG ? -a.z : a.z, i0 = NEG ? -a.w : a.w;
  mad_wide(t.hr, r1, b.x);
  mad_wide(t.cr, r1, b.y);
  mad_wide(t.cr, r0, b.x);
  mad_wide(t.hr, -i1, b.z);
  mad_wide(t.cr, -i1, b.w);
  mad_wide(t.cr, -i0, b.z);
  mad_wide(t.hi, r1, b.z);
  mad_wide(t.ci, r1, b.w);
  mad_wide(t.ci, r0, b.z);
  mad_wide(t.hi, i1, b.x);
  mad_wide(t.ci, i1, b.y);
  mad_wide(t.ci, i0, b.x);
}
// The sum as limbs of 57 bits, 2^-c of it (c < 0: a multiple).
LQ_DI int4 np_limbs(const np_acc& t, int& c) {
  const long long re = t.hr + ((t.cr + (1ll << 28)) >> 29), im = t.hi + ((t.ci + (1ll << 28)) >> 29);
  const unsigned long long mag = (unsigned long long)((re ^ (re >> 63)) | (im ^ (im >> 63)));
  c = mag ? 7 - __clzll((long long)mag) : 0;
  const long long half = c > 0 ? 1ll << (c - 1) : 0;
  int4 q;
  fx_split(c > 0 ? (re + half) >> c : re << -c, q.x, q.y);
  fx_split(c > 0 ? (im + half) >> c : im << -c, q.z, q.w);
  return q;
}
LQ_DI int4 np_add(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
LQ_DI int4 np_sub(int4 a, int4 b) { return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
// sum over mu' = 0..3 of cg(mu') (s[nu(mu') b'] r[mu' a'] - s[nu(mu') a'] r[mu' b']), nu = 1, 0, 3, 2 and cg = -, +, -, +;
// element (mu, c) of s at (3 mu + c) ls, of r at (3 mu + c) lr
LQ_DI np_acc np_pair(const int4* s, int ls, const int4* r, int lr, int ap, int bp) {
  np_acc t = {0, 0, 0, 0};
#pragma unroll
  for (int m = 0; m < 4; m++) {
    const int nm = m ^ 1;
    const int4 s0 = s[(3 * nm + bp) * ls], r0 = r[(3 * m + ap) * lr];
    const int4 s1 = s[(3 * nm + ap) * ls], r1 = r[(3 * m + bp) * lr];
    if (m & 1) {
      np_mac<false>(t, s0, r0);
      np_mac<true>(t, s1, r1);
    } else {
      np_mac<true>(t, s0, r0);
      np_mac<false>(t, s1, r1);
    }
  }
  return t;
}

// The sets of large entries as bits 3 nu + b of a word for each row 3 mu + a.  Colours c' for which some mu' and {a', b', c'} have
// (nu(mu'), b') in x and (mu', a') in y.
LQ_DI int np_third_colour(int x, int y) {
  x = ((x & 0x1c7) << 3) | ((x >> 3) & 0x1c7);                             // bit (mu', b')
  const int x1 = ((x >> 1) & 0x6db) | ((x & 0x249) << 2), y1 = ((y >> 1) & 0x6db) | ((y & 0x249) << 2);  // colour c' + 1
  const int x2 = ((x >> 2) & 0x249) | ((x << 1) & 0xdb6), y2 = ((y >> 2) & 0x249) | ((y << 1) & 0xdb6);  // c' + 2
  const int p = (x1 & y2) | (x2 & y1);
  return (p | p >> 3 | p >> 6 | p >> 9) & 7;
}
// colours of the sources of spin g and g + 2
LQ_DI int np_source_colour(int z, int g) { return (z >> (3 * g) | z >> (3 * g + 6)) & 7; }
// Bit 0: W1 has a term of three large entries, bit 1: W2 has; the eighth j of all terms.
LQ_DI int np_large_terms(const int* row, int j) {
  int found = 0;
  for (int m = j; m < 48; m += 8) {  // H Z: (mu, g) and the order of a, b, c
    const int mu = m & 3, g = (m >> 2) & 1, o = m >> 3;
    const int a = o >> 1, b = (a + 1 + (o & 1)) % 3, c = 3 - a - b;
    if (np_third_colour(row[3 * mu + a], row[3 * g + c] | row[3 * g + 6 + c]) &
        np_source_colour(row[3 * (mu ^ 1) + b], g))
      found |= 2;
  }
  for (int m = j; m < 12; m += 8) {  // T U: mu and c
    const int mu = m & 3, c = m >> 2;
    const int u = np_source_colour(row[c] | row[6 + c], 0) | np_source_colour(row[3 + c] | row[9 + c], 1);
    if (np_third_colour(row[3 * mu + (c + 1) % 3], row[3 * (mu ^ 1) + (c + 2) % 3]) & u) found |= 1;
  }
  return found;
}

LQ_DI void np_fma(double2& t, double2 a, double2 b, double sg) {  // t += sg a b
  const double x = sg * a.x, y = sg * a.y;
  t.x = fma(x, b.x, fma(-y, b.y, t.x));
  t.y = fma(x, b.y, fma(y, b.x, t.y));
}
// np_pair in FP64
LQ_DI double2 np_pair64(const double2* s, int ls, const double2* r, int lr, int ap, int bp) {
  double2 t = make_double2(0.0, 0.0);
  for (int m = 0; m < 4; m++) {
    const double sg = m & 1 ? 1.0 : -1.0;
    const int nm = m ^ 1;
    np_fma(t, s[(3 * nm + bp) * ls], r[(3 * m + ap) * lr], sg);
    np_fma(t, s[(3 * nm + ap) * ls], r[(3 * m + bp) * lr], -sg);
  }
  return t;
}
// One site in FP64 by the whole block: its entries S (as staged), room for V and Z; adds this thread's part to w1, w2.
LQ_DI void np_site64(const double2* S, double2* Vv, double2* Z, double2& w1, double2& w2) {
  __syncthreads();
  for (int e = threadIdx.x; e < 72; e += NP_T) {
    const int c = e / 24, g = (e / 12) & 1, col = e % 12;
    const double2 a = S[col * 12 + 3 * g + c], b = S[col * 12 + 3 * g + 6 + c];
    Vv[e] = make_double2(a.x + b.x, a.y + b.y);
    const int gz = e / 36, cp = (e / 12) % 3, row = e % 12;
    const double2 u = S[(3 * gz + cp) * 12 + row], v = S[(3 * gz + 6 + cp) * 12 + row];
    Z[e] = make_double2(u.x - v.x, u.y - v.y);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 144 + 36; e += NP_T) {
    if (e < 144) {
      const int mu = (e & 7) >> 1, ai = e & 1, k = e >> 3;
      const int c = k / 6, g = (k / 3) & 1, cp = k % 3;
      const int a = (c + 1 + ai) % 3, b = (c + 2 - ai) % 3;
      const double2 h = np_pair64(S + 3 * mu + a, 12, Vv + (c * 2 + g) * 12, 1, (cp + 1) % 3, (cp + 2) % 3);
      np_fma(w2, h, Z[(g * 3 + cp) * 12 + 3 * (mu ^ 1) + b], (mu ^ ai) & 1 ? 1.0 : -1.0);
    } else {
      const int mu = e & 3, k = (e - 144) >> 2;
      const int c = k / 3, cp = k % 3;
      const double2 h = np_pair64(S + 3 * mu + (c + 1) % 3, 12, S + 3 * (mu ^ 1) + (c + 2) % 3, 12, (cp + 1) % 3, (cp + 2) % 3);
      const double2* v = Vv + c * 24;
      const double2 u0 = v[cp], u1 = v[6 + cp], u2 = v[12 + 3 + cp], u3 = v[12 + 9 + cp];
      np_fma(w1, h, make_double2(u0.x - u1.x + (u2.x - u3.x), u0.y - u1.y + (u2.y - u3.y)), mu & 1 ? 1.0 : -1.0);
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(NP_T, 3) k_nucleon_point(int S3, int groups, long long V, const double2* prop,
                                                           long long prop_stride, int t0, double2* partial) {
  extern __shared__ __align__(16) int4 np_sm[];
  int4* S = np_sm;                         // [site][column 3 nu + b][row 3 mu + a]
  int4* Vv = S + NP_SITES * 144;           // [site][c][g][column]
  int4* Z = Vv + NP_SITES * 72;            // [site][g][c'][row]
  __shared__ int blk[NP_SITES][9];         // largest exponent of the entries of colours (a, b)
  __shared__ int scale[NP_SITES][7];       // rho_a, kappa_b and their sum
  __shared__ int large[NP_SITES][12];      // rows' large entries
  __shared__ int found[NP_SITES];          // np_large_terms; 0 for a site that is not summed in fixed point
  enum { FIXED, ZERO, NONFINITE, TINY };
  __shared__ int kind[NP_SITES];
  const int slice = blockIdx.y;
  const double2* P = prop + (long long)blockIdx.z * prop_stride + (long long)(t0 + slice) * S3 * 12;
  double2 w1 = make_double2(0.0, 0.0), w2 = make_double2(0.0, 0.0);
  for (int grp = 0; grp < groups; grp++) {
    const int y0 = (blockIdx.x * groups + grp) * NP_SITES;
    const int ns = min(NP_SITES, S3 - y0);
    if (ns <= 0) break;
    if (grp) __syncthreads();
    for (int q = threadIdx.x; q < NP_SITES * 12; q += NP_T) {
      large[q / 12][q % 12] = 0;
      if (q < NP_SITES * 9) blk[q / 9][q % 9] = 1;
      if (q < NP_SITES) found[q] = 0;
    }
    __syncthreads();
    double2* Sd = reinterpret_cast<double2*>(S);
    for (int q = threadIdx.x; q < ns * 144; q += NP_T) {
      const int col = q / (ns * 12), r = q - col * (ns * 12);
      const int site = r / 12, row = r - site * 12;
      const double2 v = __ldg(P + ((long long)col * V + y0) * 12 + r);
      Sd[site * 144 + col * 12 + row] = v;
      atomicMax(&blk[site][3 * (row % 3) + col % 3], max(fx_exponent(v.x), fx_exponent(v.y)));
    }
    __syncthreads();
    if (threadIdx.x < ns) {
      const int* e = blk[threadIdx.x];
      int* sc = scale[threadIdx.x];
      int rho[3], kap[3], top = 1;
#pragma unroll
      for (int b = 0; b < 3; b++) kap[b] = max(max(e[b], e[3 + b]), e[6 + b]);
#pragma unroll
      for (int a = 0; a < 3; a++) rho[a] = max(max(e[3 * a] - kap[0], e[3 * a + 1] - kap[1]), e[3 * a + 2] - kap[2]);
#pragma unroll
      for (int b = 0; b < 3; b++) {
        top = max(top, kap[b]);
        kap[b] = max(max(e[b] - rho[0], e[3 + b] - rho[1]), e[6 + b] - rho[2]);
      }
      sc[6] = 0;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        sc[k] = rho[k];
        sc[3 + k] = kap[k];
        sc[6] += rho[k] + kap[k];
      }
      // (top 1: a product of three is zero; TINY: a term's last places may be denormals, which FP64 keeps)
      kind[threadIdx.x] = top == 2047 ? NONFINITE : top == 1 ? ZERO : sc[6] < 3 * 1023 - 900 ? TINY : FIXED;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < ns * 144; q += NP_T) {  // in place
      const int site = q / 144, e = q - site * 144, col = e / 12, row = e - col * 12;
      const int E = scale[site][row % 3] + scale[site][3 + col % 3];
      const double2 v = Sd[q];
      int4 l;
      fx_split(fx_of(v.x, E), l.x, l.y);
      fx_split(fx_of(v.y, E), l.z, l.w);
      S[q] = l;
      if (max(fx_exponent(v.x), fx_exponent(v.y)) >= E - 1) atomicOr(&large[site][row], 1 << col);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < ns * 72; q += NP_T) {
      const int site = q / 72, e = q - site * 72;
      {  // V: e = (c, g, column)
        const int c = e / 24, g = (e / 12) & 1, col = e % 12;
        Vv[q] = np_add(S[site * 144 + col * 12 + 3 * g + c], S[site * 144 + col * 12 + 3 * g + 6 + c]);
      }
      {  // Z: e = (g, c', row)
        const int g = e / 36, cp = (e / 12) % 3, row = e % 12;
        Z[q] = np_sub(S[site * 144 + (3 * g + cp) * 12 + row], S[site * 144 + (3 * g + 6 + cp) * 12 + row]);
      }
    }
    if (threadIdx.x < 8 * ns) {
      static_assert(NP_T == 8 * NP_SITES, "eight threads a site");
      const int site = threadIdx.x >> 3;
      const int f = kind[site] == FIXED ? np_large_terms(large[site], threadIdx.x & 7) : 0;
      if (f) atomicOr(&found[site], f);
    }
    __syncthreads();
    // H and T in units of 2^58 2^(the scales of their entries - 2 FX_BIAS)
    for (int q = threadIdx.x; q < ns * 144; q += NP_T) {
      const int site = q / 144, e = q - site * 144;
      if (found[site] != 3) continue;
      const int mu = (e & 7) >> 1, ai = e & 1, k = e >> 3;
      const int c = k / 6, g = (k / 3) & 1, cp = k % 3;
      const int a = (c + 1 + ai) % 3, b = (c + 2 - ai) % 3;
      const np_acc h = np_pair(S + site * 144 + 3 * mu + a, 12, Vv + site * 72 + (c * 2 + g) * 12, 1, (cp + 1) % 3,
                               (cp + 2) % 3);
      np_acc t = {0, 0, 0, 0};
      int sh;
      const int4 hl = np_limbs(h, sh);
      np_mac<false>(t, hl, Z[site * 72 + (g * 3 + cp) * 12 + 3 * (mu ^ 1) + b]);
      const int s = scale[site][6] - 3 * FX_BIAS + 2 * 58 + sh;
      const double re = fx_sum<29, false>(t.hr, t.cr, s), im = fx_sum<29, false>(t.hi, t.ci, s);
      const bool pos = (mu ^ ai) & 1;  // eps_{abc} cg(mu) = +1
      w2.x += pos ? re : -re;
      w2.y += pos ? im : -im;
    }
    for (int q = threadIdx.x; q < ns * 36; q += NP_T) {
      const int site = q / 36, e = q - site * 36;
      if (found[site] != 3) continue;
      const int mu = e & 3, k = e >> 2;
      const int c = k / 3, cp = k % 3;
      const int a0 = (c + 1) % 3, b0 = (c + 2) % 3;
      const np_acc h = np_pair(S + site * 144 + 3 * mu + a0, 12, S + site * 144 + 3 * (mu ^ 1) + b0, 12, (cp + 1) % 3,
                               (cp + 2) % 3);
      // U, four entries of V: below 2^60, shifted by 3 into limbs
      const int4* v = Vv + site * 72 + c * 24;
      const int4 u0 = v[cp], u1 = v[6 + cp], u2 = v[12 + 3 + cp], u3 = v[12 + 9 + cp];
      int4 u;
      fx_split((fx_join(u0.x, u0.y) - fx_join(u1.x, u1.y) + fx_join(u2.x, u2.y) - fx_join(u3.x, u3.y) + 4) >> 3, u.x, u.y);
      fx_split((fx_join(u0.z, u0.w) - fx_join(u1.z, u1.w) + fx_join(u2.z, u2.w) - fx_join(u3.z, u3.w) + 4) >> 3, u.z, u.w);
      np_acc t = {0, 0, 0, 0};
      int sh;
      const int4 hl = np_limbs(h, sh);
      np_mac<false>(t, hl, u);
      const int s = scale[site][6] - 3 * FX_BIAS + 2 * 58 + sh + 3;
      const double re = fx_sum<29, false>(t.hr, t.cr, s), im = fx_sum<29, false>(t.hi, t.ci, s);
      w1.x += mu & 1 ? re : -re;
      w1.y += mu & 1 ? im : -im;
    }
    // the other sites, one at a time
    for (int site = 0; site < ns; site++) {
      if (found[site] == 3 || kind[site] == ZERO) continue;
      if (kind[site] == NONFINITE) {
        if (threadIdx.x == 0) w2.x = w2.y = w1.x = w1.y = nan("");
        continue;
      }
      __syncthreads();  // the site's limbs are read no more
      for (int q = threadIdx.x; q < 144; q += NP_T)
        Sd[q] = __ldg(P + ((long long)(q / 12) * V + y0 + site) * 12 + q % 12);
      np_site64(Sd, reinterpret_cast<double2*>(Vv), reinterpret_cast<double2*>(Z), w1, w2);
    }
  }
  __shared__ double red[4][NP_T / 32];
  double v[4] = {w1.x, w1.y, 0.5 * w2.x, 0.5 * w2.y};
#pragma unroll
  for (int q = 0; q < 4; q++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = v[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double r = 0.0;
    for (int w = 0; w < NP_T / 32; w++) r += red[threadIdx.x][w];
    const long long o = (((long long)blockIdx.z * gridDim.y + slice) * gridDim.x + blockIdx.x) * 2;
    reinterpret_cast<double*>(partial + o)[threadIdx.x] = r;
  }
}

// W[p][t] = sum over the blocks of (prop p, slice t), one warp each, in a fixed order.
__global__ void __launch_bounds__(128) k_nucleon_point_sum(int nblk, int n, const double2* partial, double2* W) {
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  const double2* p = partial + (long long)i * nblk * 2;
  for (int b = lane; b < nblk; b += 32) {
    const double2 x = p[2 * b], y = p[2 * b + 1];
    v[0] += x.x;
    v[1] += x.y;
    v[2] += y.x;
    v[3] += y.y;
  }
#pragma unroll
  for (int q = 0; q < 4; q++)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  if (lane == 0) {
    W[2 * i] = make_double2(v[0], v[1]);
    W[2 * i + 1] = make_double2(v[2], v[3]);
  }
}

// The tensor-core block kernel (nucleon_tc.cu) unless LQCD_NUCLEON_TC=0 selects the FP32-FMA
// one; read at every call
bool use_tensor_cores() {
  const char* e = getenv("LQCD_NUCLEON_TC");
  return e ? atoi(e) != 0 : true;
}

}  // namespace

// Stages per block: as many as leave two rounds of three blocks an SM, so that small calls still
// fill the chip (a block's final sums cost a fiftieth of one stage).
static int np_groups(long long S3, int n_prop, int n_t) {
  const long long total = (S3 + NP_SITES - 1) / NP_SITES * n_t * n_prop;
  return (int)std::max(1LL, std::min((long long)NP_GROUPS, total / (152 * 3 * 2)));
}
static int np_blocks(long long S3, int groups) {
  return (int)((S3 + NP_SITES * groups - 1) / (NP_SITES * groups));
}

int lq_nucleon_point(const lqcd_lattice* L, int n_prop, const double2* prop, int t0, int n_t, double2* partial,
                     double2* W, cudaStream_t st) {
  const int S3 = (int)L->S3;
  const int groups = np_groups(S3, n_prop, n_t), nblk = np_blocks(S3, groups);
  if (cudaFuncSetAttribute(k_nucleon_point, cudaFuncAttributeMaxDynamicSharedMemorySize, NP_SMEM) != cudaSuccess) {
    cudaGetLastError();
    lq_set_error("nucleon_point: shared-memory opt-in failed");
    return LQCD_ECUDA;
  }
  k_nucleon_point<<<dim3((unsigned)nblk, (unsigned)n_t, (unsigned)n_prop), NP_T, NP_SMEM, st>>>(
      S3, groups, L->V, prop, (long long)12 * L->V * 12, t0, partial);
  RC_LAUNCH();
  k_nucleon_point_sum<<<(unsigned)((n_t * n_prop + 3) / 4), 128, 0, st>>>(nblk, n_t * n_prop, partial, W);
  return launched_here();
}

long long lq_nucleon_point_partial_words(const lqcd_lattice* L, int n_prop, int n_t) {
  return (long long)np_blocks(L->S3, np_groups(L->S3, n_prop, n_t)) * n_t * n_prop * 2;
}

extern "C" int lqcd_nucleon_point(lqcd_lattice* L, int n_prop, const double* prop, int t0, int n_t, double* W,
                                  void* stream) {
  if (!L || !prop || !W || n_prop < 1 || n_t < 1 || t0 < 0 || t0 + n_t > L->dims[0] || n_prop > 65535) {
    lq_set_error("nucleon_point: bad arguments (1 <= n_prop, slices t0..t0+n_t-1 inside the lattice)");
    return LQCD_EBADARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  void* partial = nullptr;
  const size_t bytes = sizeof(double2) * (size_t)lq_nucleon_point_partial_words(L, n_prop, n_t);
  if (cudaMallocAsync(&partial, bytes, st) != cudaSuccess) {
    cudaGetLastError();
    lq_set_error("nucleon_point: device allocation failed");
    return LQCD_ENOMEM;
  }
  const int rc = lq_nucleon_point(L, n_prop, (const double2*)prop, t0, n_t, (double2*)partial, (double2*)W, st);
  cudaFreeAsync(partial, st);
  return rc;
}

extern "C" int lqcd_level_mean(long long size, int count, const double* in, double* out, void* stream) {
  if (!in || !out || size < 1 || count < 1) {
    lq_set_error("level_mean: bad arguments");
    return LQCD_EBADARG;
  }
  long long blocks = (size + 511) / 512;
  if (blocks > 152 * 32) blocks = 152 * 32;
  k_level_mean<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(size, count, 1.0 / count, (count & (count - 1)) == 0,
                                                                 (const double2*)in, (double2*)out);
  return launched_here();
}

extern "C" int lqcd_nucleon_blocks(lqcd_lattice* L, const lqcd_slab* slab, int n, const double* s, int conj, int t0,
                                   int n_t, double* B, void* stream) {
  if (!L || !slab || !s || !B || n < 1 || n > 1024 || n_t < 1 || slab->t0 < 0 || slab->t1 < slab->t0 ||
      slab->t1 >= L->dims[0] || t0 < slab->t0 || t0 + n_t - 1 > slab->t1) {
    lq_set_error("nucleon_blocks: bad arguments (1 <= n <= 1024, slices t0..t0+n_t-1 inside the slab)");
    return LQCD_EBADARG;
  }
  const int S3 = (int)L->S3;
  const long long nsite = (long long)(slab->t1 - slab->t0 + 1) * S3;
  if (use_tensor_cores())
    return lq_nucleon_blocks_tc(n, nsite, (const double2*)s, conj, S3, (long long)(t0 - slab->t0) * S3, n_t,
                                (double2*)B, (cudaStream_t)stream);
  const int nti = (n + TI - 1) / TI, ntj = (n + TJ - 1) / TJ, ntk = (n + TK - 1) / TK;
  {
    // static + dynamic shared memory exceed the 48 KB default: opt in once per device
    static std::mutex mu;
    static std::vector<int> opted;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
      cudaGetLastError();
      lq_set_error("nucleon_blocks: no current device");
      return LQCD_ECUDA;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (std::find(opted.begin(), opted.end(), dev) == opted.end()) {
      if (cudaFuncSetAttribute(k_nucleon_block, cudaFuncAttributeMaxDynamicSharedMemorySize, TOT_BYTES) !=
          cudaSuccess) {
        cudaGetLastError();
        lq_set_error("nucleon_blocks: shared-memory opt-in failed");
        return LQCD_ECUDA;
      }
      opted.push_back(dev);
    }
  }
  k_nucleon_block<<<dim3((unsigned)(nti * ntj), (unsigned)ntk, (unsigned)n_t), 256, TOT_BYTES, (cudaStream_t)stream>>>(
      n, nsite, (const double2*)s, conj, S3, (long long)(t0 - slab->t0) * S3, S3, (double2*)B);
  return launched_here();
}

extern "C" int lqcd_nucleon_contract(int n, int n_x, const double* B_xi, int n_y, const double* B_eta, double* W,
                                     void* stream) {
  if (!B_xi || !B_eta || !W || n < 1 || n > 1024 || n_x < 1 || n_y < 1 || (long long)n_x * n_y >= (1LL << 31)) {
    lq_set_error("nucleon_contract: bad arguments");
    return LQCD_EBADARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  // parts: about four blocks per SM over all pairs, no more than there are tiles
  const long long ngy = (n_y + CT_NY - 1) / CT_NY, nt = (n + CT - 1) / CT;
  long long nsplit = (152 * 4 + n_x * ngy - 1) / (n_x * ngy);
  nsplit = std::max(1LL, std::min(nsplit, (long long)n * nt * nt));
  void* scratch = nullptr;
  if (nsplit > 1 && cudaMallocAsync(&scratch, sizeof(double) * 4 * (size_t)(n_x * (long long)n_y * nsplit), st) != cudaSuccess) {
    cudaGetLastError();
    scratch = nullptr;
    nsplit = 1;  // no scratch to be had: one part per pair, summed in place
  }
  double* part = scratch ? (double*)scratch : W;
  k_nucleon_contract<<<(unsigned)(n_x * ngy * nsplit), CT * CT, 0, st>>>(n, n_y, (int)nsplit, (const double2*)B_xi,
                                                                         (const double2*)B_eta, part);
  int rc = launched_here();
  if (!rc) {
    k_contract_sum<<<(unsigned)((long long)n_x * n_y), 128, 0, st>>>((int)nsplit, part, W);
    rc = launched_here();
  }
  if (scratch) cudaFreeAsync(scratch, st);
  return rc;
}
