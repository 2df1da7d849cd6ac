// Gauge-field preparation: even-odd link packing in three precisions with
// an SU(3) check, and the clover blocks A(x) with their inverses.
//
// Clover term (Sheikholeslami-Wohlert), added to the diagonal of D:
//   A(x) = 1/(2 kappa) + c_sw (i/4) sum_{mu,nu} sigma_mu_nu Fhat_mu_nu(x),
//   Fhat_mu_nu = (Q_mu_nu - Q_mu_nu^dag) / 8,  Q = the four plaquette leaves.
// In the chiral basis sigma_mu_nu = (i/2)[g_mu, g_nu] is block diagonal:
//   sigma_0k = diag(+s_k, -s_k),  sigma_jk = -eps_jkl diag(s_l, s_l),
// so with E_l = Fhat_0l and M_1 = Fhat_23, M_2 = Fhat_31, M_3 = Fhat_12,
//   A = diag(B+, B-),  B+- = 1/(2 kappa) + sum_l s_l (x) H+-_l,
//   H+-_l = c_sw (i/2) (+-E_l - M_l)   (Hermitian 3x3),
//   B = [[d + H_3, H_1 - i H_2], [H_1 + i H_2, d - H_3]].
// Open time BC: the link U_0 leaving the last time slice is absent, so every
// leaf through it is zero.
#include <algorithm>
#include <cstdio>

#include "internal.h"

namespace lq {

typedef cx<double> cd;

LQ_DI su3<double> ld_nat(const double2* U, long long i, int mu) {
  su3<double> u;
  const double2* b = U + (i * 4 + mu) * 9;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    double2 v = b[k];
    u.m[k / 3][k % 3] = {v.x, v.y};
  }
  return u;
}

LQ_DI void nat_coords(const Geom& g, long long i, int x[4]) {
  x[3] = (int)(i % g.L[3]);
  i /= g.L[3];
  x[2] = (int)(i % g.L[2]);
  i /= g.L[2];
  x[1] = (int)(i % g.L[1]);
  x[0] = (int)(i / g.L[1]);
}

// max(a, b) that keeps a NaN of either
LQ_DI double max_nan(double a, double b) { return a >= b ? a : (a == a ? b : a); }

// 3x3 complex matrices in fixed point (fxnum.cuh): entries q 2^-58 in limbs, as the links are stored.  A
// product is 27 complex multiply-adds of 12 integer ones each, a tenth of the time of the FP64
// product, and its entries are rounded at 2^-58 (FP64 rounds an entry of size 1 at 2^-53).
struct mcl {
  int4 m[3][3];  // (re1, re0, im1, im0)
};

LQ_DI void mc_mac(long long& hh, long long& cr, int a1, int a0, int b1, int b0) {
  mad_wide(hh, a1, b1);
  mad_wide(cr, a1, b0);
  mad_wide(cr, a0, b1);
}
// entry of a product as 64-bit integers: sum over k of a_k b_k with the imaginary part of a (CA) or b (CB) negated
template <bool CA, bool CB, int N = 3>
LQ_DI longlong2 mc_dot(const int4 (&a)[N], const int4 (&b)[N]) {
  long long hr = 0, cr = 1ll << 28, hi = 0, ci = 1ll << 28;  // (the halves round the shifts below)
#pragma unroll
  for (int k = 0; k < N; k++) {
    const int ai1 = CA ? -a[k].z : a[k].z, ai0 = CA ? -a[k].w : a[k].w;
    const int bi1 = CB ? -b[k].z : b[k].z, bi0 = CB ? -b[k].w : b[k].w;
    mc_mac(hr, cr, a[k].x, a[k].y, b[k].x, b[k].y);
    mc_mac(hr, cr, -ai1, -ai0, bi1, bi0);
    mc_mac(hi, ci, a[k].x, a[k].y, bi1, bi0);
    mc_mac(hi, ci, ai1, ai0, b[k].x, b[k].y);
  }
  return make_longlong2(hr + (cr >> 29), hi + (ci >> 29));
}
LQ_DI int4 mc_limbs(longlong2 q) {
  int4 v;
  fx_split(q.x, v.x, v.y);
  fx_split(q.y, v.z, v.w);
  return v;
}
// ------------------------------------------------------------- link packing
LQ_DI int4 limbs_of(double a, double b, int e) {
  int4 v;
  fx_split(fx_of(a, e), v.x, v.y);
  fx_split(fx_of(b, e), v.z, v.w);
  return v;
}

// Square of a link's deviation from SU(3): the largest entry of U U^dag - 1 (Hermitian: the upper triangle) and det U - 1.
LQ_DI double su3_deviation(const su3<double>& u) {
  double dev = 0.0;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++) {
      cd e = {a == b ? -1.0 : 0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 3; k++) fma_cc(e, u.m[b][k], u.m[a][k]);
      dev = max_nan(dev, norm2(e));
    }
  cd det = {-1.0, 0.0};
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const cd minor = u.m[1][k1] * u.m[2][k2] - u.m[1][k2] * u.m[2][k1];
    fma_c(det, u.m[0][k], minor);
  }
  return max_nan(dev, norm2(det));
}
// The same from the limbs (an eighth of the FP64 operations): false where the link is so far from SU(3), by 2^-10, that a
// sum might not fit.
LQ_DI bool su3_deviation(const int4 (&u)[3][3], double& dev) {
  bool near = true;
  auto add = [&](longlong2 v, bool one) {
    if (one) v.x -= 1ll << 58;
    near = near && llabs(v.x) < (1ll << 48) && llabs(v.y) < (1ll << 48);
    const double re = fx_to_double<false>(v.x, -58), im = fx_to_double<false>(v.y, -58);
    dev = fmax(dev, re * re + im * im);
  };
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = a; b < 3; b++) add(mc_dot<false, true>(u[a], u[b]), a == b);
  int4 m[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    const int4 n = u[1][k2];
    const int4 l[2] = {u[1][k1], make_int4(-n.x, -n.y, -n.z, -n.w)}, r[2] = {u[2][k2], u[2][k1]};
    m[k] = mc_limbs(mc_dot<false, false>(l, r));
  }
  add(mc_dot<false, false>(u[0], m), true);
  return near;
}

// Natural to packed links in the three precisions and the largest deviation from SU(3), a thread a link (direction
// blockIdx.y).  24^3 x 48: 0.75 ms with a thread a site, the deviation in FP64 and an atomic a thread; 0.36 ms so.
__global__ void __launch_bounds__(128) k_pack_links(Geom g, const double2* U, int4* U64, float4* U32, uint2* U16,
                                                    unsigned long long* maxdev) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long dv = 0;
  if (i < 2 * g.Vh) {
    const int mu = blockIdx.y;
    int x[4];
    nat_coords(g, i, x);
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const long long cb = i >> 1;
    const su3<double> u = ld_nat(U, i, mu);
    int4 q[3][3];
    int ex = 0;
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const cd e = u.m[k / 3][k % 3];
      q[k / 3][k % 3] = limbs_of(e.re, e.im, FX_LINK_E);
      ex = max(ex, max(fx_exponent(e.re), fx_exponent(e.im)));
    }
    double dev = 0.0;  // the largest of the squares, one root at the end
    if (ex > 1023 || !su3_deviation(q, dev)) dev = su3_deviation(u);  // (entries of 2 and more: not limbs)
    dev = sqrt(dev);
    if (!(dev == dev)) dev = 1e300;  // NaN counts as non-unitary
    dv = (unsigned long long)__double_as_longlong(dev);
    const long long base = (long long)(p * 4 + mu);
#pragma unroll
    for (int k = 0; k < 9; k++) U64[(base * 9 + k) * g.Vh + cb] = q[k / 3][k % 3];
    float r[12];
#pragma unroll
    for (int k = 0; k < 6; k++) {
      r[2 * k] = (float)u.m[k / 3][k % 3].re;
      r[2 * k + 1] = (float)u.m[k / 3][k % 3].im;
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
      U32[(base * 3 + k) * g.Vh + cb] = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
      __half2 h0 = __floats2half2_rn(r[4 * k], r[4 * k + 1]);
      __half2 h1 = __floats2half2_rn(r[4 * k + 2], r[4 * k + 3]);
      U16[(base * 3 + k) * g.Vh + cb] = make_uint2(*reinterpret_cast<uint32_t*>(&h0), *reinterpret_cast<uint32_t*>(&h1));
    }
  }
#pragma unroll
  for (int k = 16; k; k >>= 1) dv = max(dv, __shfl_xor_sync(0xffffffffu, dv, k));
  if ((threadIdx.x & 31) == 0 && dv) atomicMax(maxdev, dv);
}

// ------------------------------------------------------------------ clover
LQ_DI mcl link_bc(const Geom& g, const int4* U, const int x[4], int mu) {
  mcl u;
  if (g.bc_t == 0 && mu == 0 && x[0] == g.L[0] - 1) {
#pragma unroll
    for (int k = 0; k < 9; k++) u.m[k / 3][k % 3] = make_int4(0, 0, 0, 0);
    return u;
  }
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const int4* b = U + (long long)(p * 4 + mu) * 9 * g.Vh + eo_index(g, x);
#pragma unroll
  for (int k = 0; k < 9; k++) u.m[k / 3][k % 3] = __ldg(b + (long long)k * g.Vh);
  return u;
}

LQ_DI longlong2 mm_ij(const mcl& a, const mcl& b, int i, int j) {  // (a b)_ij
  const int4 r[3] = {a.m[i][0], a.m[i][1], a.m[i][2]}, c[3] = {b.m[0][j], b.m[1][j], b.m[2][j]};
  return mc_dot<false, false>(r, c);
}
LQ_DI longlong2 mmd_ij(const mcl& a, const mcl& b, int i, int j) {  // (a b^dag)_ij
  const int4 r[3] = {a.m[i][0], a.m[i][1], a.m[i][2]}, c[3] = {b.m[j][0], b.m[j][1], b.m[j][2]};
  return mc_dot<false, true>(r, c);
}
LQ_DI longlong2 mdm_ij(const mcl& a, const mcl& b, int i, int j) {  // (a^dag b)_ij
  const int4 r[3] = {a.m[0][i], a.m[1][i], a.m[2][i]}, c[3] = {b.m[0][j], b.m[1][j], b.m[2][j]};
  return mc_dot<true, false>(r, c);
}
LQ_DI mcl mc_mul(const mcl& a, const mcl& b) {
  mcl r;
#pragma unroll
  for (int k = 0; k < 9; k++) r.m[k / 3][k % 3] = mc_limbs(mm_ij(a, b, k / 3, k % 3));
  return r;
}
// a p^dag - q^dag b
LQ_DI mcl mc_staple(const mcl& a, const mcl& p, const mcl& q, const mcl& b) {
  mcl r;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    const longlong2 x = mmd_ij(a, p, k / 3, k % 3), y = mdm_ij(q, b, k / 3, k % 3);
    r.m[k / 3][k % 3] = mc_limbs(make_longlong2(x.x - y.x, x.y - y.y));
  }
  return r;
}

LQ_DI void shift(const Geom& g, const int x[4], int mu, int d, int y[4]) {
#pragma unroll
  for (int k = 0; k < 4; k++) {  // (no indexing by mu: the coordinates stay in registers)
    int v = x[k] + (k == mu ? d : 0);
    if (v < 0) v += g.L[k];
    if (v >= g.L[k]) v -= g.L[k];
    y[k] = v;
  }
}

// Fhat_mu_nu(x) = (Q - Q^dag)/8, Q = sum of the 4 leaves at x (mu -> nu):
//   L1 = U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag,
//   L2 = U_nu(x) U_mu(x+nu-mu)^dag U_nu(x-mu)^dag U_mu(x-mu),
//   L3 = U_mu(x-mu)^dag U_nu(x-mu-nu)^dag U_mu(x-mu-nu) U_nu(x-nu),
//   L4 = U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) U_mu(x)^dag.
// Q - Q^dag = M - M^dag with L3, L4 replaced by -L3^dag, -L4^dag, which pairs the leaves on a
// common outer link: ten products a plane instead of twelve.
//   M = U_mu(x) { U_nu(x+mu) [U_nu(x) U_mu(x+nu)]^dag - [U_mu(x-nu) U_nu(x-nu+mu)]^dag U_nu(x-nu) }
//     + { U_nu(x) [U_nu(x-mu) U_mu(x-mu+nu)]^dag - [U_mu(x-mu-nu) U_nu(x-nu)]^dag U_nu(x-mu-nu) } U_mu(x-mu)
// The result is 8 Fhat in units of 2^-58 (anti-Hermitian; the entries (i, j), i >= j, are filled in).
LQ_DI void fhat(const Geom& g, const int4* U, const int x[4], int mu, int nu, longlong2 (&f)[3][3]) {
  int xpm[4], xpn[4], xmm[4], xmn[4], xmmpn[4], xmmmn[4], xmnpm[4];
  shift(g, x, mu, 1, xpm);
  shift(g, x, nu, 1, xpn);
  shift(g, x, mu, -1, xmm);
  shift(g, x, nu, -1, xmn);
  shift(g, xmm, nu, 1, xmmpn);
  shift(g, xmm, nu, -1, xmmmn);
  shift(g, xmn, mu, 1, xmnpm);
  const mcl un = link_bc(g, U, xmn, nu);
  const mcl t1 = mc_staple(link_bc(g, U, xpm, nu), mc_mul(link_bc(g, U, x, nu), link_bc(g, U, xpn, mu)),
                           mc_mul(link_bc(g, U, xmn, mu), link_bc(g, U, xmnpm, nu)), un);
  longlong2 q[3][3];
  {
    const mcl u = link_bc(g, U, x, mu);
#pragma unroll
    for (int k = 0; k < 9; k++) q[k / 3][k % 3] = mm_ij(u, t1, k / 3, k % 3);
  }
  const mcl t2 = mc_staple(link_bc(g, U, x, nu), mc_mul(link_bc(g, U, xmm, nu), link_bc(g, U, xmmpn, mu)),
                           mc_mul(link_bc(g, U, xmmmn, mu), un), link_bc(g, U, xmmmn, nu));
  {
    const mcl u = link_bc(g, U, xmm, mu);
#pragma unroll
    for (int k = 0; k < 9; k++) {
      const longlong2 v = mm_ij(t2, u, k / 3, k % 3);
      q[k / 3][k % 3].x += v.x;
      q[k / 3][k % 3].y += v.y;
    }
  }
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b <= a; b++) f[a][b] = make_longlong2(q[a][b].x - q[b][a].x, q[a][b].y + q[b][a].y);
}

// Pack the 6x6 Hermitian block B into 36 reals: 6 diagonal, then the 15
// entries below the diagonal row by row.
LQ_DI void pack_herm6(const cd B[6][6], double out[36]) {
#pragma unroll
  for (int r = 0; r < 6; r++) out[r] = B[r][r].re;
  int q = 6;
#pragma unroll
  for (int r = 1; r < 6; r++)
#pragma unroll
    for (int c = 0; c < r; c++) {
      // Hermitian part of the pair (r,c), (c,r)
      out[q] = 0.5 * (B[r][c].re + B[c][r].re);
      out[q + 1] = 0.5 * (B[r][c].im - B[c][r].im);
      q += 2;
    }
}

// In-place Gauss-Jordan inversion with partial pivoting (6x6 complex), all indices static so that
// the block stays in registers (row swaps are selects).  Returns false for a singular block.
LQ_DI bool invert6(cd (&M)[6][6]) {
  int piv[6];
  bool ok = true;
#pragma unroll
  for (int col = 0; col < 6; col++) {
    int p = col;
    double best = norm2(M[col][col]);
#pragma unroll
    for (int r = col + 1; r < 6; r++) {
      const double v = norm2(M[r][col]);
      if (v > best) {
        best = v;
        p = r;
      }
    }
    piv[col] = p;
    if (!(best > 0.0)) ok = false;
#pragma unroll
    for (int r = col + 1; r < 6; r++) {
      const bool sw = r == p;
#pragma unroll
      for (int c = 0; c < 6; c++) {
        const cd a = M[col][c], b = M[r][c];
        M[col][c] = {sw ? b.re : a.re, sw ? b.im : a.im};
        M[r][c] = {sw ? a.re : b.re, sw ? a.im : b.im};
      }
    }
    const cd d = M[col][col];
    const double dn = norm2(d);
    const cd inv = {d.re / dn, -d.im / dn};
    M[col][col] = {1.0, 0.0};
#pragma unroll
    for (int c = 0; c < 6; c++) M[col][c] = M[col][c] * inv;
#pragma unroll
    for (int r = 0; r < 6; r++) {
      if (r == col) continue;
      const cd mf = {-M[r][col].re, -M[r][col].im};
      M[r][col] = {0.0, 0.0};
#pragma unroll
      for (int c = 0; c < 6; c++) fma_c(M[r][c], mf, M[col][c]);
    }
  }
  // undo the row swaps on the columns, last first
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const int col = 5 - k;
#pragma unroll
    for (int c = col + 1; c < 6; c++) {
      const bool sw = c == piv[col];
#pragma unroll
      for (int r = 0; r < 6; r++) {
        const cd a = M[r][col], b = M[r][c];
        M[r][col] = {sw ? b.re : a.re, sw ? b.im : a.im};
        M[r][c] = {sw ? a.re : b.re, sw ? a.im : b.im};
      }
    }
  }
  return ok;
}

// i Fhat of one plane per thread (Hermitian: 3 real diagonal entries, then the entries (1,0), (2,0),
// (2,1)), planes 0-2 = (0,1) (0,2) (0,3), 3-5 = (2,3) (3,1) (1,2), into G[plane * 9 + k][parity][site],
// for the h sites of either parity from c0 (the 2 h sites from 2 c0 in natural order: a block's threads share
// links).
//
// 10 products of 3 x 3 matrices a plane in fixed point (2160 complex products a site and 6 planes), on the integer pipe: links
// have |U| <= 1 and need no exponent.  A thread a plane keeps the matrices in registers, where one thread for the whole
// site spilled 1.7 KB.  24^3 x 48, with k_clover_blocks: 20.6 ms with twelve products a plane, products
// without fused multiply-adds, an augmented elimination and all in one thread; 8.9 ms with the ten products in FP64, at
// the FP64 pipe's rate; 5.1 ms so (3.1 ms this kernel).
__global__ void __launch_bounds__(128) k_fhat(Geom g, const int4* U, long long c0, long long h, double* G) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * h) return;
  int x[4];
  nat_coords(g, 2 * c0 + i, x);
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const int pl = blockIdx.y;
  const int mu = pl < 3 ? 0 : (pl == 3 ? 2 : pl == 4 ? 3 : 1);
  const int nu = pl < 3 ? pl + 1 : (pl == 3 ? 3 : pl == 4 ? 1 : 2);
  longlong2 f[3][3];
  fhat(g, U, x, mu, nu, f);
  constexpr int EX = FX_LINK_E - FX_BIAS - 3;
  const long long nc = 2 * h;
  double* out = G + pl * 9 * nc + p * h + (i >> 1);
#pragma unroll
  for (int a = 0; a < 3; a++) out[a * nc] = -fx_to_double<false>(f[a][a].y, EX);
  const int ra[3] = {1, 2, 2}, rb[3] = {0, 0, 1};
#pragma unroll
  for (int k = 0; k < 3; k++) {  // i f
    out[(3 + 2 * k) * nc] = -fx_to_double<false>(f[ra[k]][rb[k]].y, EX);
    out[(4 + 2 * k) * nc] = fx_to_double<false>(f[ra[k]][rb[k]].x, EX);
  }
}

LQ_DI int block_exponent(const double pk[36]) {
  int e = 1;
#pragma unroll
  for (int k = 0; k < 36; k++) e = max(e, fx_exponent(pk[k]));
  return e;
}

// The two clover blocks B+- = 1/(2 kappa) + sum_l s_l (x) H+-_l, H+-_l = (c_sw/2)(+-i E_l - i M_l), from G,
// and their inverses on even sites; one thread per (site, block), the h sites of either parity from c0.
__global__ void __launch_bounds__(128) k_clover_blocks(Geom g, long long c0, long long h, const double* G, double kappa,
                                                       double csw, int4* A64, int4* Ai64, int* A64e, int* Ai64e,
                                                       float4* A32, float4* Ai32, int* fail) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nc = 2 * h, Vh = g.Vh;
  if (i >= nc) return;
  const int p = i >= h;
  const long long cb = c0 + i - p * h;
  const int blk = blockIdx.y;
  const double d = 1.0 / (2.0 * kappa);
  cd H[3][3][3];
#pragma unroll
  for (int l = 0; l < 3; l++) {
    double h[9];
#pragma unroll
    for (int k = 0; k < 9; k++) {
      if (csw == 0.0) {
        h[k] = 0.0;
      } else {
        const double e = G[(l * 9 + k) * nc + i], m = G[((3 + l) * 9 + k) * nc + i];
        h[k] = (0.5 * csw) * (blk == 0 ? e - m : -e - m);
      }
    }
#pragma unroll
    for (int a = 0; a < 3; a++) H[l][a][a] = {h[a], 0.0};
    const int ra[3] = {1, 2, 2}, rb[3] = {0, 0, 1};
#pragma unroll
    for (int k = 0; k < 3; k++) {
      H[l][ra[k]][rb[k]] = {h[3 + 2 * k], h[4 + 2 * k]};
      H[l][rb[k]][ra[k]] = {h[3 + 2 * k], -h[4 + 2 * k]};
    }
  }
  cd B[6][6];
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const cd dd = {a == b ? d : 0.0, 0.0};
      B[a][b] = dd + H[2][a][b];
      B[3 + a][3 + b] = dd - H[2][a][b];
      B[a][3 + b] = H[0][a][b] - ti(H[1][a][b]);
      B[3 + a][b] = H[0][a][b] + ti(H[1][a][b]);
    }
  double pk[36];
  pack_herm6(B, pk);
  int ex = block_exponent(pk);
  A64e[((long long)p * 2 + blk) * Vh + cb] = ex;
#pragma unroll
  for (int k = 0; k < 18; k++) A64[((long long)p * 36 + blk * 18 + k) * Vh + cb] = limbs_of(pk[2 * k], pk[2 * k + 1], ex);
#pragma unroll
  for (int k = 0; k < 9; k++)
    A32[((long long)p * 18 + blk * 9 + k) * Vh + cb] =
        make_float4((float)pk[4 * k], (float)pk[4 * k + 1], (float)pk[4 * k + 2], (float)pk[4 * k + 3]);
  if (p != 0) return;
  if (!invert6(B)) {
    atomicExch(fail, 1);
#pragma unroll
    for (int r = 0; r < 6; r++)
#pragma unroll
      for (int c = 0; c < 6; c++) B[r][c] = {0.0, 0.0};
  }
  pack_herm6(B, pk);
  ex = block_exponent(pk);
  Ai64e[(long long)blk * Vh + cb] = ex;
#pragma unroll
  for (int k = 0; k < 18; k++) Ai64[((long long)blk * 18 + k) * Vh + cb] = limbs_of(pk[2 * k], pk[2 * k + 1], ex);
#pragma unroll
  for (int k = 0; k < 9; k++)
    Ai32[((long long)blk * 9 + k) * Vh + cb] =
        make_float4((float)pk[4 * k], (float)pk[4 * k + 1], (float)pk[4 * k + 2], (float)pk[4 * k + 3]);
}

}  // namespace lq

// ------------------------------------------------------------------ launchers
int lq_launch_pack_links(const lq::Geom& g, const double2* U, int4* U64, float4* U32, uint2* U16,
                         unsigned long long* maxdev, cudaStream_t st) {
  const long long V = 2 * g.Vh;
  lq::k_pack_links<<<dim3((unsigned)((V + 127) / 128), 4), 128, 0, st>>>(g, U, U64, U32, U16, maxdev);
  lq_count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Sites of a parity at a time: the planes' scratch (108 doubles a pair of sites, 453 MB) stops growing with the lattice.
// Runs small enough for L2 to hold it (1 << 17) gain nothing: 6.91 instead of 6.82 ms for 24^3 x 48.
constexpr long long CLOVER_CHUNK = 1 << 19;

int lq_launch_clover(const lq::Geom& g, const int4* U, double kappa, double csw, int4* A64, int4* Ai64,
                     int* A64e, int* Ai64e, float4* A32, float4* Ai32, int* fail, cudaStream_t st) {
  const long long Vh = g.Vh;
  long long chunk = std::min(Vh, CLOVER_CHUNK);
  double* G = nullptr;
  while (csw != 0.0 && cudaMallocAsync((void**)&G, sizeof(double) * 108 * chunk, st) != cudaSuccess) {
    cudaGetLastError();
    G = nullptr;
    if (chunk <= 1024) {
      lq_set_error("set_gauge: device allocation of the clover scratch failed");
      return LQCD_ENOMEM;
    }
    chunk = (chunk + 7) / 8;  // a nearly full device: shorter runs
  }
  for (long long c0 = 0; c0 < Vh; c0 += chunk) {
    const long long h = std::min(chunk, Vh - c0);
    const unsigned nb = (unsigned)((2 * h + 127) / 128);
    if (G) {
      lq::k_fhat<<<dim3(nb, 6), 128, 0, st>>>(g, U, c0, h, G);
      lq_count_launch();
    }
    lq::k_clover_blocks<<<dim3(nb, 2), 128, 0, st>>>(g, c0, h, G, kappa, csw, A64, Ai64, A64e, Ai64e, A32, Ai32, fail);
    lq_count_launch();
  }
  if (G) cudaFreeAsync(G, st);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
