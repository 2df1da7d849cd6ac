// Gauge-link force of the domain-local pseudofermion action
//   S = phi^dag (D_L^dag D_L)^{-1} phi,   X = (D_L^dag D_L)^{-1} phi,  Y = D_L X,
//   F^a_rho(x) = dS/domega  for U_rho(x) -> exp(i omega T_a) U_rho(x)
//              = -2 Re <Y, (dD_L/domega) X>,        T_a = lambda_a / 2.
//
// Hopping part (link l = U_rho(x), both ends in the slab, boundary sign f):
//   F^a = f Re tr[i T_a (l W1 - W2 l^dag)],
//   W1 = sum_s ((1 - g_rho) X(x+rho))_s (x) Y(x)_s^dag,
//   W2 = sum_s ((1 + g_rho) X(x))_s (x) Y(x+rho)_s^dag      (3x3 colour outer products).
// Clover part: with Xi_mn(z)[b][a] = sum_{s,t} sigma_mn[s][t] X(z)[t][b] conj(Y(z)[s][a])
// and K_mn = c_sw (i/4) (Xi_mn + Xi_mn^dag) (zero outside the slab),
//   F^a = -1/2 Re tr[i T_a G],  G = sum_{s != rho} ( l M_a + M_c ),
// where, for the plaquette above the link (corners x, x+rho, x+rho+s, x+s;
// b = U_s(x+rho), c = U_rho(x+s)^dag, d = U_s(x)^dag, K = K_{rho s}):
//   M_a = b c d K(x) + K(x+rho) b c d + b K(x+rho+s) c d + b c K(x+s) d,
// and for the plaquette below (w = x-s; a' = U_rho(w), b' = U_s(w+rho), d' = U_s(w)^dag):
//   M_c = -[d' K(w) a' b' + d' a' K(w+rho) b' + d' a' b' K(x+rho) + K(x) d' a' b'] l^dag.
// Each of the four leaves of the clover at z is one plaquette entered at a
// different corner, so summing over the link's two plaquettes per plane and
// their four corners covers every leaf that contains the link.
//
// What is computed.  K^dag = -K, so with the insertions on a link (z, s) of plane (rho, s),
//   B(z) = K_{rho s}(z) U_s(z) + U_s(z) K_{rho s}(z+s),
// shared by the two rho links that end in it,
//   M_a = B(x+rho) c d - b c B(x)^dag,
//   M_c l = B(w)^dag a' b' - d' a' B(w+rho),
// and, as Re tr[i T_a Z] sees only the anti-Hermitian part of Z, the terms of the form C l^dag
// join l C^dag: one product with l is left,
//   F^a = Re tr[i T_a l { f (W1 + W2^dag) - (1/2) sum_s (M_a - (M_c l)^dag) }].
// That is 31 3x3 products a link (25 here, 6 its share of the B) where the plain sum takes 63, and
// W1, W2 from half spinors.  Only links within one slice of the slab have a force; X, Y, K
// and B are held for those slices alone.  The kernels are bound by the FP64 pipe: on the 12-slice
// slab of 24^3 x 48 the plain form over all links took 47.6 ms, this one 5.3 ms.  Under open
// time BC the link leaving the last time slice is absent (zero): every
// product through it vanishes and its own force is zero.
#include <algorithm>

#include "dslash.cuh"
#include "internal.h"

namespace lq {

typedef cx<double> cd;
typedef su3<double> M3;

LQ_DI M3 zero3() {
  M3 r;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) r.m[a][b] = {0.0, 0.0};
  return r;
}
LQ_DI M3 mul(const M3& a, const M3& b) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      cd t = a.m[i][0] * b.m[0][j];
      fma_c(t, a.m[i][1], b.m[1][j]);
      fma_c(t, a.m[i][2], b.m[2][j]);
      r.m[i][j] = t;
    }
  return r;
}
LQ_DI M3 dagm(const M3& a) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) r.m[i][j] = conj(a.m[j][i]);
  return r;
}
LQ_DI M3 add(const M3& a, const M3& b) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) r.m[i][j] = a.m[i][j] + b.m[i][j];
  return r;
}
LQ_DI M3 scl(double s, const M3& a) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) r.m[i][j] = s * a.m[i][j];
  return r;
}

LQ_DI long long nidx(const Geom& g, const int x[4]) {
  return (((long long)x[0] * g.L[1] + x[1]) * g.L[2] + x[2]) * g.L[3] + x[3];
}
LQ_DI void ncoords(const Geom& g, long long i, int x[4]) {
  x[3] = (int)(i % g.L[3]);
  i /= g.L[3];
  x[2] = (int)(i % g.L[2]);
  i /= g.L[2];
  x[1] = (int)(i % g.L[1]);
  x[0] = (int)(i / g.L[1]);
}
LQ_DI void shifted(const Geom& g, const int x[4], int mu, int d, int y[4]) {
#pragma unroll
  for (int k = 0; k < 4; k++) {  // (no indexing by mu: the coordinates stay in registers)
    int v = x[k] + (k == mu ? d : 0);
    if (v < 0) v += g.L[k];
    if (v >= g.L[k]) v -= g.L[k];
    y[k] = v;
  }
}

// U_mu(x) from the even-odd FP64 link store; zero for the absent open-BC link.
LQ_DI M3 link(const Geom& g, const FieldPtrs& f, const int x[4], int mu) {
  if (g.bc_t == 0 && mu == 0 && x[0] == g.L[0] - 1) return zero3();
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  return LinkIO<64>::load(f, p, mu, g.Vh, nidx(g, x) >> 1);
}

// plane index of the unordered pair {mu, nu}: (0,1)(0,2)(0,3)(1,2)(1,3)(2,3)
LQ_DI int plane_of(int mu, int nu) {
  int a = mu < nu ? mu : nu, b = mu < nu ? nu : mu;
  return a == 0 ? b - 1 : (a == 1 ? b + 1 : 5);
}

// Slices whose links can have a force: one more than the slab on both sides, held in slots
// 0 .. nsl-1 (the whole lattice in natural order when that covers it).
struct ForceSlices {
  int first, nsl, T;  // slot 0 is slice `first`; slot k slice (first + k) mod T
  int base, held;     // the arrays hold the `held` slots from `base` on (mod T)
  int out0, out1;     // the links of slots out0 .. out1 - 1 are computed
  long long s3;
};
LQ_DI int slot_of(const ForceSlices& fs, int t) {
  const int k = t - fs.first;
  return k < 0 ? k + fs.T : (k >= fs.T ? k - fs.T : k);
}
// Index of site x in the arrays over the slots, -1 outside them.
LQ_DI long long sidx(const Geom& g, const ForceSlices& fs, const int x[4]) {
  int k = slot_of(fs, x[0]);
  if (k >= fs.nsl) return -1;
  k -= fs.base;
  if (k < 0) k += fs.T;
  if (k >= fs.held) return -1;
  return k * fs.s3 + ((long long)x[1] * g.L[2] + x[2]) * g.L[3] + x[3];
}

// K_{mu nu}(z) (ordered pair; K_{nu mu} = -K_{mu nu}), stored for mu < nu.
LQ_DI M3 load_K(const Geom& g, const ForceSlices& fs, const double2* K, const int z[4], int mu, int nu) {
  const long long i = sidx(g, fs, z);
  if (i < 0) return zero3();
  const double2* b = K + (i * 6 + plane_of(mu, nu)) * 9;
  M3 r;
  const double s = mu < nu ? 1.0 : -1.0;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    double2 v = b[k];
    r.m[k / 3][k % 3] = {s * v.x, s * v.y};
  }
  return r;
}
// B_{s,rho}(z), rho != s, stored [site][s][rho without s]; zero outside the slots.
LQ_DI M3 load_B(const Geom& g, const ForceSlices& fs, const double2* B, const int z[4], int s, int rho) {
  const long long i = sidx(g, fs, z);
  if (i < 0) return zero3();
  const double2* b = B + (i * 12 + s * 3 + (rho > s ? rho - 1 : rho)) * 9;
  M3 r;
#pragma unroll
  for (int k = 0; k < 9; k++) {
    double2 v = b[k];
    r.m[k / 3][k % 3] = {v.x, v.y};
  }
  return r;
}

// Per site of the slab: K_mn = c_sw (i/4)(Xi + Xi^dag) for the 6 planes.
// sigma in the chiral basis: sigma_0k = diag(s_k, -s_k), sigma_jk = -eps_jkl diag(s_l, s_l).
__global__ void k_force_K(Geom g, ForceSlices fs, int t0, int t1, double csw, const double2* X, const double2* Y,
                          double2* K) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= fs.held * fs.s3) return;
  const int t = (int)((fs.first + fs.base + q / fs.s3) % fs.T);
  const long long i = t * fs.s3 + q % fs.s3;
  double2* out = K + q * 54;
  if (t < t0 || t > t1) {
    for (int k = 0; k < 54; k++) out[k] = make_double2(0.0, 0.0);
    return;
  }
  cd x[12], y[12];
#pragma unroll
  for (int k = 0; k < 12; k++) {
    double2 a = X[i * 12 + k], b = Y[i * 12 + k];
    x[k] = {a.x, a.y};
    y[k] = {b.x, b.y};
  }
  // O[chi][s][t][b][a] = X[2chi+t][b] conj(Y[2chi+s][a]), combined per Pauli matrix
  const int pl_l[6] = {1, 2, 3, 3, 2, 1};
  const double pl_up[6] = {1, 1, 1, -1, 1, -1};
  const double pl_dn[6] = {-1, -1, -1, -1, 1, -1};
#pragma unroll
  for (int pl = 0; pl < 6; pl++) {  // unrolled: each plane keeps the two products it needs
    M3 xi = zero3();
#pragma unroll
    for (int chi = 0; chi < 2; chi++) {
      const double sg = chi == 0 ? pl_up[pl] : pl_dn[pl];
      const int o = 6 * chi;
#pragma unroll
      for (int b = 0; b < 3; b++)
#pragma unroll
        for (int a = 0; a < 3; a++) {
          // O_st = X[t][b] conj(Y[s][a]) within the chirality block
          cd O00 = cmulc(y[o + 0 + a], x[o + 0 + b]);
          cd O01 = cmulc(y[o + 0 + a], x[o + 3 + b]);
          cd O10 = cmulc(y[o + 3 + a], x[o + 0 + b]);
          cd O11 = cmulc(y[o + 3 + a], x[o + 3 + b]);
          cd v;
          if (pl_l[pl] == 1) v = O01 + O10;            // sigma_1 = [[0,1],[1,0]]
          else if (pl_l[pl] == 2) v = ti(O10 - O01);   // sigma_2 = [[0,-i],[i,0]]
          else v = O00 - O11;                          // sigma_3 = diag(1,-1)
          xi.m[b][a] = xi.m[b][a] + sg * v;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = 0; b < 3; b++) {
        cd h = xi.m[a][b] + conj(xi.m[b][a]);
        cd kk = (0.25 * csw) * ti(h);
        out[pl * 9 + a * 3 + b] = make_double2(kk.re, kk.im);
      }
  }
}

LQ_DI cd tr_mul(const M3& a, const M3& b) {
  cd t = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int k = 0; k < 3; k++) t = t + a.m[i][k] * b.m[k][i];
  return t;
}

// F^a = Re tr[i T_a Z] = -Im tr[T_a Z] = -Im tr[lambda_a Z] / 2
LQ_DI void project_force(const M3& Z, double* out8) {
  const M3& z = Z;
  // tr[lambda_a Z] for the 8 Gell-Mann matrices
  cd t[8];
  t[0] = z.m[1][0] + z.m[0][1];
  t[1] = ti(z.m[1][0]) - ti(z.m[0][1]);  // lambda_2 = [[0,-i],[i,0]]: tr = -i Z10 + i Z01 ... see below
  // lambda_2[0][1] = -i, [1][0] = i  ->  tr(l Z) = l01 Z10 + l10 Z01 = -i Z10 + i Z01
  t[1] = ti(z.m[0][1]) - ti(z.m[1][0]);
  t[2] = z.m[0][0] - z.m[1][1];
  t[3] = z.m[2][0] + z.m[0][2];
  t[4] = ti(z.m[0][2]) - ti(z.m[2][0]);
  t[5] = z.m[2][1] + z.m[1][2];
  t[6] = ti(z.m[1][2]) - ti(z.m[2][1]);
  const double s3 = 0.57735026918962576451;
  t[7] = s3 * (z.m[0][0] + z.m[1][1]) - (2.0 * s3) * z.m[2][2];
#pragma unroll
  for (int a = 0; a < 8; a++) out8[a] = -0.5 * t[a].im;
}

// r (+)= sign a b, a b^dag, a^dag b with fused multiply-adds.
LQ_DI M3 mul_nh(const M3& a, const M3& b) {  // a b^dag
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      cd t = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 3; k++) fma_cc(t, b.m[j][k], a.m[i][k]);
      r.m[i][j] = t;
    }
  return r;
}
LQ_DI M3 mul_hn(const M3& a, const M3& b) {  // a^dag b
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      cd t = {0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 3; k++) fma_cc(t, a.m[k][i], b.m[k][j]);
      r.m[i][j] = t;
    }
  return r;
}
LQ_DI M3 sub(const M3& a, const M3& b) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) r.m[i][j] = a.m[i][j] - b.m[i][j];
  return r;
}

// B of the twelve (s, rho) of a site: one thread per (site, s), its three rho.
__global__ void __launch_bounds__(128) k_force_B(Geom g, ForceSlices fs, const FieldPtrs* fields, int field,
                                                 const double2* K, double2* B) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= 4 * fs.held * fs.s3) return;
  const long long q = gid >> 2;
  const int s = (int)(gid & 3);
  int x[4], y[4];
  ncoords(g, q % fs.s3, x);
  x[0] = (int)((fs.first + fs.base + q / fs.s3) % fs.T);
  shifted(g, x, s, 1, y);
  const M3 u = link(g, fields[field], x, s);
#pragma unroll 1
  for (int k = 0; k < 3; k++) {
    const int rho = k < s ? k : k + 1;
    const M3 r = add(mul(load_K(g, fs, K, x, rho, s), u), mul(u, load_K(g, fs, K, y, rho, s)));
    double2* out = B + (gid * 3 + k) * 9;
#pragma unroll
    for (int e = 0; e < 9; e++) out[e] = make_double2(r.m[e / 3][e % 3].re, r.m[e / 3][e % 3].im);
  }
}

// Half spinor of (1 + S g_rho) psi, rho at run time.
template <int S>
LQ_DI void half_of(int rho, const double2* psi, cd h[6]) {
  cd p[12];
#pragma unroll
  for (int k = 0; k < 12; k++) {
    const double2 v = psi[k];
    p[k] = {v.x, v.y};
  }
  switch (rho) {
    case 0: project<0, S>(p, h); break;
    case 1: project<1, S>(p, h); break;
    case 2: project<2, S>(p, h); break;
    default: project<3, S>(p, h); break;
  }
}
// w[b][a] += sum_s u_s[b] conj(v_s[a]) over the two spins of a half spinor.
LQ_DI void outer_add(M3& w, double f, const cd u[6], const cd v[6]) {
#pragma unroll
  for (int s = 0; s < 2; s++)
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const cd fu = f * u[3 * s + b];
#pragma unroll
      for (int a = 0; a < 3; a++) fma_cc(w.m[b][a], v[3 * s + a], fu);
    }
}

// One thread per link (x, rho), natural order; links outside the slots have no force.
__global__ void __launch_bounds__(128) k_force_link(Geom g, ForceSlices fs, const FieldPtrs* fields, int field, int t0,
                                                    int t1, double csw, const double2* X, const double2* Y,
                                                    const double2* B, double* F) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= 8 * g.Vh) return;
  const long long i = gid >> 2;
  const int rho = (int)(gid & 3);
  double* out = F + gid * 8;
  int x[4];
  ncoords(g, i, x);
  const FieldPtrs f = fields[field];
  const int slot = slot_of(fs, x[0]);
  if (slot < fs.nsl ? slot < fs.out0 || slot >= fs.out1 : fs.out0 > 0) return;  // another launch's
  if (slot >= fs.nsl || (g.bc_t == 0 && rho == 0 && x[0] == g.L[0] - 1)) {
    for (int a = 0; a < 8; a++) out[a] = 0.0;
    return;
  }
  M3 Z = zero3();
  int xr[4];
  shifted(g, x, rho, 1, xr);
  // ---- clover part: -(1/2) sum_s (M_a - (M_c l)^dag), without the factor
  if (csw != 0.0) {
#pragma unroll 1
    for (int k = 0; k < 3; k++) {
      const int s = k < rho ? k : k + 1;
      int z[4];
      {  // plaquette above: corners x, x+rho, x+rho+s, x+s
        shifted(g, x, s, 1, z);
        const M3 c = link(g, f, z, rho);                      // U_rho(x+s)
        const M3 p = mul(link(g, f, x, s), c);                // (c d)^dag
        Z = add(Z, mul_nh(load_B(g, fs, B, xr, s, rho), p));  // B(x+rho) c d
        const M3 bc = mul_nh(link(g, f, xr, s), c);
        Z = sub(Z, mul_nh(bc, load_B(g, fs, B, x, s, rho)));  // b c B(x)^dag
      }
      {  // plaquette below: w = x - s, corners w, w+rho, x+rho, x
        int w[4];
        shifted(g, x, s, -1, w);
        shifted(g, w, rho, 1, z);
        const M3 a = link(g, f, w, rho);
        const M3 ab = mul(a, link(g, f, z, s));
        Z = sub(Z, mul_hn(ab, load_B(g, fs, B, w, s, rho)));  // (a' b')^dag B(w)
        const M3 ab2 = mul(a, load_B(g, fs, B, z, s, rho));
        Z = add(Z, mul_hn(ab2, link(g, f, w, s)));            // B(w+rho)^dag a'^dag U_s(w)
      }
    }
    Z = scl(-0.5, Z);
  }
  // ---- hopping part: f (W1 + W2^dag)
  if (x[0] >= t0 && x[0] <= t1 && xr[0] >= t0 && xr[0] <= t1) {
    // a time link that wraps (periodic / antiperiodic only) carries the boundary sign
    const double sg = rho == 0 && x[0] == g.L[0] - 1 && g.bc_t == 2 ? -1.0 : 1.0;
    const long long iy = nidx(g, xr);
    cd u[6], v[6];
    half_of<-1>(rho, X + iy * 12, u);
    half_of<-1>(rho, Y + i * 12, v);
    outer_add(Z, sg, u, v);
    half_of<+1>(rho, Y + iy * 12, u);
    half_of<+1>(rho, X + i * 12, v);
    outer_add(Z, sg, u, v);
  }
  project_force(mul(link(g, f, x, rho), Z), out);
}

}  // namespace lq

int lq_force(const lqcd_lattice* L, int field, const lqcd_slab& dom, const double2* X, const double2* Y, double* F,
             cudaStream_t st) {
  lq::ForceSlices fs;
  fs.T = L->dims[0];
  fs.s3 = L->S3;
  const int want = dom.t1 - dom.t0 + 3;
  fs.nsl = want >= fs.T ? fs.T : want;
  fs.first = want >= fs.T ? 0 : (dom.t0 + fs.T - 1) % fs.T;
  // K and B take three times the K of all slices that the plain form held (54 complex numbers a site).  Where that is
  // more than 2 GB, only as many slices at a time as keep within it: the links of a slice need B of the slices
  // on either side, and that K of one more.
  constexpr int WORDS = 54 + 108;
  const double room = std::max(54.0 * 16 * L->V, 2e9);
  int run = fs.nsl;  // slots of links at a time
  if (L->csw != 0.0 && (double)WORDS * 16 * fs.nsl * fs.s3 > room)
    run = std::max(1, (int)(room / ((double)WORDS * 16 * fs.s3)) - 3);
  if (run + 3 >= fs.nsl) run = fs.nsl;
  double2 *K = nullptr, *B = nullptr;
  const long long room_sites = (run < fs.nsl ? run + 3 : fs.nsl) * fs.s3;
  if (L->csw != 0.0) {
    if (cudaMallocAsync((void**)&K, sizeof(double2) * WORDS * (size_t)room_sites, st) != cudaSuccess) {
      cudaGetLastError();
      lq_set_error("link_force: allocation failed");
      return LQCD_ENOMEM;
    }
    B = K + 54 * room_sites;
  }
  for (fs.out0 = 0; fs.out0 < fs.nsl; fs.out0 += run) {
    fs.out1 = std::min(fs.out0 + run, fs.nsl);
    fs.base = run < fs.nsl ? (fs.out0 + fs.T - 1) % fs.T : 0;
    fs.held = run < fs.nsl ? run + 3 : fs.nsl;
    if (L->csw != 0.0) {
      const long long sites = fs.held * fs.s3;
      lq::k_force_K<<<(unsigned)((sites + 127) / 128), 128, 0, st>>>(L->g, fs, dom.t0, dom.t1, L->csw, X, Y, K);
      lq_count_launch();
      lq::k_force_B<<<(unsigned)((4 * sites + 127) / 128), 128, 0, st>>>(L->g, fs, L->d_fields, field, K, B);
      lq_count_launch();
    }
    lq::k_force_link<<<(unsigned)((4 * L->V + 127) / 128), 128, 0, st>>>(L->g, fs, L->d_fields, field, dom.t0, dom.t1,
                                                                          L->csw, X, Y, B, F);
    lq_count_launch();
  }
  if (K) cudaFreeAsync(K, st);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    lq_set_error(std::string("link_force: ") + cudaGetErrorString(e));
    return LQCD_ECUDA;
  }
  return 0;
}
