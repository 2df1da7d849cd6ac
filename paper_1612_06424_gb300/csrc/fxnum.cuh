// Fixed-point numbers of the FP64-accurate stencil (fx.cuh): conversions between FP64 and 57-bit
// integers with an exponent, and the 29-bit limbs that they are stored in.
#pragma once

#include <cuda_runtime.h>

#ifndef LQ_DI
#define LQ_DI __device__ __forceinline__
#endif

namespace lq {

constexpr int FX_BIAS = 1079;  // value of a spinor component: q 2^(E - FX_BIAS)
constexpr int FX_NAN = 1 << 14;  // exponent of a spinor with a non-finite component

// acc += a b (32 x 32 + 64 bits) as one instruction: written in C++ it became a product and a 64-bit
// addition, which more than doubled the instructions of the kernels built on it
LQ_DI void mad_wide(long long& acc, int a, int b) { asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b)); }

LQ_DI int fx_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// q with x = q 2^(E - FX_BIAS), rounded; E at most 4 below x's exponent.
LQ_DI long long fx_of(double x, int E) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)(hi & 0xfffff) | (ex ? 0x100000u : 0u);
  const long long m = ((long long)mh << 32) | (unsigned)__double2loint(x);
  const int sh = E - (ex ? ex : 1) - 4;  // q = m 2^-sh
  long long q;
  if (sh <= 0)
    q = m << -sh;
  else
    q = sh < 60 ? (m + (1ll << (sh - 1))) >> sh : 0ll;
  return hi < 0 ? -q : q;
}
LQ_DI void fx_split(long long q, int& q1, int& q0) {
  q0 = (int)((unsigned)q << 3) >> 3;
  q1 = (int)((q - q0) >> 29);
}
LQ_DI long long fx_join(int q1, int q0) { return ((long long)q1 << 29) + q0; }

// v 2^e rounded to nearest.  DEN: also below the normal range, else zero there.
template <bool DEN = true>
LQ_DI double fx_to_double(long long v, int e) {
  if (v == 0) return 0.0;
  unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int c = __clzll((long long)m);
  m <<= c;
  const int ex = 1086 - c + e;  // biased exponent of the leading bit
  long long bits = ((long long)(ex - 1) << 52) + (long long)(m >> 11) + (long long)((m >> 10) & 1);
  if (ex <= 0) {  // below the normal range: m 2^(ex - 12) units of the last place
    const int s = 12 - ex;
    bits = !DEN ? 0 : s < 64 ? (long long)(m >> s) + (long long)((m >> (s - 1)) & 1) : s == 64 ? (long long)(m >> 63) : 0;
  }
  if (ex >= 2047) bits = 0x7ff0000000000000ll;
  return __longlong_as_double(v < 0 ? bits | (long long)0x8000000000000000ull : bits);
}

// (hh 2^L + cr) 2^(e - L) rounded once: the two partial sums of a product in limbs of L bits, cr joined at the
// precision that hh leaves free
template <int L, bool DEN>
LQ_DI double fx_sum(long long hh, long long cr, int e) {
  const int k = min(max(__clzll(hh < 0 ? ~hh : hh) - 2, 0), L);
  const int s = L - k;
  return fx_to_double<DEN>((hh << k) + (s ? (cr + (1ll << (s - 1))) >> s : cr), e - k);
}

// exponent of the links' fixed scale: value q 2^-58
constexpr int FX_LINK_E = FX_BIAS - 58;

}  // namespace lq
