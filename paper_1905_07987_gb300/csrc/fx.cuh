// 64-bit block fixed point on the integer pipe.
//
// GB300 issues 2 FP64 lane operations per clock and SM but 64 lane operations of the 32 x 32 + 64
// bit integer multiply-add (measured: 1.7 DFMA against 63 mad.wide.s32).  A dot product with a
// fixed table therefore costs a tenth as an integer one: the inputs of a block share a power-of-two
// scale, X = x 2^(1082 - E) with |x| < 2^(E - 1022), so |X| < 2^60; an input and a table entry
// are split into a signed high word and a signed low word, X = xh 2^32 + xl, and
//   sum X T = (sum xh th) 2^64 + (sum xh tl + xl th) 2^32 + ...
// takes three multiply-adds per term, exactly accumulated in 64 bits: with table rows of
// sum |T| < 2^61 (the host's scaling) and up to 9 terms no sum reaches 2^63.  What three leave out,
// xl tl, is up to a quarter of the last place of the high sum per term: 2^-59 of the largest
// possible result.  That is enough for the derivatives, whose sums the step size scales down; the
// products whose results go into the state take a fourth multiply-add and are off by one unit of
// X' = sum X T / 2^(64 - SH) < 2^(57 + SH).  A chain of FP64 FMAs rounds at 2^-53 of each partial
// sum.  Inputs within 2^-7 of the bound are converted exactly.
#pragma once
#include <cuda_runtime.h>
#include "ader_internal.h"

namespace ader {

// x 2^(1075 + SH - E) rounded towards zero, below 2^(53 + SH); `over` gets its sign bit set when
// |x| >= 2^(E - 1022) (also for infinities and NaN).  E >= 128, so subnormal x give 0.
template <int SH = 7>
__device__ __forceinline__ long long fx_in(double x, int E, int& over) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int s = E - (int)((hi >> 20) & 0x7ffu);
  over |= s;  // negative: too large
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  asm("shr.b64 %0, %1, %2;" : "=l"(m) : "l"(m << SH), "r"(s));  // shifts of 64 and more give 0
  const long long g = (long long)((int)hi >> 31);
  return ((long long)m ^ g) - g;
}

// r 2^k as a double (rounded to nearest); results below the normal range give 0.
__device__ __forceinline__ double fx_out(long long r, int k) {
  const unsigned long long g = (unsigned long long)(r >> 63);
  const unsigned long long a = ((unsigned long long)r ^ g) - g;
  const int lz = __clzll((long long)a);
  const unsigned long long nrm = a << (lz & 63);
  const int e = 1085 + k - lz;  // biased exponent - 1: the mantissa's leading one adds to it
  const unsigned long long b =
      ((unsigned long long)(unsigned)e << 52) + (nrm >> 11) + ((nrm >> 10) & 1u);
  const bool z = a == 0 || e < 0;
  return __longlong_as_double(z ? 0ll : (long long)(b | (g & 0x8000000000000000ull)));
}

// To and from binary32 by 32-bit conversions (the 64-bit ones run at the FP64 pipe's rate): r within
// a few units of binary32's last place or 2^8, |x| < 2^62 within one.
__device__ __forceinline__ float fx_float(long long r) {
  return fmaf((float)(int)(r >> 32), 4294967296.0f, (float)(unsigned)r);
}
__device__ __forceinline__ long long fx_from_float(float x) {
  const float h = rintf(x * 0x1p-32f);
  return ((long long)(int)h << 32) + (long long)(int)fmaf(h, -4294967296.0f, x);
}

// The two words of X: X = h 2^32 + l.
__device__ __forceinline__ fx2 fx_split(long long X) {
  const unsigned l = (unsigned)X;
  return {(int)((unsigned)((unsigned long long)X >> 32) + (l >> 31)), (int)l};
}

// a b / 2^64 (the low words' product left out)
__device__ __forceinline__ long long fx_mul(fx2 a, fx2 b) {
  const long long c = (long long)a.h * b.l + ((long long)a.l * b.h + (1ll << 31));
  return (long long)a.h * b.h + (int)(c >> 32);
}

// Sum of products, sum X T / 2^(64 - SH).  LL: with the low words' products, to 2^-16 of the last place
// of the high sum, as products of their upper halves.
template <int SH, bool LL = true>
struct FxAcc {
  long long s1 = 0, s0 = 1ll << (31 - SH);
  __device__ __forceinline__ void mac(fx2 x, fx3 t) {
    s1 += (long long)x.h * t.h;
    s0 += (long long)x.h * t.l;
    s0 += (long long)x.l * t.h;
    if (LL) s0 += (long long)(x.l >> 16) * t.q;
  }
  __device__ __forceinline__ long long get() const {
    const long long t = s1 + (int)(s0 >> 32);
    return SH ? (long long)(((unsigned long long)t << SH) | ((unsigned)s0 >> (32 - SH))) : t;
  }
};

// The same for a table row T of n entries.
template <int n, int SH, bool LL = true>
__device__ __forceinline__ long long fx_dot(const fx2 (&X)[n], const fx3* T) {
  FxAcc<SH, LL> a;
#pragma unroll
  for (int m = 0; m < n; ++m) a.mac(X[m], T[m]);
  return a.get();
}

}  // namespace ader
