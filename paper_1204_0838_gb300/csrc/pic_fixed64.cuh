// pic_fixed64.cuh -- 64-bit fixed-point arithmetic of the FP64 push.
//
// The cubic shape factors, the gather (a 4x4x4 weighted sum per field
// component) and the Esirkepov deposit (products of shape-factor sums) of the
// FP64 push run as integer arithmetic: on this GPU the integer multiply-add
// pipe retires 32x32->64-bit products many times faster than the FP64 pipe
// retires FMAs, and integer adds into shared memory are native, where a double
// add is a compare-and-swap loop.
//
// A number x is an int64 in units of 2^-k, split centred at 32 bits:
// x = hi 2^32 + lo with -2^31 <= lo < 2^31.  The product of two,
//   x y / 2^64 = xh yh + (xh yl + xl yh) / 2^32 + xl yl / 2^64,
// takes three 32x32->64 multiply-adds into two accumulators; the cross
// products' sum M is added through its high word, so that a product needs no
// 64-bit shifts.  The last term is dropped: it
// is below 1/4 unit and has zero mean, so that sums of thousands of products
// add up no drift, and a sum of products of zeros is zero.
//
// Scales and the range of M (|M| + 2^31 < 2^63):
// - gather: fields |x| < 2^60 at 2^sF, weights at 2^63 (at most 2/3, products
//   of two at most 4/9): sums of 8 have |sum xh wl| <= 8 x 2^28 x 2^31 = 2^62, and
//   their high words go to the first accumulator before more is added; sums of
//   16 have |sum xl wh| <= 2^31 x (2^31 + 16), since the weights sum to one;
// - deposit factors: S and D = S1 - S of one axis at 2^62, |S| + |D| <= 6/5,
//   times factors at 2^63 that are at most 2/3 and 1/3:
//   |M| <= 2^62 (3/5 + 2/3 + 1/3);
// - current: |P| < 2^63 times A < 1/2 at 2^63: |M| <= 2^62 (1 + 1/2).
#pragma once

#include <cuda_runtime.h>

namespace pic {

struct S32 {
  int hi, lo;
};

// a b + c, one 32x32->64 multiply-add: the pair of a low multiply-add with carry
// and a high one is one instruction.  (mad.wide in inline assembly becomes a
// multiply and an add; the C expression is reassociated and, where the compiler
// knows an operand to be non-negative, widened to 64-bit multiplies.)
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("{ .reg .u32 l, h, m, n; mov.b64 {l, h}, %3; mad.lo.cc.s32 m, %1, %2, l; madc.hi.s32 n, %1, %2, h;"
      " mov.b64 %0, {m, n}; }"
      : "=l"(d)
      : "r"(a), "r"(b), "l"(c));
  return d;
}

__device__ __forceinline__ S32 split32(long long x) {
  return {(int)((unsigned long long)(x + 0x80000000LL) >> 32), (int)x};
}

struct Acc32 {
  long long H, M;
};
__device__ __forceinline__ Acc32 acc32_init() { return {0LL, 1LL << 31}; }  // rounds the high word of M
__device__ __forceinline__ void acc32(Acc32& a, S32 x, S32 w) {
  a.H = mad_wide(x.hi, w.hi, a.H);
  a.M = mad_wide(x.hi, w.lo, a.M);
  a.M = mad_wide(x.lo, w.hi, a.M);
}
__device__ __forceinline__ long long acc32_result(const Acc32& a) { return a.H + (a.M >> 32); }
// Twice the result, with one more bit, for a sum that began at {0, kRound2}.
constexpr long long kRound2 = 1LL << 30;
__device__ __forceinline__ long long acc32_result2(const Acc32& a) { return 2 * a.H + (a.M >> 31); }

// x w / 2^64 for one product; floor64 without the rounding, for factors whose
// last unit does not add up.
__device__ __forceinline__ long long mul64(S32 x, S32 w) {
  Acc32 a = acc32_init();
  acc32(a, x, w);
  return acc32_result(a);
}
__device__ __forceinline__ long long floor64(S32 x, S32 w) {
  Acc32 a = {0LL, 0LL};
  acc32(a, x, w);
  return acc32_result(a);
}

// round(v 2^k) for |v| 2^k < 2^63, from the bit pattern of v (integer
// instructions only; zero and subnormal v give 0).
__device__ __forceinline__ long long to_fixed(double v, int k) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long m = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
  const int sh = e - 1075 + k;  // |v| 2^k = m 2^sh, sh <= 10 by the caller's bound
  const int l = max(sh, 0), r = min(max(-sh, 0), 62);
  long long X = ((m << l) + ((1LL << r) >> 1)) >> r;
  X = e == 0 ? 0 : X;
  return b < 0 ? -X : X;
}

// A staged field value v as round(v 2^k), k = 59 + 1023 - emax for the largest
// biased exponent emax of a tile or block (below 2047): |v| 2^k < 2^60.
constexpr int kFieldBits = 60;
constexpr int kFieldMinExp = 82;  // smallest biased exponent that sets a scale (k <= 1000)
__device__ __forceinline__ long long field_fixed(long long b, int emax) {
  const int e = (int)((b >> 52) & 0x7FF);
  const unsigned long long m = (unsigned long long)(b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000ull;
  unsigned long long X = (m << 8) >> min(emax - e, 63);  // one bit below the unit
  X = e == 0 ? 0ull : (X + 1) >> 1;
  const long long n = b >> 63;
  return ((long long)X ^ n) - n;
}

// o 2^63 for 0 <= o < 1 (what falls below 2^-63 is cut off).
__device__ __forceinline__ long long offset63(double o) {
  const long long b = __double_as_longlong(o);
  const int e = (int)(b >> 52);
  const unsigned long long m = (unsigned long long)(b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000ull;
  return (long long)((m << 10) >> min(1022 - e, 63));
}

// 2^k as a double, for -1022 <= k <= 1023.
__device__ __forceinline__ double exp2i(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }

// x 2^-k as a double, rounded to nearest, with integer instructions only (a
// conversion and a multiply run at the FP64 rate); the result must be normal.
__device__ __forceinline__ double fixed_to_double(long long x, int k) {
  const unsigned long long a = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // 53 bits, carry into the exponent
  long long b = ((long long)(1085 - lz - k) << 52) + (long long)r;
  b = x == 0 ? 0 : b;
  return __longlong_as_double(x < 0 ? b | (long long)0x8000000000000000ull : b);
}

__device__ __forceinline__ S32 third64() { return {0x55555555, 0x55555555}; }  // 1/3 at 2^64

// Cubic B-spline weights at 2^K (62 or 63) of the nodes c-1, c, c+1, c+2 for
// u = t - 1/2 = U / 2^63, t in [0, 1) the offset in the cell:
//   w0, w3 = (1/48 + u^2/4) -+ (u/8 + u^3/6), w1, w2 = (23/48 - u^2/4) -+ (5u/8 -
// u^3/2), the cubic's pieces in even and odd parts.  Within a few units, and
// they sum to one exactly.
template <int K>
__device__ __forceinline__ void spline_fixed(long long U, long long (&w)[4]) {
  constexpr long long kOne48 = K == 63 ? 192153584101141163LL : 96076792050570581LL;  // 2^K / 48
  constexpr long long k23_48 = (1LL << (K - 1)) - kOne48;
  constexpr int sh = 63 - K;
  const S32 u = split32(U);
  const long long q = floor64(u, u);                       // u^2 at 2^62
  const long long c = floor64(u, split32(q));              // u^3 at 2^61
  const long long c3 = floor64(split32(c), third64());     // u^3 / 3 at 2^61
  const long long e = q >> (sh + 1), u3 = U >> (3 + sh);   // u^2 / 4, u / 8 at 2^K
  const long long e0 = kOne48 + e, e1 = k23_48 - e;
  const long long o0 = u3 + (sh ? c3 : 2 * c3);
  const long long o1 = u3 + (U >> (1 + sh)) - (sh ? c : 2 * c);
  w[0] = e0 - o0;
  w[1] = e1 - o1;
  w[2] = e1 + o1;
  w[3] = e0 + o0;
}
__device__ __forceinline__ void spline63(long long U, S32 (&w)[4]) {
  long long v[4];
  spline_fixed<63>(U, v);
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = split32(v[k]);
}
constexpr long long kHalf63 = 1LL << 62;  // 1/2 at 2^63

// Sum over 4x4x4 nodes of a staged component (split words at 2^sF), weights wde
// over the first two axes and wf over the last, both at 2^63: at 2^sF.
__device__ __forceinline__ long long gather64(const int2* __restrict__ s, int sd, int se, const S32 (&wde)[4][4],
                                              const S32 (&wf)[4]) {
  Acc32 sum = {0LL, kRound2};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    // the two cross sums apart: three chains of multiply-adds instead of two
    long long H = 0, M = kRound2, N = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int2 v = s[i * sd + j * se + c];
        H = mad_wide(v.y, wde[i][j].hi, H);
        M = mad_wide(v.y, wde[i][j].lo, M);
        N = mad_wide(v.x, wde[i][j].hi, N);
      }
      if (i & 1) {  // M stays below 2^62 + 2^32 (see above)
        H += M >> 32;
        M = (long long)(unsigned)M;
      }
    }
    const Acc32 a = {H, M + N};
    acc32(sum, split32(acc32_result2(a)), wf[c]);
  }
  return acc32_result2(sum);
}

}  // namespace pic
