// pic_fixed64.cuh -- 64-bit fixed-point arithmetic of the FP64 push.
//
// The cubic shape factors, the gather (a 4x4x4 weighted sum per field
// component) and the Esirkepov deposit (products of shape-factor sums) of the
// FP64 push run as integer arithmetic: on this GPU the integer multiply-add
// pipe retires 32x32->64-bit products many times faster than the FP64 pipe
// retires FMAs, and a 64-bit integer add into shared memory is a native 32-bit
// atomic plus a carry, where a double add is a compare-and-swap loop.
//
// Formats:
// - a "value" x is an int64 in units of 2^-k for a scale k chosen per tile
//   (fields) or per tile and component (current), split centred:
//   x = hi 2^31 + lo with -2^30 <= lo < 2^30;
// - a "weight" W is a non-negative int64 below 2^62 holding w 2^62 for
//   0 <= w < 1 (shape factors, Esirkepov factors), split as
//   W = hi 2^31 + lo with 0 <= lo < 2^31.
//
// x W / 2^62 = xh Wh + (xh Wl + xl Wh) / 2^31 + xl Wl / 2^62: three 32x32->64
// multiply-adds into two accumulators (the two cross products share a scale).
// The last term is dropped; its xl is centred, so that it is below half a unit
// and has zero mean, and a sum of products of zeros is zero.  Range of the
// second accumulator: a gather sums 16 products with |x| < 2^58 and weights
// that sum to at most one, |sum xh Wl| < 16 x 2^27 x 2^31 = 2^62 and
// |sum xl Wh| <= 2^30 x 2^31; a deposit product has |x| <= 2^62, |xh Wl| < 2^62
// and |xl Wh| < 2^61; both stay within 2^63.
#pragma once

#include <cuda_runtime.h>

namespace pic {

struct S31 {
  int hi, lo;
};

// a b + c, one 32x32->64 multiply-add.  Spelt out: from the C expression the
// compiler widens operands that it knows to be non-negative and multiplies in
// 64 bits (16 instructions per acc31 instead of 3).
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// Centred split of a value; plain split of a weight (>= 0).
__device__ __forceinline__ S31 split31(long long x) {
  return {(int)((x + (1LL << 30)) >> 31), ((int)((unsigned)x << 1)) >> 1};
}
__device__ __forceinline__ S31 splitw(long long W) { return {(int)(W >> 31), (int)(W & 0x7FFFFFFFLL)}; }

struct Acc31 {
  long long H, M;
};
__device__ __forceinline__ Acc31 acc31_init() { return {0LL, 1LL << 30}; }  // rounds the shift
__device__ __forceinline__ void acc31(Acc31& a, S31 x, S31 w) {
  a.H = mad_wide(x.hi, w.hi, a.H);
  a.M = mad_wide(x.hi, w.lo, a.M);
  a.M = mad_wide(x.lo, w.hi, a.M);
}
__device__ __forceinline__ long long acc31_result(const Acc31& a) { return a.H + (a.M >> 31); }

// x W / 2^62 for one product.
__device__ __forceinline__ long long mul62(S31 x, S31 w) {
  Acc31 a = acc31_init();
  acc31(a, x, w);
  return acc31_result(a);
}

// round(v 2^k) for |v| 2^k < 2^62, from the bit pattern of v (integer
// instructions only; zero and subnormal v give 0).
__device__ __forceinline__ long long to_fixed(double v, int k) {
  const long long b = __double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7FF);
  const long long m = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
  const int sh = e - 1075 + k;  // |v| 2^k = m 2^sh, sh <= 9 by the caller's bound
  const int l = max(sh, 0), r = min(max(-sh, 0), 62);
  long long X = ((m << l) + ((1LL << r) >> 1)) >> r;
  X = e == 0 ? 0 : X;
  return b < 0 ? -X : X;
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

// Cubic B-spline weights at 2^62 of the nodes c-1, c, c+1, c+2 for an offset
// T / 2^62 in [0, 1): w3 = t^3/6, w1 = 2/3 - t^2 + t^3/2, w2 = 1/6 + (t + t^2 -
// t^3)/2 (= 2/3 - s^2 + s^3/2 with s = 1 - t), w0 = 1 - w1 - w2 - w3 (= s^3/6):
// within a few units of 2^-62, and they sum to one.
__device__ __forceinline__ void spline62(long long T, long long (&w)[4]) {
  constexpr long long kOne = 1LL << 62, kTwo3 = 3074457345618258603LL, kSixth = 768614336404564651LL;
  const S31 t = splitw(T);
  const long long t2 = mad_wide(t.hi, t.hi, mad_wide(t.hi, t.lo, 1LL << 29) >> 30);
  const long long t3 = mul62(splitw(t2), t);
  w[3] = mul62(splitw(t3), splitw(kSixth));
  w[1] = kTwo3 - t2 + (t3 >> 1);
  w[2] = kSixth + ((T + t2 - t3) >> 1);
  w[0] = max(kOne - w[1] - w[2] - w[3], 0LL);  // clamps a rounding below zero
}
__device__ __forceinline__ void spline62(long long T, S31 (&w)[4]) {
  long long v[4];
  spline62(T, v);
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = splitw(v[k]);
}

// S / 2 + D / 3 = ((3 S + 2 D) / 2) / 3 for weights S and S + D (the sum of up
// to 3 x 2^62 is formed unsigned).
__device__ __forceinline__ long long third62(long long S, long long D) {
  constexpr long long kThird = 1537228672809129301LL;
  const unsigned long long v = 3ull * (unsigned long long)S + 2ull * (unsigned long long)D;
  return mul62(splitw((long long)(v >> 1)), splitw(kThird));
}

// Sum over 4x4x4 nodes of a staged component (split words), weights wde over
// the first two axes and wf over the last.
__device__ __forceinline__ long long gather64(const int2* __restrict__ s, int sd, int se, const S31 (&wde)[4][4],
                                              const S31 (&wf)[4]) {
  Acc31 sum = acc31_init();
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    Acc31 a = acc31_init();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int2 v = s[i * sd + j * se + c];
        acc31(a, {v.y, v.x}, wde[i][j]);
      }
    acc31(sum, split31(acc31_result(a)), wf[c]);
  }
  return acc31_result(sum);
}

__device__ __forceinline__ unsigned atom_add_u32_shared(unsigned* a, unsigned v) {
  unsigned old;
  asm volatile("atom.shared.add.u32 %0, [%1], %2;"
               : "=r"(old)
               : "r"((unsigned)__cvta_generic_to_shared(a)), "r"(v)
               : "memory");
  return old;
}

__device__ __forceinline__ void red_add_u32_shared(unsigned* a, unsigned v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(a)), "r"(v) : "memory");
}

}  // namespace pic
