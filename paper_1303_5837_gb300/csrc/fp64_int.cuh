// fp64_int.cuh -- reciprocal and reciprocal square root of FP64 values in
// 64-bit fixed point.  On this part one FP64 warp instruction holds the FP64
// pipe of its SM sub-partition for 64 clocks and the library's reciprocal,
// division and square root take 375, 436 and 620 clocks of dependent ones; the
// panel kernels' column chains wait for them.  Both functions here take the
// hardware's single-precision approximation of the leading bits (relative
// error e below 2^-21) and one third-order Householder step in integers.
#pragma once
#include <cuda_runtime.h>

namespace cagb {

// Exponent fields for which the functions below hold; zeros, subnormals,
// infinities, NaN and values near the ends of the range are outside.
__device__ __forceinline__ bool int_range(double v) {
  const unsigned E = (unsigned)((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ffu;
  return E - 64u < 0x7ffu - 128u;
}

// 2^63 / m, m = |v| / 2^(E - 1023) in [1, 2): at most 16 units off (truncations
// of 1, 4 and 8 units, e^3 below 1).
__device__ __forceinline__ unsigned long long recip_q62(unsigned long long M) {
  float x;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(__uint_as_float(0x3f800000u | (unsigned)(M >> 29))));
  const unsigned long long m = (M | (1ull << 52)) << 11;                                  // m / 2 in Q64
  const unsigned long long x0 = (unsigned long long)(unsigned)(x * 2147483648.0f) << 32;  // 2 x in Q62
  const long long e = (long long)((1ull << 62) - __umul64hi(m, x0));
  const long long f = e + (__mul64hi(e, e) << 2);
  return x0 + (unsigned long long)(__mul64hi(f, (long long)(x0 >> 1)) << 3);
}

// 1 / v, relative error below 1.02 2^-53; v in int_range.
__device__ __forceinline__ double recip_near(double v) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((bits >> 52) & 0x7ff);
  const unsigned long long mant = (recip_q62(bits & ((1ull << 52) - 1)) + 512) >> 10;  // in [2^52, 2^53]
  return __longlong_as_double((long long)(((bits >> 63) << 63) | (((unsigned long long)(2044 - E) << 52) + mant)));
}

// The correctly rounded 1 / v, or 0 where the last ten bits of 2^63 / m lie
// within 24 of a tie (1 in 20) or v is outside int_range.
__device__ __forceinline__ double recip_exact_or_zero(double v) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((bits >> 52) & 0x7ff);
  const unsigned long long y = recip_q62(bits & ((1ull << 52) - 1));
  const bool sure = (unsigned)(E - 64) < 0x7ffu - 128u && (unsigned)((int)(y & 1023) - 512 + 24) > 48u;
  const unsigned long long mant = (y + 512) >> 10;
  return !sure ? 0.0
               : __longlong_as_double((long long)(((bits >> 63) << 63) | (((unsigned long long)(2044 - E) << 52) + mant)));
}

// 1 / sqrt(v), relative error below 1.05 2^-53; v > 0 in int_range.
__device__ __forceinline__ double rsqrt_near(double v) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int e0 = (int)(bits >> 52) - 1023, k = e0 >> 1, odd = e0 & 1;  // v = m 4^k, m in [1, 4)
  const unsigned long long M = bits & ((1ull << 52) - 1);
  float x;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(__uint_as_float(((127u + odd) << 23) | (unsigned)(M >> 29))));
  const unsigned long long m = (M | (1ull << 52)) << (10 + odd);                 // Q62
  const unsigned long long r0 = (unsigned long long)(unsigned)(fminf(x, 1.0f) * 2147483648.0f);  // Q31
  const long long e = (long long)((1ull << 60) - __umul64hi(m, r0 * r0));        // 1 - m r0^2, Q60
  const long long f = (e >> 1) + ((3 * (__mul64hi(e, e) << 4)) >> 3);            // e / 2 + 3 e^2 / 8
  const unsigned long long y = (r0 << 31) + (unsigned long long)(__mul64hi(f, (long long)(r0 << 31)) << 4);  // Q62
  return __longlong_as_double((long long)(((unsigned long long)(1021 - k) << 52) + ((y + 256) >> 9)));
}

}  // namespace cagb
