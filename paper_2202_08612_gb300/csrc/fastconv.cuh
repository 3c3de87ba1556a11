// The hi/lo bfloat16 split of the split-precision path, kept off the FP64 pipe
// (on GB300 it retires about two FP64 operations per clock and SM, so an FP64
// subtraction or a double -> bf16 rounding per element bounds an otherwise
// memory-bound pass): one FP64 -> FP32 conversion, then FP32 work only.
#pragma once
#include <cuda_bf16.h>

namespace mlcc3 {

// binary64 -> binary32, round to nearest even, on the integer pipe where the result
// is a normal number (a conversion there is an FP64 operation, two per clock and SM).
__device__ __forceinline__ float narrow_f64(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if (((hi >> 20) & 0x7ff) - 897u < 253u) {
    const unsigned long long m = (((unsigned long long)hi << 32) | lo) + 0x0fffffffu + ((lo >> 29) & 1u);
    return __uint_as_float((((unsigned)(m >> 29) - 0xC0000000u) & 0x7fffffffu) | (hi & 0x80000000u));
  }
  if (((hi << 1) | lo) == 0) return __uint_as_float(hi);  // zeros, as in the padding of a tile
  return __double2float_rn(x);
}

// binary32 -> binary64 (exact) on the integer pipe, for numbers that are not subnormal.
__device__ __forceinline__ double widen_normal(float f) {
  const unsigned int b = __float_as_uint(f);
  const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
  const unsigned int e = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
  if (e == 0) return __longlong_as_double((long long)sign);
  const unsigned long long ex = e == 255 ? 0x7FFull : (unsigned long long)(e + 896);
  return __longlong_as_double((long long)(sign | (ex << 52) | ((unsigned long long)m << 29)));
}

// The same for any number: subnormals by the hardware conversion.
__device__ __forceinline__ double widen_f32(float f) {
  return (__float_as_uint(f) << 1) - 1u < 0xFFFFFFu ? (double)f : widen_normal(f);
}

// sum[i] += f[i], one look for subnormals for all of them.
template <int N>
__device__ __forceinline__ void widen_add(double (&sum)[N], const float (&f)[N]) {
  unsigned least = ~0u;
#pragma unroll
  for (int i = 0; i < N; ++i) least = min(least, (__float_as_uint(f[i]) << 1) - 1u);
  if (least < 0xFFFFFFu) {
#pragma unroll
    for (int i = 0; i < N; ++i) sum[i] += (double)f[i];
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) sum[i] += widen_normal(f[i]);
  }
}
template <int N>
__device__ __forceinline__ void widen_add(double (&sum)[N], const double (&f)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) sum[i] += f[i];
}

// x ~ hi + lo with hi = bf16(f), lo = bf16(f - hi), f = binary32(x); f - hi is
// exact in binary32 (it keeps the 16 low bits of f's significand).
__device__ __forceinline__ void split_hi_lo(double x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
  const float f = __double2float_rn(x);
  hi = __float2bfloat16_rn(f);
  lo = __float2bfloat16_rn(f - __bfloat162float(hi));
}

// The same split of a binary32 value (no conversion from binary64).
__device__ __forceinline__ void split_hi_lo(float f, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
  hi = __float2bfloat16_rn(f);
  lo = __float2bfloat16_rn(f - __bfloat162float(hi));
}

// x scaled by +1 (mode 0), -1 (mode 1, a sign flip of the bit pattern) or s.
__device__ __forceinline__ double scaled(double x, int mode, double s) {
  if (mode == 0) return x;
  if (mode == 1) return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
  return s * x;
}

__device__ __forceinline__ float scaled(float x, int mode, double s) {
  if (mode == 0) return x;
  if (mode == 1) return -x;
  return (float)s * x;
}

}  // namespace mlcc3
