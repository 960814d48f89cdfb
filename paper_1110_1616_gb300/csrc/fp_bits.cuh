// Conversions between IEEE-754 binary32 and binary64 done with integer
// operations on the bit patterns, from the two formats' definitions (sign,
// biased exponent, fraction; binary32 bias 127, binary64 bias 1023).
//
// On this part the FP64 pipe runs at a small fraction of the FP32 rate and the
// hardware conversions to and from binary64 issue on it; these routines use
// the integer pipe.
//
// Flush-to-zero semantics, as the mixed path is compiled with FP32 denormals
// flushed: a binary32 subnormal input converts to a signed zero, and a
// binary64 value below the smallest binary32 normal, 2^-126, converts to a
// signed zero. Otherwise both are exact IEEE
// conversions: widening is exact, narrowing rounds to nearest, ties to even,
// overflows to infinity, and keeps infinities and NaNs (NaNs made quiet).
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace amrdev {

__host__ __device__ __forceinline__ uint32_t f32_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return u;
#endif
}
__host__ __device__ __forceinline__ float f32_from(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, 4);
  return f;
#endif
}
__host__ __device__ __forceinline__ double f64_from(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double d;
  std::memcpy(&d, &b, 8);
  return d;
#endif
}
__host__ __device__ __forceinline__ void f64_split(double d, uint32_t& hi, uint32_t& lo) {
#ifdef __CUDA_ARCH__
  hi = (uint32_t)__double2hiint(d);
  lo = (uint32_t)__double2loint(d);
#else
  uint64_t b;
  std::memcpy(&b, &d, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
#endif
}

// binary32 -> binary64: the 8-bit exponent re-biased by 1023 - 127 = 896
// (255, infinity / NaN, maps to 2047), the 23 fraction bits placed at the top
// of the 52.
__host__ __device__ __forceinline__ double widen_bits(float f) {
  const uint32_t u = f32_bits(f);
  const uint32_t s = u & 0x80000000u;
  const uint32_t e = (u >> 23) & 0xffu;
  const uint32_t rebias = e == 255u ? 0x70000000u : 0x38000000u;  // 1792 or 896, at bit 20
  const uint32_t hi = e == 0u ? s : (s | (((u & 0x7fffffffu) >> 3) + rebias));
  const uint32_t lo = e == 0u ? 0u : (u << 29);
  return f64_from(hi, lo);
}

// binary64 -> binary32, round to nearest even: the 52-bit fraction cut to its
// top 23 bits, the 29 dropped bits deciding the rounding; a carry out of the
// fraction increments the exponent (and reaches infinity from the largest
// finite value), as the rounding definition requires.
__host__ __device__ __forceinline__ float narrow_bits(double d) {
  uint32_t hi, lo;
  f64_split(d, hi, lo);
  const uint32_t s = hi & 0x80000000u;
  const int E = (int)((hi >> 20) & 0x7ffu);
  if (E == 0x7ff) {
    const bool nan = ((hi & 0xfffffu) | lo) != 0u;
    return f32_from(s | 0x7f800000u | (nan ? 0x400000u | ((hi & 0xfffffu) << 3) | (lo >> 29) : 0u));
  }
  const int e = E - 896;
  if (e >= 255) return f32_from(s | 0x7f800000u);
  if (e <= 0) return f32_from(s);  // below the smallest binary32 normal: flushed
  const uint32_t m = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t rest = lo & 0x1fffffffu;
  uint32_t r = ((uint32_t)e << 23) | m;
  if (rest > 0x10000000u || (rest == 0x10000000u && (r & 1u))) r += 1u;
  return f32_from(s | r);
}

// ---------------------------------------------------------------- FP64 order on the integer pipe
// Comparisons, sign tests and the minmod selection of binary64 values from
// their bit patterns, with IEEE results for every operand (signed zeros equal,
// every comparison with a NaN false). An FP64 compare occupies the FP64 pipe
// (2 lanes per SM here) for as long as a multiply; these take a handful of
// integer instructions on the otherwise idle ALU pipe.
constexpr uint64_t F64_SIGN = 0x8000000000000000ull, F64_INF = 0x7ff0000000000000ull;

__host__ __device__ __forceinline__ uint64_t f64_bits(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t b;
  std::memcpy(&b, &d, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double f64_of(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  std::memcpy(&d, &b, 8);
  return d;
#endif
}
// x > 0: a positive pattern from 1 (the smallest subnormal) to infinity
__host__ __device__ __forceinline__ bool gt_zero(double x) { return f64_bits(x) - 1ull < F64_INF; }
__host__ __device__ __forceinline__ bool lt_zero(double x) { return (f64_bits(x) ^ F64_SIGN) - 1ull < F64_INF; }
__host__ __device__ __forceinline__ bool gt_zero(float x) { return x > 0.0f; }
__host__ __device__ __forceinline__ bool lt_zero(float x) { return x < 0.0f; }
// x >= 0: positive, or a zero of either sign
__host__ __device__ __forceinline__ bool ge_zero(double x) {
  const uint64_t b = f64_bits(x);
  return b <= F64_INF || b == F64_SIGN;
}
__host__ __device__ __forceinline__ bool le_zero(double x) { return ge_zero(f64_of(f64_bits(x) ^ F64_SIGN)); }
// the patterns as signed integers in the values' order (both zeros 0; NaNs
// beyond the infinities)
__host__ __device__ __forceinline__ int64_t f64_key(double x) {
  const int64_t b = (int64_t)f64_bits(x), m = b >> 63;
  return (b ^ (m & (int64_t)~F64_SIGN)) - m;
}
__host__ __device__ __forceinline__ bool gt_bits(double a, double b) {
  const int64_t ka = f64_key(a), kb = f64_key(b);
  return ka > kb && ka <= (int64_t)F64_INF && kb >= -(int64_t)F64_INF;
}
// a <= b for a >= 0 (or NaN) and any b
__host__ __device__ __forceinline__ bool le_pos(double a, double b) {
  const int64_t ka = (int64_t)f64_bits(a), kb = f64_key(b);
  return ka <= kb && kb <= (int64_t)F64_INF;
}
// |a| <= b for b >= 0 (or NaN)
__host__ __device__ __forceinline__ bool abs_le(double a, double b) {
  const uint64_t ma = f64_bits(a) & ~F64_SIGN, mb = f64_bits(b);
  return ma <= mb && mb <= F64_INF;
}
// the larger of two non-negative values, and x < infinity for x >= 0 or NaN
__host__ __device__ __forceinline__ double max_pos(double a, double b) { return f64_bits(a) > f64_bits(b) ? a : b; }
__host__ __device__ __forceinline__ float max_pos(float a, float b) { return a > b ? a : b; }
__host__ __device__ __forceinline__ bool finite_pos(double x) { return f64_bits(x) < F64_INF; }
__host__ __device__ __forceinline__ bool finite_pos(float x) { return x < INFINITY; }
// minmod: 0 unless a and b have the same strict sign, else the one of smaller
// magnitude
__host__ __device__ __forceinline__ double minmod_bits(double a, double b) {
  const uint64_t ba = f64_bits(a), bb = f64_bits(b);
  const uint64_t ma = (ba & ~F64_SIGN) - 1ull, mb = (bb & ~F64_SIGN) - 1ull;  // a zero wraps beyond every magnitude
  const bool a_small = ma <= mb;
  const uint64_t large = a_small ? mb : ma, r = a_small ? ba : bb;
  return f64_of(((int64_t)(ba ^ bb) >= 0 && large < F64_INF) ? r : 0ull);
}

}  // namespace amrdev
