// Conversions between FP64, FP32 and double-float on the integer and FP32 pipes.
//
// A conversion instruction between FP64 and FP32 runs on the FP64 pipe, at 1/64 of the FP32
// rate on GB300, so a layout pass that converts every real with them is bound there and not
// by HBM (double-float links of 24^3x48 from the FP64 master: 345 us for 0.11 ms of HBM
// traffic). The functions below take the bits apart instead. Each gives the value of the
// instruction sequence it replaces, bit for bit: inside the exponent range stated it is
// exact arithmetic on the bits, outside it (subnormals, infinities, NaN, the ends of the
// range) it is that sequence itself.
#pragma once

#include "field.cuh"

namespace lqcd {
namespace cv {

__host__ __device__ inline unsigned long long bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ inline double double_of(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
#endif
}
__host__ __device__ inline unsigned bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned b;
  __builtin_memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ inline float float_of(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  __builtin_memcpy(&x, &b, 4);
  return x;
#endif
}
__host__ __device__ inline int round_to_int(float x) {  // nearest, ties to even
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)__builtin_rintf(x);
#endif
}

// (float)x, round to nearest even
__host__ __device__ inline float to_float(double x) {
  const unsigned long long b = bits_of(x), u = b & 0x7fffffffffffffffULL;
  const unsigned e = (unsigned)(u >> 52), sign = (unsigned)(b >> 32) & 0x80000000u;
  if (u == 0) return float_of(sign);
  if (e < 897u || e > 1149u) return (float)x;
  unsigned f = (unsigned)(u >> 29) - (896u << 23);
  const unsigned rem = (unsigned)u & 0x1fffffffu;
  f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;
  return float_of(sign | f);
}

// (double)x
__host__ __device__ inline double to_double(float x) {
  const unsigned b = bits_of(x), u = b & 0x7fffffffu, e = u >> 23;
  const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
  if (u == 0) return double_of(sign);
  if (e - 1u >= 254u) return (double)x;
  return double_of(sign | (((unsigned long long)u << 29) + (896ULL << 52)));
}

// hi = (float)x, lo = (float)(x - (double)hi)
__host__ __device__ inline void to_df(double x, float& hi, float& lo) {
  const unsigned long long b = bits_of(x), u = b & 0x7fffffffffffffffULL;
  const unsigned e = (unsigned)(u >> 52), sign = (unsigned)(b >> 32) & 0x80000000u;
  if (u == 0) {
    hi = float_of(sign);
    lo = 0.0f;
    return;
  }
  if (e < 949u || e > 1149u) {
    hi = (float)x;
    lo = (float)(x - (double)hi);
    return;
  }
  unsigned f = (unsigned)(u >> 29) - (896u << 23);
  const unsigned rem = (unsigned)u & 0x1fffffffu;
  const unsigned up = (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;
  f += up;
  hi = float_of(sign | f);
  // x - hi in units of the last place of x's 53 bits: at most 2^28 in magnitude, and the
  // unit 2^(e - 1075) is a normal FP32 number, so the product is exact
  int r = (int)rem - (int)(up << 29);
  if (sign) r = -r;
  lo = r == 0 ? 0.0f : (float)r * float_of((e - 948u) << 23);
}

// (double)hi + (double)lo, rounded once
__host__ __device__ inline double from_df(float hi, float lo) {
  const unsigned b = bits_of(hi), e = (b >> 23) & 255u;
  if (e >= 53u && e < 255u) {
    // lo in units of the last place of a 53-bit hi, with hi's sign taken out; at most 2^28 in
    // magnitude for a normalised pair. Below a power of two the last place is half as large.
    const float u = lo * float_of((306u - e) << 23), t = (b >> 31) ? -u : u;
    if (fabsf(t) <= 268435456.0f && (t >= 0.0f || (b & 0x7fffffu))) {
      const unsigned long long m =
          ((unsigned long long)((b & 0x7fffffu) | 0x800000u) << 29) + (unsigned long long)(long long)round_to_int(t);
      return double_of(((unsigned long long)(b & 0x80000000u) << 32) | (((unsigned long long)(e + 895u) << 52) + m));
    }
  }
  return (double)hi + (double)lo;
}

}  // namespace cv
}  // namespace lqcd
