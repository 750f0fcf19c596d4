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

#include <cuda_bf16.h>
#include <cuda_fp16.h>

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

// The sequences replaced, for values outside the stated ranges: calls, so that they stay behind
// their branch. Written as expressions the compiler ran them for every value beside the integer
// path and chose afterwards, and the FP64 pipe was paid as before. Per call, so and now: an
// upload at 16^3x32 in double-float 32.0 -> 8.8 us, in FP32 14.6 -> 7.5, a copy there from FP64 to
// FP32 26.3 -> 13.0, at 32^3x64 247 -> 107. Zeros are no call either: a point source is zeros.
__host__ __device__ __noinline__ inline float to_float_any(double x) { return (float)x; }
__host__ __device__ __noinline__ inline double to_double_any(float x) { return (double)x; }
__host__ __device__ __noinline__ inline float2 to_df_any(double x) {
  const float hi = (float)x;
  return make_float2(hi, (float)(x - (double)hi));
}
__host__ __device__ __noinline__ inline unsigned to_half_any(double x) { return __half_as_ushort(__double2half(x)); }
__host__ __device__ __noinline__ inline unsigned to_bf16_any(double x) {
  return __bfloat16_as_ushort(__double2bfloat16(x));
}

// The 24 leading bits of |x|, FP32's exponent before them, as if x were truncated; rem: the
// 29 bits below. For 2^-126 <= |x| < 2^127.
__host__ __device__ inline unsigned float_bits(unsigned hi, unsigned lo) {
  return (((hi & 0x7fffffffu) << 3) | (lo >> 29)) - (896u << 23);
}
__host__ __device__ inline bool zero_bits(unsigned hi, unsigned lo) { return !((hi & 0x7fffffffu) | lo); }
// 1 where those round up (nearest, ties to even)
__host__ __device__ inline unsigned rounds_up(unsigned f, unsigned rem) {
  return (rem + 0x0fffffffu + (f & 1u)) >> 29;
}

// (float)x, round to nearest even
__host__ __device__ inline float to_float(double x) {
  const unsigned long long b = bits_of(x);
  const unsigned h = (unsigned)(b >> 32), l = (unsigned)b, e = (h >> 20) & 0x7ffu;
  if (e - 897u > 252u) return zero_bits(h, l) ? float_of(h) : to_float_any(x);
  const unsigned f = float_bits(h, l);
  return float_of((h & 0x80000000u) | (f + rounds_up(f, l & 0x1fffffffu)));
}

// the bits of __double2half(x) (the last binade's carry is infinity) and __double2bfloat16(x)
__host__ __device__ inline unsigned to_half(double x) {
  const unsigned long long b = bits_of(x);
  const unsigned h = (unsigned)(b >> 32), e = (h >> 20) & 0x7ffu;
  if (e > 1038u) return to_half_any(x);
  const unsigned sign = (h >> 16) & 0x8000u, sticky = (unsigned)b ? 1u : 0u;
  if (e < 1009u) {  // below 2^-14: the multiple of 2^-24
    const unsigned r = e < 995u ? 24u : 1019u - e, m = (h & 0xfffffu) | 0x100000u, q = m >> r;
    const unsigned rem = ((m << 1) & ((2u << r) - 1u)) | sticky;
    return sign | (q + ((rem + (1u << r) - 1u + (q & 1u)) >> (r + 1u)));
  }
  const unsigned f = ((h & 0x7fffffffu) >> 10) - (1008u << 10);
  const unsigned rem = ((h & 0x3ffu) << 1) | sticky;
  return sign | (f + ((rem + 0x3ffu + (f & 1u)) >> 11));
}
__host__ __device__ inline unsigned to_bf16(double x) {
  const unsigned long long b = bits_of(x);
  const unsigned h = (unsigned)(b >> 32), e = (h >> 20) & 0x7ffu;
  if (e - 897u > 252u) return zero_bits(h, (unsigned)b) ? h >> 16 : to_bf16_any(x);
  const unsigned f = ((h & 0x7fffffffu) >> 13) - (896u << 7);
  const unsigned rem = ((h & 0x1fffu) << 1) | ((unsigned)b ? 1u : 0u);
  return ((h >> 16) & 0x8000u) | (f + ((rem + 0x1fffu + (f & 1u)) >> 14));
}

// (double)x
__host__ __device__ inline double to_double(float x) {
  const unsigned b = bits_of(x), u = b & 0x7fffffffu, e = u >> 23;
  const unsigned long long sign = (unsigned long long)(b & 0x80000000u) << 32;
  if (e - 1u >= 254u) return u ? to_double_any(x) : double_of(sign);
  return double_of(sign | (((unsigned long long)u << 29) + (896ULL << 52)));
}

// hi = (float)x, lo = (float)(x - (double)hi)
__host__ __device__ inline void to_df(double x, float& hi, float& lo) {
  const unsigned long long b = bits_of(x);
  const unsigned h = (unsigned)(b >> 32), l = (unsigned)b, e = (h >> 20) & 0x7ffu;
  if (e - 949u > 200u) {
    const float2 v = zero_bits(h, l) ? make_float2(float_of(h), 0.0f) : to_df_any(x);
    hi = v.x;
    lo = v.y;
    return;
  }
  const unsigned f = float_bits(h, l), rem = l & 0x1fffffffu, up = rounds_up(f, rem);
  hi = float_of((h & 0x80000000u) | (f + up));
  // x - hi in units of the last place of x's 53 bits: at most 2^28 in magnitude, and the
  // unit 2^(e - 1075) is a normal FP32 number, so the product is exact
  const int s = (h & 0x80000000u) ? -1 : 0, r = (((int)rem - (int)(up << 29)) ^ s) - s;
  lo = (float)r * float_of((e - 948u) << 23);
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
  const unsigned l = bits_of(lo);
  if (!((b | l) & 0x7fffffffu)) return double_of((unsigned long long)(b & l & 0x80000000u) << 32);
  return (double)hi + (double)lo;
}

}  // namespace cv
}  // namespace lqcd
