// FP64 reciprocal, square root and reciprocal square root for a chip whose FP64 pipe is
// narrow (an FP64 warp instruction holds its sub-partition for 64 clocks, a division or a
// square root 8-10 of them): one third-order Newton step on 62-bit integers from an FP32
// seed, about 45-55 integer instructions.  Used where the FP64 pipe sets the time: HLLC
// k_face at 16^3, N = 7: 238 -> 181 FP64 instructions per face node, 354 -> 275 us (then 226 with
// fx_visc_normal).  Results are within 0.52 units in the last place;
// zero, subnormal and very large arguments, infinities, NaN and negative radicands take the
// language's operation.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace flexi {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float seed_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float seed_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ unsigned mulhi32(unsigned a, unsigned b) { return __umulhi(a, b); }
__device__ __forceinline__ uint64_t bits_of(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double of_bits(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ float float_of_bits(unsigned b) { return __uint_as_float(b); }
__device__ __forceinline__ unsigned to_uint(float x) { return __float2uint_rz(x); }
#else
inline float seed_rcp(float x) { return 1.0f / x; }
inline float seed_rsqrt(float x) { return 1.0f / sqrtf(x); }
inline unsigned mulhi32(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
inline uint64_t bits_of(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
inline double of_bits(uint64_t b) { double x; memcpy(&x, &b, 8); return x; }
inline float float_of_bits(unsigned b) { float x; memcpy(&x, &b, 4); return x; }
inline unsigned to_uint(float x) { return (unsigned)x; }
#endif

// a b of two signed words (one multiply; the compiler may otherwise widen the operands first)
__host__ __device__ __forceinline__ int64_t mul_wide(int a, int b) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (int64_t)a * b;
#endif
}
__host__ __device__ __forceinline__ uint64_t mul_wideu(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (uint64_t)a * b;
#endif
}

// y0 (1 + t) 2^62 for y0 = Y / 2^31 and t in units of 2^-62, |t| < 2^42
__host__ __device__ __forceinline__ uint64_t newton_apply(unsigned Y, int64_t t) {
  const int th = (int)(t >> 20), tl = (int)(t & 0xfffff);
  return ((uint64_t)Y << 31) + (uint64_t)(mul_wide((int)Y, th) >> 11) + (uint64_t)(mul_wide((int)Y, tl) >> 31);
}

// 1 / m = r0 (1 + e + e^2 + O(e^3)) with e = 1 - m r0
__host__ __device__ __forceinline__ double fp64_rcp(double x) {
  const uint64_t b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const int ex = (int)((hi >> 20) & 0x7ff);
  if (ex - 1 >= 2043 || ex == 0) return 1.0 / x;
  const unsigned M = (hi << 11) | 0x80000000u | (lo >> 21);  // m 2^31, 1 <= m < 2
  unsigned Y = to_uint(seed_rcp(float_of_bits(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29))) * 2147483648.0f);
  if (Y > 0x7fffffffu) Y = 0x7fffffffu;
  const int64_t e = (int64_t)((1ull << 62) - (mul_wideu(M, Y) + mulhi32(lo << 11, Y)));  // 2^62 (1 - m r0)
  const int eh = (int)(e >> 20);
  const uint64_t r = newton_apply(Y, e + (mul_wide(eh, eh) >> 22));  // 2^62 / m
  return of_bits((((uint64_t)(unsigned)(2044 - ex)) << 52) + ((r + 0x100) >> 9) + (b & 0x8000000000000000ull));
}

// 2^62 / sqrt(m) for m = M / 2^61 in [1, 4): y0 (1 + e/2 + 3/8 e^2 + O(e^3)), e = 1 - m y0^2
__host__ __device__ __forceinline__ uint64_t rsqrt_fixed(uint64_t M, float m) {
  unsigned Y = to_uint(seed_rsqrt(m) * 2147483648.0f);
  if (Y > 0x7fffffffu) Y = 0x7fffffffu;
  const uint64_t y2 = mul_wideu(Y, Y);
  const unsigned Mh = (unsigned)(M >> 32), Ml = (unsigned)M, A = (unsigned)(y2 >> 32), B = (unsigned)y2;
  const uint64_t p = mul_wideu(Mh, A) + mulhi32(Mh, B) + mulhi32(Ml, A);  // 2^59 m y0^2
  const int64_t e = (int64_t)((1ull << 59) - 1 - p);                      // the two dropped fractions have mean one
  const int eh = (int)(e >> 18);
  return newton_apply(Y, (e << 2) + ((3 * mul_wide(eh, eh)) >> 23));
}

__host__ __device__ __forceinline__ double fp64_rsqrt(double x) {
  const uint64_t b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32);
  const int ex = (int)(hi >> 20);  // with the sign: negative arguments are out of range
  if (ex == 0 || ex >= 2046) {
#ifdef __CUDA_ARCH__
    return ::rsqrt(x);
#else
    return 1.0 / ::sqrt(x);
#endif
  }
  const int odd = (ex & 1) ^ 1;  // ex - 1023 = 2 k + odd
  const uint64_t mant = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint64_t y = rsqrt_fixed(mant << (9 + odd), float_of_bits(0x3f800000u + ((unsigned)odd << 23) + (unsigned)((mant >> 29) & 0x7fffff)));
  const int k = (ex - 1023 - odd) >> 1;
  return of_bits((((uint64_t)(unsigned)(1021 - k)) << 52) + ((y + 0x100) >> 9));
}

__host__ __device__ __forceinline__ double fp64_sqrt(double x) {
  const uint64_t b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32);
  const int ex = (int)(hi >> 20);
  if (ex == 0 || ex >= 2046) return ::sqrt(x);
  const int odd = (ex & 1) ^ 1;
  const uint64_t mant = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint64_t M = mant << (9 + odd);
  const uint64_t y = rsqrt_fixed(M, float_of_bits(0x3f800000u + ((unsigned)odd << 23) + (unsigned)((mant >> 29) & 0x7fffff)));
  // M y / 2^64 = sqrt(m) 2^59
  const unsigned Mh = (unsigned)(M >> 32), Ml = (unsigned)M, yh = (unsigned)(y >> 32), yl = (unsigned)y;
  const uint64_t mid = mul_wideu(Mh, yl) + mulhi32(Ml, yl);
  const uint64_t mid2 = mul_wideu(Ml, yh) + (unsigned)mid;
  const uint64_t s = mul_wideu(Mh, yh) + (mid >> 32) + (mid2 >> 32);
  const int k = (ex - 1023 - odd) >> 1;
  return of_bits((((uint64_t)(unsigned)(1022 + k)) << 52) + ((s + 0x40) >> 7));
}

}  // namespace flexi
