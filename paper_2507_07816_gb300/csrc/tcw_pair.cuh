// tcw_pair.cuh -- FP64 values as fp32 pairs, and the FP64 reciprocal from an fp32
// one, with integer instructions in place of FP64 conversions.
//
// A conversion between double and float holds the FP64 pipe as long as an FP64
// product does (19 cycles per warp and SM), so the ordinary range, 2^-60 <= |v| <
// 2^100, moves the bits: doubles and floats differ by 29 bits of mantissa and 896
// in the exponent.  Outside it the plain conversions and division run.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tcw {

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ bool split_range(double v) {
  return (unsigned)((__double2hiint(v) >> 20 & 0x7ff) - 963) < 160u;   // 2^-60 <= |v| < 2^100
}

// The float nearest to v (ties away from zero).
__device__ __forceinline__ float near_float(double v) {
  if (!split_range(v)) return (float)v;
  const uint64_t u = (uint64_t)__double_as_longlong(v) + (1u << 28);
  return __uint_as_float(((unsigned)(u >> 32) & 0x80000000u) | ((unsigned)(u >> 29) + 0x40000000u));
}

// 1 / v by one step of Householder's iteration of third order from the fp32
// approximation s: s (1 + e + e^2) with e = 1 - v s drops e^3, below 2^-65 (|e| <
// 2^-21.4: v rounded to 24 bits, and s off by one unit), and is rounded once.
__device__ __forceinline__ double reciprocal(double v) {
  if (!split_range(v)) return 1.0 / v;
  const unsigned u = __float_as_uint(rcp_approx(near_float(v)));   // a normal float: 2^-100 .. 2^60
  const double s = __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  const double e = fma(-v, s, 1.0);
  return fma(s, fma(e, e, e), s);
}

// v as hi + lo: hi = near_float(v), lo the float of the 29 bits below.
__device__ __forceinline__ void split_float(double v, float& hi, float& lo) {
  if (!split_range(v)) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
    return;
  }
  const uint64_t u = (uint64_t)__double_as_longlong(v) + (1u << 28);
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  hi = __uint_as_float(sign | ((unsigned)(u >> 29) + 0x40000000u));
  // what is left, in units of v's own last place
  const unsigned ev = (unsigned)__double2hiint(v) >> 20 & 0x7ffu;
  const float unit = __uint_as_float(sign | ((ev - 1023 - 52 + 127) << 23));
  lo = (float)((int)((unsigned)u & 0x1fffffffu) - (1 << 28)) * unit;
}

}  // namespace tcw
