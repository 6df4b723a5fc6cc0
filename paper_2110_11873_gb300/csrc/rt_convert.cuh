// FP64 <-> FP32 on the integer pipe: the conversion instructions run on the
// FP64 pipe (1.9 a clock and SM, measured), which then bounds every kernel
// that computes in FP32 on FP64 vectors.  The same results as the conversions
// (round to nearest even, subnormal numbers kept, NaN stays NaN).  Nothing but
// the bit intrinsics is used, so that a host test can compile this file.
#pragma once

#include <stdint.h>

namespace rt {
namespace {

__device__ __forceinline__ float to_f32(double x) {
  const uint32_t hi = __double2hiint(x), lo = __double2loint(x), ab = hi & 0x7fffffffu, sg = hi & 0x80000000u;
  if (ab - 0x38100000u < 0x47f00000u - 0x38100000u) {   // a normal number below 2^128
    const uint32_t t = __funnelshift_l(lo, ab - 0x38000000u, 3), rem = lo << 3;
    return __uint_as_float((t + (uint32_t)((rem | (t & 1u)) > 0x80000000u)) | sg);
  }
  if (ab >= 0x47f00000u) return __uint_as_float((ab > 0x7ff00000u || (ab == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u) | sg);
  const int s = 926 - (int)(ab >> 20);   // a multiple of 2^-149: the mantissa over 2^s
  if (s > 54) return __uint_as_float(sg);
  const uint64_t m = ((uint64_t)((ab & 0xfffffu) | 0x100000u) << 32) | lo;
  const uint64_t q = m >> s, rem = m << (64 - s);
  return __uint_as_float(((uint32_t)q + (uint32_t)((rem | (q & 1u)) > 0x8000000000000000ull)) | sg);
}
__device__ __forceinline__ double to_f64(float x) {
  uint32_t u = __float_as_uint(x), ab = u & 0x7fffffffu;
  const uint32_t sg = u & 0x80000000u;
  uint32_t bias = 0x38000000u;
  if (ab - 0x00800000u >= 0x7f800000u - 0x00800000u) {
    if (ab == 0) return __hiloint2double((int)sg, 0);
    if (ab >= 0x7f800000u) {   // an infinity or a NaN
      bias = 0x70000000u;
    } else {                   // subnormal: shift the leading bit to its place
      const int z = __clz(ab) - 8;
      ab = (ab << z) & 0x7fffffu;
      bias = 0x38100000u - ((uint32_t)z << 20);
    }
  }
  return __hiloint2double((int)(((ab >> 3) + bias) | sg), (int)(ab << 29));
}

}  // namespace
}  // namespace rt
