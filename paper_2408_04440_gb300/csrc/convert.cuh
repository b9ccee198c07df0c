// convert.cuh -- conversions between FP64 and FP32 / BF16 in integer
// arithmetic.  GB300's FP64 pipe, which the conversion instructions occupy,
// takes one warp instruction per about 19 cycles and SM: a pass that converts
// every entry was bound by it, not by memory.  Same results as the instructions
// (round to nearest, ties to even); values outside the narrow type's normal
// range take the instruction.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace {

__device__ inline float f32_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  if (ex < 898 || ex > 1149) return ex == 0 ? ((long long)b < 0 ? -0.0f : 0.0f) : (float)x;
  const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);
  const unsigned m = (unsigned)(r >> 29) - (896u << 23);  // modulo 2^32: exponent and fraction
  return __uint_as_float((m & 0x7fffffffu) | ((unsigned)(b >> 32) & 0x80000000u));
}
__device__ inline uint16_t bf16_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  if (ex < 898 || ex > 1149)
    return ex == 0 ? (uint16_t)((b >> 48) & 0x8000u) : __bfloat16_as_ushort(__double2bfloat16(x));
  const unsigned long long r = b + 0xfffffffffffull + ((b >> 45) & 1ull);
  return (uint16_t)((((unsigned)(r >> 45) - (896u << 7)) & 0x7fffu) | ((unsigned)(b >> 48) & 0x8000u));
}
__device__ inline double f64_of(float x) {
  const unsigned b = __float_as_uint(x);
  const unsigned ex = (b >> 23) & 0xffu;
  if (ex - 1u >= 254u)
    return (b << 1) == 0u ? __longlong_as_double((long long)((unsigned long long)b << 32)) : (double)x;
  return __longlong_as_double(
      (long long)((((unsigned long long)(b & 0x7fffffffu) << 29) + (896ull << 52)) | ((unsigned long long)(b & 0x80000000u) << 32)));
}
__device__ inline double f64_of_bf16(uint16_t v) { return f64_of(__uint_as_float((unsigned)v << 16)); }

}  // namespace
