// rng.cuh -- the counter-based normal generator of the library (device
// code shared by the sampler and the emulation nugget): Philox4x32-10
// (Salmon, Moraes, Dror, Shaw, SC'11) at counter {p mod 2^32, p >> 32,
// column, stream id}, key {seed mod 2^32, seed >> 32}; two 53-bit uniforms
// u1 in (0,1], u2 in [0,1); Box-Muller gives rows 2p (cosine) and 2p+1 (sine).
#pragma once
#include <stdint.h>

#include "rng_tables.h"

namespace {

__device__ inline void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; r++) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    uint32_t n0 = hi1 ^ c[1] ^ k0;
    uint32_t n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

// -2 ln and the sine / cosine of the pair.  GB300 issues about one FP64 warp
// instruction per 19 cycles and SM, so their number is the generator's time:
// about 32 here, against some 90 with log, sqrt, cos and sin of the library.
// The argument reductions are integer arithmetic on the 53-bit words; both
// functions are a table entry at the nearest of 256 nodes plus a short Taylor
// polynomial (the table-driven logarithm of Tang, ACM TOMS 16, 1990, with
// u1 = 2^-E m, ln m = ln c + ln(1 + r)); the square root is Goldschmidt's
// iteration from a single-precision reciprocal root.  Errors: below 1 ulp of
// ln, 2^-53 absolute in the sine and cosine (2 pi u2 rounded to FP64 before the
// library's sin and cos is off by up to 2^-51).
struct NormalTables {
  double lt[257][3], le[54][2], tt[256][2];
  __device__ void load() {  // whole CTA, then a barrier
    for (int q = threadIdx.x; q < 257 * 3; q += blockDim.x) (&lt[0][0])[q] = (&kLogTab[0][0])[q];
    for (int q = threadIdx.x; q < 54 * 2; q += blockDim.x) (&le[0][0])[q] = (&kLogExp[0][0])[q];
    for (int q = threadIdx.x; q < 256 * 2; q += blockDim.x) (&tt[0][0])[q] = (&kTrigTab[0][0])[q];
  }
};

// -2 ln(k 2^-53) for 1 <= k <= 2^53.
__device__ inline double minus_2_ln(uint64_t k, const NormalTables &T) {
  const int lz = __clzll((long long)k);                 // 10 .. 63
  const uint64_t f = (k << lz) << 1 >> 12;              // fraction bits of m = k / 2^(63 - lz) in [1, 2)
  const double m = __longlong_as_double((long long)(f | 0x3ff0000000000000ull));
  const int j = (int)((f + (1ull << 43)) >> 44);        // nearest node c = 1 + j / 256
  const int e = lz - 10 - (j >= 128 ? 1 : 0);           // from j = 128 on m / 2 is reduced: no cancellation near 1
  const double r = fma(m, T.lt[j][0], -1.0);            // |r| <= 2^-9
  double p = fma(r, 2.0 / 6.0, -2.0 / 5.0);
  p = fma(r, p, 2.0 / 4.0);
  p = fma(r, p, -2.0 / 3.0);
  p = fma(r, p, 1.0);
  double lo = T.lt[j][2] + T.le[e][1];
  lo = fma(r * r, p, lo);
  lo = fma(-2.0, r, lo);
  return (T.lt[j][1] + T.le[e][0]) + lo;                // the first sum is exact (multiples of 2^-40)
}

// sqrt(x), x = 0 or 2^-60 < x < 2^10.
__device__ inline double sqrt_of(double x) {
  // the leading 24 bits of x as FP32 and 1 / sqrt of them back as FP64, by their bits
  const uint64_t xb = (uint64_t)__double_as_longlong(x);
  const float xf = __uint_as_float((uint32_t)((xb >> 29) - ((uint64_t)(1023 - 127) << 23)));
  const uint64_t yb = ((uint64_t)__float_as_uint(rsqrtf(xf)) << 29) + ((uint64_t)(1023 - 127) << 52);
  const double y = __longlong_as_double((long long)yb);
  double g = x * y, h = __longlong_as_double((long long)(yb - (1ull << 52)));  // h = y / 2
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  const double d = fma(-g, g, x);
  g = fma(d, h, g);
  return x > 0.0 ? g : 0.0;
}

// Normals of pair p (rows 2p, 2p+1) of column col.
__device__ inline double2 normal_pair(uint64_t seed, uint32_t stream_id, long p, int col, const NormalTables &T) {
  uint32_t c[4] = {(uint32_t)((uint64_t)p & 0xffffffffu), (uint32_t)((uint64_t)p >> 32), (uint32_t)col,
                   stream_id};
  philox4x32_10(c, (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
  const uint64_t a = ((uint64_t)c[0] << 21) | (uint64_t)(c[1] >> 11);
  const uint64_t b = ((uint64_t)c[2] << 21) | (uint64_t)(c[3] >> 11);
  const double rad = sqrt_of(minus_2_ln(a + 1, T));  // u1 = (a + 1) 2^-53
  // u2 = b 2^-53: node j / 256 and the rest of the turn
  const int j = (int)((b + (1ull << 44)) >> 45);
  const long long rest = (long long)(b - ((uint64_t)j << 45));  // |rest| <= 2^44
  // rest as FP64: an integer added to the bits of 1.5 2^52
  const double t = (__longlong_as_double(0x4338000000000000ll + rest) - 6755399441055744.0) *
                   (6.283185307179586476925286766559 * 0x1p-53);
  const double t2 = t * t;
  const double sn = fma(t * t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), t);
  const double cn = t2 * fma(t2, fma(t2, -1.0 / 720.0, 1.0 / 24.0), -0.5);  // cos - 1
  const double C = T.tt[j & 255][0], S = T.tt[j & 255][1];
  return make_double2(rad * (C + fma(C, cn, -(S * sn))), rad * (S + fma(S, cn, C * sn)));
}

}  // namespace
