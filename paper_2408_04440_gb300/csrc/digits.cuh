// digits.cuh -- device side of the digit scheme of gemm_f64.h: row exponents
// and the digits of an entry.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_f64.h"

namespace gemm64 {

__device__ inline int exp_of(const int *exps, long i) { return max(exps[i] - kExpBias, kExpMin); }
// Magnitude bits of x: ordered like |x|, infinities and then NaNs on top, so
// that row maxima are taken in integers.
__device__ inline unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
// Biased exponent of a row whose largest magnitude bits are m > 0: every
// |x| < 2^(result - kExpBias).  (The sign is masked again: the compiler takes
// the mask above for an FP64 absolute value, which may keep a NaN's sign.)
__device__ inline int biased_exp(unsigned long long m) {
  const int ex = (int)(m >> 52) & 0x7ff;
  if (ex == 0x7ff) return kExpPoison;
  return (ex > 0 ? ex - 1022 : (64 - __clzll((long long)m)) - 1074) + kExpBias;
}
// x 2^(56 - e) rounded to the nearest integer (ties to even), for |x| < 2^e:
// below 2^56 in magnitude.  In integer arithmetic on the significand: the FP64
// pipe issues about one warp instruction per 19 cycles and SM, and a multiply
// and a conversion per entry there took longer than the entry's memory traffic.
// 0 where e is a poisoned row's.
__device__ inline long long to_fixed(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  if (ex > 0) m |= 1ull << 52;
  else ex = 1;
  const int sh = ex - 1019 - e;  // x 2^(56 - e) = m 2^sh, sh <= 3
  unsigned long long X;
  if (sh >= 0) {
    X = m << sh;
  } else {
    const int r = -sh < 54 ? -sh : 54;  // m < 2^53: 2^-54 m rounds to 0
    X = (m + ((1ull << (r - 1)) - 1) + ((m >> r) & 1ull)) >> r;
  }
  return (long long)b < 0 ? -(long long)X : (long long)X;
}

// The NS digits of X (|X| <= 2^56, the unit of the last digit is 2^-56): peeled
// off from the top, each rounded to nearest, so |digit 0| <= 128 and
// |digit p| <= 64 for p >= 1 and sum_p digit_p 2^(7 (NS - 1 - p)) = X exactly.
// As BF16 bits: a digit is at most eight bits wide, so the upper half of its
// FP32 pattern (formed by an add of 1.5 2^23, no conversion) is exact.
__device__ inline void digit_bits(long long X, uint32_t (&d)[NS]) {
#pragma unroll
  for (int p = 0; p < NS; p++) {
    const int sh = SLICE_BITS * (NS - 1 - p);
    const long long dg = (sh > 0) ? ((X + (1LL << (sh > 0 ? sh - 1 : 0))) >> sh) : X;
    X -= dg << sh;
    d[p] = __float_as_uint(__int_as_float(0x4B400000 + (int)dg) - 12582912.0f) >> 16;
  }
}
// Digits of v with row exponent e written d[0], d[plane], ...
__device__ inline void write_digits(double v, int e, uint16_t *d, size_t plane) {
  uint32_t g[NS];
  digit_bits(to_fixed(v, e), g);
#pragma unroll
  for (int p = 0; p < NS; p++) d[p * plane] = (uint16_t)g[p];
}
// The same for two neighbouring columns (d 4-byte aligned).
__device__ inline void write_digits2(double v0, double v1, int e, uint16_t *d, size_t plane) {
  uint32_t g0[NS], g1[NS];
  digit_bits(to_fixed(v0, e), g0);
  digit_bits(to_fixed(v1, e), g1);
#pragma unroll
  for (int p = 0; p < NS; p++) *reinterpret_cast<uint32_t *>(d + p * plane) = g0[p] | (g1[p] << 16);
}

// Digits of a batch of matrices read through a source S, K-major: one CTA of
// 256 threads per (32 rows, batch).  A first pass over k takes the rows'
// maxima, a second one (its reads hit L2) writes the digits; K is filled with
// zeros up to kpad(b).  S gives, for batch b:
//   rows(b), nk(b), kpad(b) (a multiple of 32);
//   load(b, r, k), for r < rows(b), k < nk(b);
//   dst(b, r): offset of row r's digit plane 0 (k contiguous; even);
//   e(b, r): its exponent's index;
// and digits, exps, plane (elements between planes), flag (set when a row
// holds an infinity or a NaN).  KFAST: k, not r, is contiguous in the source.
template <class S, bool KFAST>
__global__ void __launch_bounds__(256) k_source_digits(const S s) {
  __shared__ double blk[32][33];
  __shared__ unsigned long long red[8][33];
  __shared__ int se[32];
  const int b = blockIdx.x, r0 = blockIdx.y * 32, rows = s.rows(b), nk = s.nk(b);
  if (r0 >= rows) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (KFAST) {
    for (int q = 0; q < 4; q++) {
      const int r = r0 + w + 8 * q;
      unsigned long long m = 0;
      if (r < rows)
        for (int k = lane; k < nk; k += 32) m = max(m, mag_bits(s.load(b, r, k)));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) red[0][w + 8 * q] = m;
    }
    __syncthreads();
  } else {
    unsigned long long m = 0;
    if (r0 + lane < rows) {
#pragma unroll 4
      for (int k = w; k < nk; k += 8) m = max(m, mag_bits(s.load(b, r0 + lane, k)));
    }
    red[w][lane] = m;
    __syncthreads();
    if (w == 0) {
      for (int q = 1; q < 8; q++) m = max(m, red[q][lane]);
      red[0][lane] = m;
    }
  }
  if (w == 0) {
    const unsigned long long m = red[0][lane];
    const int eb = m > 0 ? biased_exp(m) : 0;
    if (r0 + lane < rows) s.exps[s.e(b, r0 + lane)] = eb;
    if (eb == kExpPoison && s.flag) *s.flag = 1;
    se[lane] = max(eb - kExpBias, kExpMin);
  }
  const int h = threadIdx.x >> 4, c = 2 * (threadIdx.x & 15), kp = s.kpad(b);
  for (int k0 = 0; k0 < kp; k0 += 32) {
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int r = r0 + (KFAST ? w + 8 * q : lane), k = k0 + (KFAST ? lane : w + 8 * q);
      v[q] = r < rows && k < nk ? s.load(b, r, k) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; q++) {
      if (KFAST) blk[w + 8 * q][lane] = v[q];
      else blk[lane][w + 8 * q] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const int rr = h + 16 * q;
      if (r0 + rr < rows)
        write_digits2(blk[rr][c], blk[rr][c + 1], se[rr], s.digits + s.dst(b, r0 + rr) + k0 + c, s.plane);
    }
  }
}

}  // namespace gemm64
