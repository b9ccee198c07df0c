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
  const int sh = ex - 1019 - e;  // x 2^(56 - e) = m 2^sh, sh <= 3 (<= 6 and m < 2^50 for denormal rows)
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

// 2^e for integer e in the normal range (exact).
__device__ inline double exp2i(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
// fixed_scaled for any s: near the ends of the FP64 range, and NaN where s
// carries the poison of a row with an infinity or a NaN.
static __device__ __noinline__ double fixed_scaled_any(long long hi, unsigned lo, int s) {
  if (s > kExpPoison / 2) return __longlong_as_double(0x7ff8000000000000ll);
  const double x = fma((double)hi, 0x1p-31, (double)lo * 0x1p-63);
  const int s1 = max(-1000, min(1000, s));
  return x * exp2i(s1) * exp2i(max(-1000, min(1000, s - s1)));
}
// Adds the chunk's sum_g G_g 2^-7(g+2), for the group sums G_g of one output
// (column x of r[g]), to the exact fixed-point accumulator (hi, lo) of value
// hi 2^-31 + lo 2^-63 (lo unsigned, below 2^32).  Each G_g is an integer held
// exactly in FP32 (below 2^24, see the header), so the chunk's sum is formed
// in integer arithmetic: groups 2..7 by Horner in 64 bits, T = sum_{g>=2}
// G_g 2^(7(7-g)), |T| < 2^59 (|G_g| < 2^24 for g >= 1 with KCHUNK = 384:
// at most two products of a leading digit, |d_0| <= 128, and g - 1 of
// trailing digits, |d_p| <= 64, per K term), and groups 0..1 as Q = 2^7 G_0
// + G_1, |Q| < 2^30 (|G_0| <= 384 * 2^14, |G_1| <= 384 * 2^14).  The chunk's value is Q 2^-21 + T 2^-63
// = (2^10 Q + floor(T / 2^32)) 2^-31 + (T mod 2^32) 2^-63; the low word's
// carry moves into hi, which grows by less than 2^41 per chunk.  No FP64
// instruction runs per chunk: the FP64 pipe, GB300's slowest unit, is used for
// one add per output at the end of the item.
static_assert(NS == 8 && SLICE_BITS == 7 && KCHUNK <= 384, "fold_groups is written for 8 digits of 7 bits");
__device__ __forceinline__ void fold_groups(const uint32_t (&r)[NS][2], int x, long long &hi, unsigned &lo) {
  int gi[NS];
#pragma unroll
  for (int g = 0; g < NS; g++) gi[g] = __float2int_rn(__uint_as_float(r[g][x]));  // exact: integers below 2^24
  long long t = gi[2];
#pragma unroll
  for (int g = 3; g < NS; g++) t = t * 128 + gi[g];
  const long long q = gi[0] * 128 + gi[1];
  const unsigned l = lo + (unsigned)t;  // low 32 bits of T, modulo 2^32
  hi += q * 1024 + (t >> 32) + (l < lo ? 1 : 0);  // arithmetic shift: floor; carry of the low word
  lo = l;
}
// (hi 2^-31 + lo 2^-63) 2^s rounded once to FP64 (ties to even), for s that
// keeps the result in the normal range: normalised, rounded and packed in
// integer arithmetic.  Two conversions, an FMA and a multiply on the FP64 pipe
// took about 20 k cycles per 128 x 64 block, as long as the MMAs of K = 256.
// s out of range: the same value through FP64 arithmetic (fixed_scaled_any).
__device__ __forceinline__ double fixed_scaled(long long hi, unsigned lo, int s) {
  const bool neg = hi < 0;
  // |hi 2^32 + lo| = ahi 2^32 + alo
  const unsigned alo = neg ? 0u - lo : lo;
  const unsigned long long ahi = (unsigned long long)(neg ? ~hi + (lo == 0u) : hi);
  unsigned long long t;  // the leading 64 bits, top bit set
  int lz;
  bool sticky = false;
  if (ahi != 0) {
    lz = __clzll((long long)ahi);
    t = ahi << lz;
    if (lz >= 32) {
      t |= (unsigned long long)alo << (lz - 32);
    } else {
      t |= (unsigned long long)alo >> (32 - lz);
      sticky = (alo << lz) != 0u;
    }
  } else {
    if (alo == 0u) return s > kExpPoison / 2 ? fixed_scaled_any(hi, lo, s) : 0.0;  // a poisoned row's digits are 0
    const int l = __clz((int)alo);
    t = (unsigned long long)alo << (32 + l);
    lz = 64 + l;
  }
  const int e = 1055 - lz + s;  // biased exponent
  if (e < 1 || e > 2045) return fixed_scaled_any(hi, lo, s);
  unsigned long long m = t >> 11;
  const unsigned rem = (unsigned)t & 0x7ffu;
  m += (rem > 0x400u || (rem == 0x400u && (sticky || (m & 1ull)))) ? 1ull : 0ull;
  m += (unsigned long long)(e - 1) << 52;  // the implicit bit adds one to the exponent; so does a carry
  return __longlong_as_double((long long)(m | (neg ? 0x8000000000000000ull : 0ull)));
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
