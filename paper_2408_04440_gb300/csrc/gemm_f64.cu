// gemm_f64.cu -- FP64-accurate tile update on the BF16 tensor cores for the
// FP64-class tiles of the mixed-precision factor (see gemm_f64.h for the
// digit scheme and why every tensor-core sum is exact).
//
// Warp roles (640 threads, one CTA per SM, persistent over the item list):
//   warp 0      TMA producer: per K stage the NS digit planes of the A block
//               (128 x 32) and of the B block (64 x 32), 96 KB.
//   warp 1      TMEM allocator + MMA issuer: per 16-deep K step the 36 digit
//               products with p + q < NS, product (p, q) into the group
//               accumulator g = p + q (TMEM columns g * 64 .. g * 64 + 63).
//               The digit planes of B are contiguous in a stage and so are the
//               groups in TMEM, so digit p of A meets up to four digits of B
//               in one MMA of N = 256: 12 MMAs instead of 36.  A 64-column MMA
//               is bound by its operand reads from shared memory (6 KB for 32
//               cycles of math); merged, a K step reads 120 KB instead of 216.
//   warps 2..3  idle (registers come in groups of four warps)
//   warps 4..19 epilogue (four warps per TMEM lane quarter, 16 columns each;
//               eight warps of 32 columns left the schedulers idle between
//               dependent integer steps):
//               every KCHUNK of K, the 8 group accumulators are folded in
//               integer arithmetic into exact fixed-point accumulators
//               (fold_groups), rounded to FP64 once per item (fixed_scaled);
//               after the last chunk the row scales are applied and the block
//               is subtracted from the FP64 output.
// The 8 accumulators fill TMEM, so the MMA warp waits for the epilogue to
// drain them before the next chunk.
#include <cuda_bf16.h>

#include <algorithm>

#include "digits.cuh"
#include "gemm_f64.h"
#include "gemm_tc.h"
#include "tc.cuh"

namespace gemm64 {
namespace {

constexpr int A_SL = BM * BK * 2;                     // one A digit plane: 8 KB
constexpr int B_SL = BN * BK * 2;                     // one B digit plane: 4 KB
constexpr int STAGE_BYTES = NS * (A_SL + B_SL);       // 96 KB
constexpr int RING_BYTES = STAGES * STAGE_BYTES;
constexpr int BAR_BYTES = 128;
constexpr int SMEM_BYTES = RING_BYTES + BAR_BYTES + 1024;  // + alignment slack
constexpr int NTHREADS = 640;
constexpr int EPI_WARP0 = 4;                                // warps 4..19: epilogue
constexpr int EC = 16;                                      // output columns per epilogue thread
constexpr int EPI_THREADS = NTHREADS - 32 * EPI_WARP0;
constexpr uint32_t TMEM_COLS = 512;
constexpr int QMERGE = 4;  // digits of B per MMA (N = 256, the widest)
constexpr int CHUNK_STAGES = KCHUNK / BK;
static_assert(NS * BN <= (int)TMEM_COLS, "group accumulators must fit in TMEM");

struct Shared {
  uint64_t full[STAGES];
  uint64_t empty[STAGES];
  uint64_t tfull;
  uint64_t tempty;
  uint64_t done;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Shared) <= BAR_BYTES, "barrier block");

__device__ inline bool failed(const int *st) { return *((volatile const int *)st) != DEV_OK; }

__device__ inline void raise_timeout(Shared *sh, int *status) {
  sh->abort = 1;
  status_timeout(status, 4);
}

// ------------------------------------------------------------- digits
// A 32 x 32 block (256 threads) in shared memory, row rr with exponent
// exp(rr), to its digit planes at d + rr * ld: a half warp per row, two
// columns per lane.
template <class Exp>
__device__ inline void write_block_digits(const double (&blk)[32][33], Exp exp, uint16_t *d, size_t ld, size_t plane) {
  const int h = threadIdx.x >> 4, c = 2 * (threadIdx.x & 15);
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int rr = h + 16 * q;
    write_digits2(blk[rr][c], blk[rr][c + 1], exp(rr), d + (size_t)rr * ld + c, plane);
  }
}

// Row exponents: one CTA per (32 rows, listed tile, stripe of the columns):
// lane = row, warps stride the stripe's columns; exp[base + r] =
// max(exp[base + r], e_r) with every |x_rc| < 2^e_r (the stripes combine
// through the atomic maximum).
__global__ void __launch_bounds__(256)
    k_rowexp64(const double *__restrict__ t64, const float *__restrict__ t32, const unsigned char *__restrict__ cls,
               const int4 *__restrict__ jobs, int nb, int *__restrict__ exps, const int *st) {
  if (failed(st)) return;
  __shared__ unsigned long long red[8][33];
  int4 jb = jobs[blockIdx.y];
  size_t base = (size_t)jb.x * nb * nb;
  bool f64 = cls[jb.x] == EMU_CLASS_FP64;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int r = blockIdx.x * 32 + lane;
  unsigned long long m = 0;
  for (int c = blockIdx.z * 8 + w; c < nb; c += 8 * gridDim.z) {
    size_t o = base + r + (size_t)c * nb;
    double x = f64 ? t64[o] : (double)t32[o];
    m = max(m, mag_bits(x));
  }
  red[w][lane] = m;
  __syncthreads();
  if (w == 0) {
    for (int q = 1; q < 8; q++) m = max(m, red[q][lane]);
    if (m > 0) atomicMax(&exps[jb.z + r], biased_exp(m));
  }
}

// The NS digit planes of each listed tile.  One CTA per (32 x 32 block,
// tile): the block is read column by column (coalesced in the column-major
// tile), transposed in shared memory, and each digit plane is written row by
// row (coalesced in the row-major plane).
__global__ void __launch_bounds__(256)
    k_slice64(const double *__restrict__ t64, const float *__restrict__ t32, const unsigned char *__restrict__ cls,
              const int4 *__restrict__ jobs, int nb, const int *__restrict__ exps, uint16_t *__restrict__ digits,
              const int *st) {
  if (failed(st)) return;
  __shared__ double blk[32][33];
  int4 jb = jobs[blockIdx.y];
  size_t base = (size_t)jb.x * nb * nb;
  bool f64 = cls[jb.x] == EMU_CLASS_FP64;
  int nbb = nb / 32;
  int r0 = (blockIdx.x % nbb) * 32, c0 = (blockIdx.x / nbb) * 32;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int c = w; c < 32; c += 8) {
    size_t o = base + (r0 + lane) + (size_t)(c0 + c) * nb;
    blk[lane][c] = f64 ? t64[o] : (double)t32[o];
  }
  __syncthreads();
  size_t plane = (size_t)nb * nb;
  write_block_digits(blk, [&](int rr) { return exp_of(exps, (long)jb.z + r0 + rr); },
                     digits + (size_t)jb.y * NS * plane + (size_t)r0 * nb + c0, nb, plane);
}

// Row exponents of a dense column-major block X[0:nrows, col0:col0+ncols]
// (the residuals of the empirical covariance): one CTA per (32 rows, column
// stripe), lane = row, warps stride columns; exps[r] = max(exps[r], e) with
// every |x| < 2^e.
__global__ void __launch_bounds__(256)
    k_rowexp_dense(const double *__restrict__ X, long ld, int nrows, long col0, long ncols, int *__restrict__ exps,
                   const int *st) {
  if (failed(st)) return;
  __shared__ unsigned long long red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane;
  unsigned long long m = 0;
  if (r < nrows)
    for (long c = (long)blockIdx.y * 8 + w; c < ncols; c += 8L * gridDim.y) m = max(m, mag_bits(X[r + (col0 + c) * ld]));
  red[w][lane] = m;
  __syncthreads();
  if (w == 0 && r < nrows) {
    for (int q = 1; q < 8; q++) m = max(m, red[q][lane]);
    if (m > 0) atomicMax(&exps[r], biased_exp(m));
  }
}

// Digit planes of that block, K-major: plane p, row r (< npad), column c
// (< kpad); rows >= nrows and columns >= ncols are zero.  One CTA per 32x32
// block, transposed through shared memory.
__global__ void __launch_bounds__(256)
    k_slice_dense(const double *__restrict__ X, long ld, int nrows, long col0, long ncols, int npad, long kpad,
                  const int *__restrict__ exps, uint16_t *__restrict__ digits, const int *st) {
  if (failed(st)) return;
  __shared__ double blk[32][33];
  const long c0 = (long)blockIdx.x * 32;
  const int r0 = blockIdx.y * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int cc = w; cc < 32; cc += 8) {
    const int r = r0 + lane;
    const long c = c0 + cc;
    blk[lane][cc] = (r < nrows && c < ncols) ? X[r + (col0 + c) * ld] : 0.0;
  }
  __syncthreads();
  write_block_digits(blk, [&](int rr) { return exp_of(exps, r0 + rr); }, digits + (size_t)r0 * kpad + c0, kpad,
                     (size_t)npad * kpad);
}

// Digits of Z columns per matrix block: one CTA per (sample c < s_pad, block).
// The exponent covers the block's rows of column c; samples c >= s are zero.
// Blocks begin and end at multiples of the tile size: a thread takes two rows,
// one 4-byte store per digit.  16384 x 1024: 145 -> 110 us (read twice, once
// from L2, and eight digits written: 402 MB).
__global__ void __launch_bounds__(256)
    k_slicez64(const double *__restrict__ Z, long ldz, int s, int s_pad, const int2 *__restrict__ blocks, long zcols,
               int2 whole, int *__restrict__ exps, uint16_t *__restrict__ digits, const int *st) {
  if (failed(st)) return;
  __shared__ unsigned long long red[8];
  __shared__ int s_e;
  int c = blockIdx.x, b = blockIdx.y;
  int2 blk = blocks ? blocks[b] : whole;
  const double *z = Z + blk.x + (size_t)c * ldz;
  unsigned long long m = 0;
  if (c < s) {
#pragma unroll 4
    for (int r = threadIdx.x; r < blk.y; r += 256) m = max(m, mag_bits(z[r]));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (int)(blockDim.x >> 5); q++) m = max(m, red[q]);
    const int eb = m > 0 ? biased_exp(m) : kExpBias;
    s_e = max(eb - kExpBias, kExpMin);
    exps[(long)b * s_pad + c] = eb;
  }
  __syncthreads();
  const int e = s_e;
  size_t plane = (size_t)s_pad * zcols;
  uint16_t *d = digits + (size_t)c * zcols + blk.x;
#pragma unroll 2
  for (int r = 2 * threadIdx.x; r < blk.y; r += 512)
    write_digits2(c < s ? z[r] : 0.0, c < s ? z[r + 1] : 0.0, e, d + r, plane);
}

// ------------------------------------------------------- blocked TRSM
constexpr int NQ = TW / 32;  // 32-column quarters of a block
static_assert(TW % 32 == 0 && TW % BN == 0, "block width");

// Row exponent (as the readers clamp it) and digits of one row of a
// TW-column block held NQ values per lane (columns lane + 32 q): the exponent
// is written to *e_out by lane 0 (0 for a row of zeros), plane p of column c
// at d[c + p plane].
__device__ inline void row_digits_tw(const double (&x)[NQ], int *e_out, uint16_t *d, size_t plane) {
  const int lane = threadIdx.x & 31;
  unsigned long long m = 0;
#pragma unroll
  for (int q = 0; q < NQ; q++) m = max(m, mag_bits(x[q]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int eb = m > 0 ? biased_exp(m) : 0;
  if (lane == 0) *e_out = eb;
  const int e = max(eb - kExpBias, kExpMin);
#pragma unroll
  for (int q = 0; q < NQ; q++) write_digits(x[q], e, d + 32 * q + lane, plane);
}

// Digits of L_kk's column blocks: one CTA per (32 rows, block J), warp w
// rows 4w..4w+3 of the 32, lane = columns lane + 32 q of the block.
__global__ void __launch_bounds__(256)
    k_lkk_digits(const double *__restrict__ L, int nb, int *__restrict__ exps, uint16_t *__restrict__ digits,
                 const int *st) {
  if (failed(st)) return;
  const int J = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c0 = J * TW;
  for (int i = 0; i < 4; i++) {
    const int r = blockIdx.x * 32 + w * 4 + i;
    if (r < (J + 1) * TW) continue;  // warp-uniform: rows no product reads
    double x[NQ];
#pragma unroll
    for (int q = 0; q < NQ; q++) x[q] = L[(size_t)r + (size_t)(c0 + 32 * q + lane) * nb];
    row_digits_tw(x, exps + (size_t)J * nb + r, digits + ((size_t)J * NS * nb + r) * TW, (size_t)nb * TW);
  }
}

// Column block J of X = A L_kk^{-T} for every listed tile, in place: the
// earlier blocks' contributions have been subtracted (digit products), so
// only L_kk's TW x TW diagonal block enters.  One CTA per (4 rows, tile),
// warp = row, lane = column of each 32-column quarter q: the earlier
// quarters' contribution is subtracted (L_kk's entries read from L2, a
// warp's 32 rows of one column at a time), then forward substitution against
// the pre-scaled diagonal 32 x 32 block.
__global__ void __launch_bounds__(128)
    k_trsm64_block(double *__restrict__ t64, int nb, const int *__restrict__ tiles, const double *__restrict__ Lkk,
                   int J, const double *__restrict__ Ls, const double *__restrict__ rinvs, int slot0,
                   int *__restrict__ exps, uint16_t *__restrict__ digits, const int *st) {
  if (failed(st)) return;
  const int z = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c0 = J * TW, r = blockIdx.x * 4 + w;
  double *X = t64 + (size_t)tiles[z] * nb * nb + r;
  double a[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) a[q] = X[(size_t)(c0 + 32 * q + lane) * nb];
#pragma unroll
  for (int q = 0; q < NQ; q++) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int qq = 0; qq < q; qq++) {
      const double *lq = Lkk + (size_t)(c0 + 32 * q + lane) + (size_t)(c0 + 32 * qq) * nb;
#pragma unroll 8
      for (int p = 0; p < 32; p += 2) {
        s0 = fma(__shfl_sync(0xffffffffu, a[qq], p), __ldg(lq + (size_t)p * nb), s0);
        s1 = fma(__shfl_sync(0xffffffffu, a[qq], p + 1), __ldg(lq + (size_t)(p + 1) * nb), s1);
      }
    }
    // Ls(p, l) = L(l, p) / L(p, p): a_l -= a_p Ls(p, l) on the unscaled a_p
    const int cb = J * NQ + q;
    double v = a[q] - (s0 + s1);
    double ld[32];
#pragma unroll
    for (int p = 0; p < 32; p++) ld[p] = (p < lane) ? Ls[(size_t)(cb * 32 + p) * 32 + lane] : 0.0;
#pragma unroll
    for (int j = 0; j < 32; j++) {
      const double vj = __shfl_sync(0xffffffffu, v, j);
      if (lane > j) v = fma(-vj, ld[j], v);
    }
    a[q] = v * rinvs[cb * 32 + lane];
  }
#pragma unroll
  for (int q = 0; q < NQ; q++) X[(size_t)(c0 + 32 * q + lane) * nb] = a[q];
  if (digits) {
    const size_t slot = (size_t)slot0 + z;
    row_digits_tw(a, exps + slot * nb + r, digits + (slot * NS * nb + r) * TW, (size_t)nb * TW);
  }
}

// Digits of whole rows of a packed FP64 matrix (launch_panel_digits): one CTA
// per PR rows, over the tile columns [tcol0, tcol0 + tcols) (tcols < 0: up to
// the row's tile): the rows' maxima in one pass, then the digits in a second
// one whose reads hit L2.  One launch where a memset, a maximum pass over all
// tiles and a slicing pass took three.
constexpr int PR = 32;
__global__ void __launch_bounds__(256)
    k_panel_digits(const double *__restrict__ t64, int NT, int nb, int row0, int tcol0, int tcols, int e_row0,
                   int *__restrict__ exps, int d_row0, long plane, long kpad, uint16_t *__restrict__ digits,
                   const int *st) {
  if (failed(st)) return;
  __shared__ double blk[32][33];
  __shared__ unsigned long long red[8][33];
  __shared__ int se[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = row0 + blockIdx.x * PR, ti = r0 / nb, rin = r0 % nb;
  const int t1 = tcols < 0 ? ti + 1 : tcol0 + tcols;
  const size_t te = (size_t)nb * nb;
  unsigned long long m = 0;
  for (int tj = tcol0; tj < t1; tj++) {
    const double *T = t64 + (size_t)tile_index(ti, tj, NT) * te + rin + lane;
#pragma unroll 4
    for (int c = w; c < nb; c += 8) m = max(m, mag_bits(T[(size_t)c * nb]));
  }
  red[w][lane] = m;
  __syncthreads();
  if (w == 0) {
    for (int q = 1; q < 8; q++) m = max(m, red[q][lane]);
    const int eb = m > 0 ? biased_exp(m) : 0;
    exps[r0 + lane - e_row0] = eb;
    se[lane] = max(eb - kExpBias, kExpMin);
  }
  for (int tj = tcol0; tj < t1; tj++) {
    const double *T = t64 + (size_t)tile_index(ti, tj, NT) * te + rin + lane;
    for (int c0 = 0; c0 < nb; c0 += 32) {
      double v[4];
#pragma unroll
      for (int q = 0; q < 4; q++) v[q] = T[(size_t)(c0 + w + 8 * q) * nb];
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 4; q++) blk[lane][w + 8 * q] = v[q];
      __syncthreads();
      write_block_digits(blk, [&](int rr) { return se[rr]; },
                         digits + (size_t)(r0 - d_row0) * kpad + (long)(tj - tcol0) * nb + c0, kpad,
                         (size_t)plane * kpad);
    }
  }
}

// The same for one tile column and nb <= kPanelCols: eight rows per CTA, read
// once into shared memory (32-row CTAs of the two-pass kernel took 27 us for
// one 512-wide tile, 16 CTAs).
constexpr int kPanelCols = 2048, P8 = 8;
__global__ void __launch_bounds__(256)
    k_panel_digits8(const double *__restrict__ t64, int NT, int nb, int row0, int tj, int *__restrict__ exps,
                    long plane, uint16_t *__restrict__ digits, const int *st) {
  if (failed(st)) return;
  extern __shared__ double pv[];  // [8][nb + 2]
  __shared__ unsigned long long red[8][P8 + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, ld = nb + 2;
  const int r0 = row0 + blockIdx.x * P8, ti = r0 / nb, rin = r0 % nb;
  // a warp reads four columns of the eight rows (64 bytes each) at a time
  const int rr = lane & 7, cc = w * 4 + (lane >> 3);
  const double *T = t64 + (size_t)tile_index(ti, tj, NT) * nb * nb + rin + rr;
  unsigned long long m = 0;
#pragma unroll 8
  for (int c = cc; c < nb; c += 32) {
    const double x = T[(size_t)c * nb];
    m = max(m, mag_bits(x));
    pv[rr * ld + c] = x;
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane < P8) red[w][lane] = m;
  __syncthreads();
  // warp w: row w
  unsigned long long mr = red[lane & 7][w];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) mr = max(mr, __shfl_xor_sync(0xffffffffu, mr, o));
  const int eb = mr > 0 ? biased_exp(mr) : 0, e = max(eb - kExpBias, kExpMin);
  if (lane == 0) exps[r0 + w] = eb;
  uint16_t *d = digits + (size_t)(r0 + w) * nb;
  for (int c = 2 * lane; c < nb; c += 64) write_digits2(pv[w * ld + c], pv[w * ld + c + 1], e, d + c, (size_t)plane * nb);
}

// ------------------------------------------------------------- GEMM
// Items of a region in groups of RG_W column blocks: in a group the row
// blocks run in order and each meets the group's columns, so that the items
// in flight on the chip share their operands' rows in L2 (152 CTAs cover about
// 19 row blocks by 8 column blocks).
constexpr int RG_W = 8;
struct Work {
  long out_off;
  int x;  // K offset in both arenas
  int a_sc, b_sc, rows_valid, cols_valid;
  int a_row, b_row;
  int total;  // K stages (0: nothing to do)
  int m, row0, col0;  // batched and dense sources
};
// First row block of column group g.
template <int SRC>
__host__ __device__ inline int group_row0(const Region &rg, int g) {
  if (SRC != SRC_SYRK) return rg.r_lo;
  const int d = (rg.c_lo + g * RG_W) * BN / BM;  // the diagonal's row block
  return d > rg.r_lo ? d : rg.r_lo;
}
template <int SRC>
__host__ __device__ inline int group_items(const Region &rg, int g) {
  const int c = rg.c_lo + g * RG_W, w = rg.c_hi - c < RG_W ? rg.c_hi - c : RG_W;
  const int h = rg.r_hi - group_row0<SRC>(rg, g);
  return h > 0 ? w * h : 0;
}
template <int SRC>
__host__ __device__ inline int region_items(const Region &rg) {
  int n = 0;
  for (int g = 0; rg.c_lo + g * RG_W < rg.c_hi; g++) n += group_items<SRC>(rg, g);
  return n;
}
struct Cursor {  // the group of the last item found; items come in ascending order
  int g = 0, base = 0;
};
// Items of the batched and dense sources.
template <int SRC>
__host__ __device__ inline int batch_items(const Region &rg) {
  const int rb = ((SRC == SRC_DENSE ? rg.rows_valid : 2 * rg.T) + BM - 1) / BM;
  if (SRC == SRC_DENSE) return rb * ((rg.cols_valid + BN - 1) / BN);
  return rg.L * rb * (((SRC == SRC_SYN ? rg.ntheta : rg.L) + BN - 1) / BN);
}
template <int SRC>
__device__ inline Work batch_work(const Region &rg, int it) {
  const int rb = ((SRC == SRC_DENSE ? rg.rows_valid : 2 * rg.T) + BM - 1) / BM;
  const int cb = ((SRC == SRC_DENSE ? rg.cols_valid : SRC == SRC_SYN ? rg.ntheta : rg.L) + BN - 1) / BN;
  const int C = it % cb, R = it / cb % rb, m = it / cb / rb;
  Work w;
  w.out_off = 0;
  w.x = 0;
  w.a_row = w.a_sc = R * BM;
  w.b_row = w.b_sc = C * BN;
  w.m = m;
  w.row0 = R * BM;
  w.col0 = C * BN;
  if (SRC == SRC_DENSE) {
    w.total = rg.nk / BK;
    w.rows_valid = rg.rows_valid - R * BM;
    w.cols_valid = rg.cols_valid - C * BN;
  } else if (SRC == SRC_SYN) {
    w.total = order_k(rg.L, m) / BK;
    w.x = order_koff(rg.L, m);
    w.a_sc += m * rg.rpad;
    w.b_sc += m * rg.cpad;
    w.rows_valid = 2 * rg.T - R * BM;
    w.cols_valid = rg.ntheta - C * BN;
  } else {
    w.total = rg.nk / BK;
    w.a_row = w.a_sc = m * rg.rpad + R * BM;
    w.b_row = w.b_sc = order_pos(rg.L, m) + C * BN;
    w.rows_valid = 2 * rg.T - R * BM;
    w.cols_valid = rg.L - m - C * BN;
    if (w.cols_valid <= 0) w.total = 0;
  }
  return w;
}
// Output offset of row `row` of an item's block, and of column cx.
template <int SRC>
__device__ inline long batch_row(const Region &rg, const Work &w, int row, long ldo) {
  const int r = w.row0 + row;
  if (SRC == SRC_DENSE) return (long)(r / rg.div) * rg.ld2 + r % rg.div + (long)w.col0 * ldo;
  const int s = r / rg.T, t = r - s * rg.T;
  if (SRC == SRC_SYN) return t + (long)rg.T * (w.col0 + (long)rg.ntheta * (2 * w.m + s));
  return t * ldo;
}

template <int SRC>
__device__ inline Work region_work(const Region &rg, Cursor &cur, int it, long ldo) {
  if constexpr (SRC >= SRC_DENSE) return batch_work<SRC>(rg, it);
  int cnt;
  while (it >= cur.base + (cnt = group_items<SRC>(rg, cur.g))) {
    cur.base += cnt;
    cur.g++;
  }
  const int q = it - cur.base, c0 = rg.c_lo + cur.g * RG_W, wd = min(RG_W, rg.c_hi - c0);
  const int R = group_row0<SRC>(rg, cur.g) + q / wd, C = c0 + q % wd;
  const int row = R * BM, col = C * BN, nb = rg.nb;
  Work w;
  w.rows_valid = BM;
  w.cols_valid = BN;
  w.total = nb / BK;
  w.x = 0;
  if (SRC == SRC_SYRK) {
    if (row + BM - 1 < col) w.total = 0;  // above the diagonal
    w.out_off = tile_index(row / nb, col / nb, rg.NT) * (long)nb * nb + row % nb + (long)(col % nb) * nb;
    w.a_row = w.a_sc = row;
    w.b_row = w.b_sc = col;
  } else if (SRC == SRC_TRSM) {
    const int z = row / nb, rin = row % nb, slot = rg.slot0 + z;
    w.total = TW / BK;
    w.out_off = (long)rg.tiles[z] * nb * nb + rin + (long)col * nb;
    w.a_row = slot * NS * nb + rin;
    w.a_sc = slot * nb + rin;
    w.b_row = rg.J * NS * nb + col;
    w.b_sc = rg.J * nb + col;
  } else {
    w.total = (row / nb + 1) * nb / BK;
    w.out_off = row + (long)col * ldo;
    w.a_row = w.a_sc = row - rg.a_row0;
    w.b_row = w.b_sc = col;
    w.rows_valid = min(BM, rg.rows_valid - row);
    w.cols_valid = min(BN, rg.cols_valid - col);
  }
  return w;
}

template <int MODE, int SRC>
__global__ void __maxnreg__(96)
    k_tc_gemm64(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
                const Item *__restrict__ items, int nitems, const Seg *__restrict__ segs, int nb, int a_plane,
                int b_plane, const int *__restrict__ a_exp, const int *__restrict__ b_exp,
                double *__restrict__ out, long ldo, int *status, const Region rg) {
  extern __shared__ uint8_t smem_raw[];
  uint32_t raw_addr = tc::smem_u32(smem_raw);
  uint32_t pad = ((raw_addr + 1023u) & ~1023u) - raw_addr;
  uint8_t *ring = smem_raw + pad;
  Shared *sh = reinterpret_cast<Shared *>(ring + RING_BYTES);
  const uint32_t ring_addr = raw_addr + pad;
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kstages = nb / BK;  // stages per segment

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      tc::mbar_init(&sh->full[s], 1);
      tc::mbar_init(&sh->empty[s], 1);
    }
    tc::mbar_init(&sh->tfull, 1);
    tc::mbar_init(&sh->tempty, EPI_THREADS);
    tc::mbar_init(&sh->done, 1);
    // one reading of the status word for all roles: an earlier failure skips the work
    sh->abort = failed(status) ? 1 : 0;
    tc::fence_barrier_init();
    tc::tma_prefetch_desc(&amap);
    tc::tma_prefetch_desc(&bmap);
  }
  if (warp == 1) {
    tc::tmem_alloc(&sh->tmem_base, TMEM_COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = sh->tmem_base;
  volatile int *abort = &sh->abort;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = *abort == 0;
      Cursor cur;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        int sg0 = 0, sg1 = 1, kst = kstages;
        Seg sd;
        if constexpr (SRC == SRC_LIST) {
          sg0 = items[it].seg_begin;
          sg1 = items[it].seg_end;
        } else {
          const Work wk = region_work<SRC>(rg, cur, it, ldo);
          kst = wk.total;
          sd.a_row = wk.a_row;
          sd.b_row = wk.b_row;
          sd.a_x = sd.b_x = wk.x;
        }
        for (int sg = sg0; sg < sg1 && ok; sg++) {
          if constexpr (SRC == SRC_LIST) sd = segs[sg];
          for (int kc = 0; kc < kst; kc++) {
            if (!tc::mbar_wait(&sh->empty[stage], phase ^ 1u, abort)) {
              raise_timeout(sh, status);
              ok = false;
              break;
            }
            tc::mbar_arrive_expect_tx(&sh->full[stage], (uint32_t)STAGE_BYTES);
            uint8_t *st = ring + stage * STAGE_BYTES;
            for (int p = 0; p < NS; p++)
              tc::tma_load_2d(st + p * A_SL, &amap, &sh->full[stage], sd.a_x + kc * BK, sd.a_row + p * a_plane);
            for (int q = 0; q < NS; q++)
              tc::tma_load_2d(st + NS * A_SL + q * B_SL, &bmap, &sh->full[stage], sd.b_x + kc * BK,
                              sd.b_row + q * b_plane);
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      // every stage's last load must have landed before the CTA exits
      for (int s = 0; s < STAGES; s++) {
        uint32_t par = (s < stage) ? phase : (phase ^ 1u);
        tc::mbar_wait_inflight(&sh->full[s], par);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t chunk = 0;
      uint32_t started = 0;
      bool ok = *abort == 0;
      Cursor cur;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        int total;  // K stages of the item
        if constexpr (SRC == SRC_LIST)
          total = (items[it].seg_end - items[it].seg_begin) * kstages;
        else
          total = region_work<SRC>(rg, cur, it, ldo).total;
        for (int ks_i = 0; ks_i < total && ok; ks_i++) {
          if (ks_i % CHUNK_STAGES == 0) {
            // the epilogue has read the previous chunk's accumulators
            if (!tc::mbar_wait(&sh->tempty, (chunk & 1u) ^ 1u, abort)) {
              raise_timeout(sh, status);
              ok = false;
              break;
            }
            tc::fence_after_sync();
            started = 0;
          }
          if (!tc::mbar_wait(&sh->full[stage], phase, abort)) {
            raise_timeout(sh, status);
            ok = false;
            break;
          }
          tc::fence_after_sync();
          uint32_t st = ring_addr + stage * STAGE_BYTES;
          const uint64_t a0 = tc::smem_desc(st, 16, 512, tc::kSwizzle64B);
          const uint64_t b0 = tc::smem_desc(st + NS * A_SL, 16, 512, tc::kSwizzle64B);
#pragma unroll
          for (int ks = 0; ks < BK / 16; ks++) {
#pragma unroll
            for (int p = 0; p < NS; p++) {
              const uint64_t ad = tc::desc_add(a0, p * A_SL + ks * 32);
              // digits q .. q + nq - 1 of B: groups p + q .. p + q + nq - 1
#pragma unroll
              for (int q = 0; q < NS - p; q += QMERGE) {
                const int nq = NS - p - q < QMERGE ? NS - p - q : QMERGE;
                const uint64_t bd = tc::desc_add(b0, q * B_SL + ks * 32);
                tc::mma_f16(tmem + (uint32_t)((p + q) * BN), ad, bd, tc::idesc_f32acc(1u /*BF16*/, BM, nq * BN),
                            p > 0 ? 1u : started);
              }
              started = 1u;  // digit 0 of A has written every group
            }
          }
          tc::mma_commit(&sh->empty[stage]);
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
          if (ks_i % CHUNK_STAGES == CHUNK_STAGES - 1 || ks_i == total - 1) {
            tc::mma_commit(&sh->tfull);
            chunk++;
          }
        }
      }
      tc::mma_commit(&sh->done);
      tc::mbar_wait_inflight(&sh->done, 0);
    }
  } else if (warp >= EPI_WARP0) {
    // ------------------------------------------------------------ epilogue
    // TMEM lane quarter warp % 4 (the lanes a warp may access), columns
    // [col0, col0 + EC) of the block
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const int col0 = ((warp - EPI_WARP0) >> 2) * EC;
    const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col0;
    uint32_t chunk = 0;
    bool ok = *abort == 0;
    Cursor cur;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
      Work item;
      if constexpr (SRC == SRC_LIST) {
        const Item li = items[it];
        item.out_off = li.out_off;
        item.a_sc = li.a_sc;
        item.b_sc = li.b_sc;
        item.rows_valid = li.rows_valid;
        item.cols_valid = li.cols_valid;
        item.total = (li.seg_end - li.seg_begin) * kstages;
      } else {
        item = region_work<SRC>(rg, cur, it, ldo);
        if (item.total == 0) continue;  // every role skips it
      }
      const int total = item.total;
      const int nchunks = (total + CHUNK_STAGES - 1) / CHUNK_STAGES;
      constexpr bool kWhole = MODE == TC64_SUB;  // every row and column exists
      double *o = out + item.out_off;
      if constexpr (SRC >= SRC_DENSE)
        o += batch_row<SRC>(rg, item, row, ldo);
      else
        o += row;
      if constexpr (kWhole) {
        // the warp's 32 rows x EC columns (two 128-byte lines per column) on
        // their way to L2 while the MMAs run
        const double *pf = o - lane + (long)(col0 + (lane >> 1)) * ldo + (lane & 1) * 16;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pf));
      }
      long long hi[EC];
      unsigned lo[EC];
#pragma unroll
      for (int x = 0; x < EC; x++) {
        hi[x] = 0;
        lo[x] = 0u;
      }
      for (int c = 0; c < nchunks; c++) {
        if (!tc::mbar_wait(&sh->tfull, chunk & 1u, abort)) {
          raise_timeout(sh, status);
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll
        for (int h = 0; h < EC / 2; h++) {
          uint32_t r[NS][2];
#pragma unroll
          for (int g = 0; g < NS; g++) tc::tmem_ld_32x32b_x2(tlane + (uint32_t)(g * BN + h * 2), r[g]);
          tc::tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 2; x++) fold_groups(r, x, hi[h * 2 + x], lo[h * 2 + x]);
        }
        tc::fence_before_sync();
        tc::mbar_arrive(&sh->tempty);
        chunk++;
      }
      if (!ok) break;
      // scales 2^(e_row + e_col), exact; then the output block
      const int ea = exp_of(a_exp, (long)item.a_sc + row);
      // in groups of 8 columns: 8 loads in flight, then 8 stores
      if (kWhole || row < item.rows_valid) {
#pragma unroll
        for (int x0 = 0; x0 < EC; x0 += 8) {
          double cv[8];
#pragma unroll
          for (int x = 0; x < 8; x++) {
            const int cx = col0 + x0 + x;
            if constexpr (MODE == TC64_SET)
              cv[x] = 0.0;
            else
              cv[x] = (kWhole || cx < item.cols_valid) ? __ldcg(o + (long)cx * ldo) : 0.0;
          }
#pragma unroll
          for (int x = 0; x < 8; x++) {
            const int cx = col0 + x0 + x;
            // columns past the last hold whatever the arena held: exponents there
            // can send fixed_scaled to its slow form (a third of the columns of
            // 129 rings, 40 of 135 us of the synthesis' products)
            if (!kWhole && cx >= item.cols_valid) continue;
            const double v = fixed_scaled(hi[x0 + x], lo[x0 + x], ea + exp_of(b_exp, (long)item.b_sc + cx));
            if (MODE == TC64_SUB)
              __stcg(o + (long)cx * ldo, cv[x] - v);
            else {
              if constexpr (SRC == SRC_ANA) {
                // order +-m, degree l = m + column; the sine sums of order 0 have no coefficient
                const long l = item.m + item.col0 + cx;
                const bool neg = item.row0 + row >= rg.T;
                if (!neg || item.m > 0) __stcg(o + l * l + l + (neg ? -item.m : item.m), v);
              } else {
                __stcg(o + (long)cx * ldo, MODE == TC64_SET ? v : cv[x] + v);
              }
            }
          }
        }
      }
    }
  }

  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace

emu_status make_map(emu_ctx *ctx, CUtensorMap *map, const void *base, uint64_t inner, uint64_t rows,
                    uint32_t box_rows) {
  return gemm_tc::make_map_bf16(ctx, map, base, inner, rows, box_rows);
}

emu_status launch_row_exponents(emu_ctx *ctx, const double *t64, const float *t32, const unsigned char *cls,
                                const int4 *d_jobs, int njobs, int nb, int *exps) {
  if (njobs <= 0) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, 8.0 * njobs * (double)nb * nb);
  k_rowexp64<<<dim3(nb / 32, njobs, 8), 256, 0, ctx->stream>>>(t64, t32, cls, d_jobs, nb, exps, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_slice(emu_ctx *ctx, const double *t64, const float *t32, const unsigned char *cls,
                        const int4 *d_jobs, int njobs, int nb, const int *exps, uint16_t *digits) {
  if (njobs <= 0) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (8.0 + 2.0 * NS) * njobs * (double)nb * nb);
  k_slice64<<<dim3((nb / 32) * (nb / 32), njobs), 256, 0, ctx->stream>>>(t64, t32, cls, d_jobs, nb, exps, digits,
                                                                         ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_slice_z(emu_ctx *ctx, const double *Z, long ldz, int s, int s_pad, const int2 *d_blocks,
                          int nblocks, long zcols, int *exps, uint16_t *digits) {
  if (nblocks <= 0 || s_pad <= 0) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (8.0 + 2.0 * NS) * (double)s_pad * zcols);
  k_slicez64<<<dim3(s_pad, nblocks), 256, 0, ctx->stream>>>(Z, ldz, s, s_pad, d_blocks, zcols, int2{0, 0}, exps,
                                                            digits, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_slice_cols(emu_ctx *ctx, const double *Z, long ldz, int s, int s_pad, int rows, int *exps,
                             uint16_t *digits) {
  if (s_pad <= 0 || rows <= 0) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (8.0 + 2.0 * NS) * (double)s_pad * rows);
  k_slicez64<<<s_pad, 256, 0, ctx->stream>>>(Z, ldz, s, s_pad, nullptr, rows, int2{0, rows}, exps, digits,
                                             ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_dense_digits(emu_ctx *ctx, const double *X, long ld, int nrows, long col0, long ncols, int npad,
                               long kpad, int *exps, uint16_t *digits) {
  if (npad % 32 != 0 || kpad % 32 != 0 || nrows > npad || ncols > kpad) return EMU_EINVAL;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (16.0 + 2.0 * NS) * (double)npad * kpad);
  EMU_CUDA_TRY(ctx, cudaMemsetAsync(exps, 0, (size_t)npad * sizeof(int), ctx->stream));
  const int ystripes = (int)std::min<long>(64, (ncols + 7) / 8);
  k_rowexp_dense<<<dim3(npad / 32, std::max(ystripes, 1)), 256, 0, ctx->stream>>>(X, ld, nrows, col0, ncols, exps,
                                                                                  ctx->d_status);
  EMU_LAUNCHED(ctx);
  k_slice_dense<<<dim3((unsigned)(kpad / 32), npad / 32), 256, 0, ctx->stream>>>(X, ld, nrows, col0, ncols, npad,
                                                                                 kpad, exps, digits, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_lkk_digits(emu_ctx *ctx, const double *Lkk, int nb, int *exps, uint16_t *digits) {
  if (nb % BM != 0) return EMU_EINVAL;
  const int nJ = nb / TW;
  if (nJ < 2) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (8.0 + 2.0 * NS) * (double)nb * TW * (nJ - 1));
  k_lkk_digits<<<dim3(nb / 32, nJ - 1), 256, 0, ctx->stream>>>(Lkk, nb, exps, digits, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_trsm_block(emu_ctx *ctx, double *t64, int nb, const int *d_tiles, int ntiles, const double *Lkk,
                             int J, const double *Ls, const double *rinvs, int slot0, int *exps, uint16_t *digits) {
  if (nb % TW != 0 || J < 0 || J >= nb / TW) return EMU_EINVAL;
  if (ntiles <= 0) return EMU_OK;
  k_trsm64_block<<<dim3(nb / 4, ntiles), 128, 0, ctx->stream>>>(t64, nb, d_tiles, Lkk, J, Ls, rinvs, slot0, exps,
                                                                digits, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

template <int MODE, int SRC>
static emu_status launch_kernel(emu_ctx *ctx, int grid, const CUtensorMap &a, const CUtensorMap &b,
                                const Item *d_items, int nitems, const Seg *d_segs, int nb, int a_plane, int b_plane,
                                const int *a_exp, const int *b_exp, double *out, long ldo, const Region &rg) {
  static std::atomic<uint64_t> attr{0};
  EMU_CUDA_TRY(ctx, smem_limit_once(attr, ctx->device, (const void *)k_tc_gemm64<MODE, SRC>, SMEM_BYTES));
  k_tc_gemm64<MODE, SRC><<<grid, NTHREADS, SMEM_BYTES, ctx->stream>>>(a, b, d_items, nitems, d_segs, nb, a_plane,
                                                                      b_plane, a_exp, b_exp, out, ldo,
                                                                      ctx->d_status, rg);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch(emu_ctx *ctx, const CUtensorMap &a, const CUtensorMap &b, const Item *d_items, int nitems,
                  const Seg *d_segs, int nb, int a_plane, int b_plane, const int *a_exp, const int *b_exp, int mode,
                  double *out64, int ldo, int max_ctas) {
  if (nitems <= 0) return EMU_OK;
  if (nb % BK != 0) return EMU_EINVAL;
  int grid = nitems < max_ctas ? nitems : max_ctas;
  return mode == TC64_SUB ? launch_kernel<TC64_SUB, SRC_LIST>(ctx, grid, a, b, d_items, nitems, d_segs, nb, a_plane,
                                                              b_plane, a_exp, b_exp, out64, ldo, Region())
                          : launch_kernel<TC64_ADD, SRC_LIST>(ctx, grid, a, b, d_items, nitems, d_segs, nb, a_plane,
                                                              b_plane, a_exp, b_exp, out64, ldo, Region());
}

emu_status launch_region(emu_ctx *ctx, int src, const CUtensorMap &a, const CUtensorMap &b, const Region &rg,
                         int a_plane, int b_plane, const int *a_exp, const int *b_exp, double *out, long ldo,
                         int max_ctas) {
  if (src < SRC_DENSE && rg.nb % BM != 0) return EMU_EINVAL;
  const int n = src == SRC_SYRK    ? region_items<SRC_SYRK>(rg)
                : src == SRC_DENSE ? batch_items<SRC_DENSE>(rg)
                : src == SRC_SYN   ? batch_items<SRC_SYN>(rg)
                : src == SRC_ANA   ? batch_items<SRC_ANA>(rg)
                                   : region_items<SRC_TRMM>(rg);
  if (n <= 0) return EMU_OK;
  const int grid = std::max(1, std::min(n, max_ctas));
#define EMU_REGION(M, S) \
  launch_kernel<M, S>(ctx, grid, a, b, nullptr, n, nullptr, rg.nb, a_plane, b_plane, a_exp, b_exp, out, ldo, rg)
  if (src == SRC_SYRK) return EMU_REGION(TC64_SUB, SRC_SYRK);
  if (src == SRC_TRSM) return EMU_REGION(TC64_SUB, SRC_TRSM);
  if (src == SRC_TRMM) return EMU_REGION(TC64_SET, SRC_TRMM);
  if (src == SRC_DENSE) return EMU_REGION(TC64_SET, SRC_DENSE);
  if (src == SRC_SYN) return EMU_REGION(TC64_SET, SRC_SYN);
  return EMU_REGION(TC64_SET, SRC_ANA);
#undef EMU_REGION
}

// Parts of a TrsmPlan, in order; off[i] is part i's start, the last entry the size.
static void trsm_plan_parts(int nb, int slots, size_t (&off)[7]) {
  const size_t nJ = nb / TW, plane = (size_t)nb * TW;
  const size_t bytes[6] = {slots * nb * sizeof(int),
                           slots * NS * plane * sizeof(uint16_t),
                           nJ * nb * sizeof(int),
                           std::max<size_t>(nJ - 1, 1) * NS * plane * sizeof(uint16_t),
                           (size_t)nb * 32 * sizeof(double),
                           (size_t)nb * sizeof(double)};
  off[0] = 0;
  for (int i = 0; i < 6; i++) off[i + 1] = off[i] + ((bytes[i] + 255) & ~(size_t)255);
}
size_t trsm_plan_bytes(int nb, int slots) {
  size_t off[7];
  trsm_plan_parts(nb, slots, off);
  return off[6];
}
emu_status trsm_plan_init(emu_ctx *ctx, TrsmPlan *P, char *base, int nb, int slots) {
  if (nb % TW != 0 || nb % BM != 0) return EMU_EINVAL;
  size_t off[7];
  trsm_plan_parts(nb, slots, off);
  P->xexp = reinterpret_cast<int *>(base + off[0]);
  P->xdig = reinterpret_cast<uint16_t *>(base + off[1]);
  P->lexp = reinterpret_cast<int *>(base + off[2]);
  P->ldig = reinterpret_cast<uint16_t *>(base + off[3]);
  P->ls = reinterpret_cast<double *>(base + off[4]);
  P->rinv = reinterpret_cast<double *>(base + off[5]);
  emu_status s = make_map(ctx, &P->mx, P->xdig, TW, (uint64_t)slots * NS * nb, BM);
  return s == EMU_OK ? make_map(ctx, &P->ml, P->ldig, TW, std::max<uint64_t>(nb / TW - 1, 1) * NS * nb, BN) : s;
}
emu_status trsm_plan_prep(emu_ctx *ctx, const TrsmPlan &P, const double *Lkk, int nb) {
  emu_status s = launch_trsm64_prep(ctx, Lkk, nb, P.ls, P.rinv);
  return s == EMU_OK ? launch_lkk_digits(ctx, Lkk, nb, P.lexp, P.ldig) : s;
}
emu_status trsm_plan_solve(emu_ctx *ctx, const TrsmPlan &P, double *t64, int nb, const int *d_tiles, int n,
                           const double *Lkk, int slot0) {
  if (n <= 0) return EMU_OK;
  const int nJ = nb / TW;
  Region rg;
  rg.nb = nb;
  rg.r_hi = n * (nb / BM);
  rg.tiles = d_tiles;
  rg.slot0 = slot0;
  for (int J = 0; J < nJ; J++) {
    const bool last = J + 1 == nJ;
    emu_status s = launch_trsm_block(ctx, t64, nb, d_tiles, n, Lkk, J, P.ls, P.rinv, slot0, P.xexp,
                                     last ? nullptr : P.xdig);
    if (s != EMU_OK || last) return s;
    rg.J = J;
    rg.c_lo = (J + 1) * (TW / BN);
    rg.c_hi = nb / BN;
    if ((s = launch_region(ctx, SRC_TRSM, P.mx, P.ml, rg, nb, nb, P.xexp, P.lexp, t64, nb, ctx->sm_count)) != EMU_OK)
      return s;
  }
  return EMU_OK;
}

emu_status launch_panel_digits(emu_ctx *ctx, const double *t64, int NT, int nb, int row0, int nrows, int tcol0,
                               int tcols, int e_row0, int *exps, int d_row0, long plane, long kpad,
                               uint16_t *digits) {
  if (nb % PR != 0 || row0 % PR != 0 || nrows % PR != 0 || kpad % 2 != 0) return EMU_EINVAL;
  if (nrows <= 0) return EMU_OK;
  ProfScope ps(ctx, PROF_SPLIT, 0.0, (8.0 + 2.0 * NS) * nrows * (double)kpad);
  if (tcols == 1 && nb <= kPanelCols && e_row0 == 0 && d_row0 == 0 && kpad == nb) {
    static std::atomic<uint64_t> attr{0};
    const int sm = P8 * (nb + 2) * (int)sizeof(double);
    EMU_CUDA_TRY(ctx, smem_limit_once(attr, ctx->device, (const void *)k_panel_digits8,
                                      P8 * (kPanelCols + 2) * (int)sizeof(double)));
    k_panel_digits8<<<nrows / P8, 256, sm, ctx->stream>>>(t64, NT, nb, row0, tcol0, exps, plane, digits, ctx->d_status);
    EMU_LAUNCHED(ctx);
    return EMU_OK;
  }
  k_panel_digits<<<nrows / PR, 256, 0, ctx->stream>>>(t64, NT, nb, row0, tcol0, tcols, e_row0, exps, d_row0, plane,
                                                      kpad, digits, ctx->d_status);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

}  // namespace gemm64
