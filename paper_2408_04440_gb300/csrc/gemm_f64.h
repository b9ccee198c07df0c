// gemm_f64.h -- FP64-accurate tile update C -= A B^T on the BF16 tensor cores
// (gemm_f64.cu), for the FP64-class tiles of the mixed-precision factor.
//
// Ozaki scheme (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 2012), in fixed point: every row r of
// an operand tile is scaled by a power of two 2^-e_r so that its entries lie
// in (-1, 1), then written as NS digits of SLICE_BITS bits each,
//   x 2^-e_r = sum_p s_p 2^-(SLICE_BITS (p + 1)),   s_p integers, |s_p| <= 2^SLICE_BITS,
// every digit exact in BF16.  A product of two digits is an integer below
// 2^14; the sum of the (g + 1) products with p + q = g over K <= KCHUNK terms
// stays below 2^24, so the tensor cores accumulate each diagonal group g
// exactly in FP32.  Every KCHUNK the epilogue folds the groups, scaled by
// 2^-7(g+2), in integer arithmetic and adds them in FP64; it applies the row
// scales at the end.
// NS = 8 digits carry 57 bits, so the products with p + q < NS give the dot
// products to FP64 accuracy relative to the rows' largest entries.
#pragma once
#include <cuda.h>

#include "emu_internal.h"

namespace gemm64 {

constexpr int BM = 128;        // output rows of an item (TMEM lanes)
constexpr int BN = 64;         // output columns of an item; 8 groups x 64 = 512 TMEM columns
constexpr int BK = 32;         // K per pipeline stage
constexpr int STAGES = 2;
constexpr int NS = 8;          // digits per operand entry
constexpr int SLICE_BITS = 7;
// K accumulated exactly in FP32 between two drains of the group accumulators:
// |sum| <= 384 (2 * 128 * 64 + 6 * 64^2) = 15,728,640 < 2^24 (leading digits
// |d_0| <= 128, the others <= 64).  256 drained 1.5 times as often.
constexpr int KCHUNK = 384;

// One BM x BN output block: the sum over its segments of A_seg B_seg^T.
// Operand row r of digit plane p sits at arena row (row + p * plane); every
// entry of a row carries the scale 2^e of that row, read from an exponent
// array (A: a_exp[a_sc + r], B: b_exp[b_sc + c]), so all segments of an item
// share one scale per row and their digit products add exactly.
struct Seg {
  int a_row, b_row;  // arena rows of digit plane 0 of the A and B blocks
  int a_x, b_x;      // K offset of the segment in each arena
};
struct Item {
  long out_off;                // element offset of the block in the FP64 output
  int a_sc, b_sc;              // exponent indices of the block's first A row / B row
  int seg_begin, seg_end;      // segments [seg_begin, seg_end)
  int rows_valid, cols_valid;  // rows / columns of the block that exist (TC64_ADD)
};
// out -= A B^T (factor) / out += A B^T / out = A B^T (the last two bounded by rows_valid, cols_valid)
enum { TC64_SUB = 0, TC64_ADD = 1, TC64_SET = 2 };

// 2-D BF16 tensor map over a digit arena of `inner` columns, box rows x 32.
emu_status make_map(emu_ctx *ctx, CUtensorMap *map, const void *base, uint64_t inner, uint64_t rows,
                    uint32_t box_rows);

// Exponent arrays hold e + kExpBias, so that a zeroed array (cudaMemset 0)
// holds the lowest exponent; readers clamp e at kExpMin.  A row below 2^kExpMin
// loses nothing by that: the last digit's unit is then 2^-1080, below FP64's
// smallest number.  A row with an infinity or a NaN holds kExpPoison: its digits
// are zeros and every product with it is NaN, as in floating point.
constexpr int kExpBias = 1024;
constexpr int kExpMin = -kExpBias;
constexpr int kExpPoison = 1 << 20;

// Row exponents of listed tiles: jobs {tile, -, exponent base}; a tile is read
// from the FP64 arena when its class is FP64, else from the FP32 master.  Row
// r gets exp[base + r] = max(exp[base + r], e) with max_c |x_rc| < 2^e, so
// tiles that share rows share the largest exponent.
emu_status launch_row_exponents(emu_ctx *ctx, const double *t64, const float *t32, const unsigned char *cls,
                                const int4 *d_jobs, int njobs, int nb, int *exps);
// Digit planes of listed tiles: jobs {tile, slot, exponent base}; plane p of
// slot s at rows (s * NS + p) * nb of a digit arena with nb columns.
emu_status launch_slice(emu_ctx *ctx, const double *t64, const float *t32, const unsigned char *cls,
                        const int4 *d_jobs, int njobs, int nb, const int *exps, uint16_t *digits);
// Digits of the columns of Z (samples) for each matrix block of rows
// [row0, row0 + nrows): plane p, row c (sample), column = row of Z; one
// exponent per (block, sample): exps[blk * s_pad + c].  blocks = {row0, nrows}.
emu_status launch_slice_z(emu_ctx *ctx, const double *Z, long ldz, int s, int s_pad, const int2 *d_blocks,
                          int nblocks, long zcols, int *exps, uint16_t *digits);

// The same for one block of all `rows` rows (no block list).
emu_status launch_slice_cols(emu_ctx *ctx, const double *Z, long ldz, int s, int s_pad, int rows, int *exps,
                             uint16_t *digits);

// Row exponents and digit planes of a dense column-major FP64 block
// X[0:nrows, col0:col0+ncols] (leading dimension ld): exps[r] for r < npad
// (zeroed first), plane p of row r at digits + (p * npad + r) * kpad, K-major,
// zero beyond nrows / ncols.  npad and kpad are multiples of 32.
emu_status launch_dense_digits(emu_ctx *ctx, const double *X, long ld, int nrows, long col0, long ncols, int npad,
                               long kpad, int *exps, uint16_t *digits);

// Blocked FP64-class panel TRSM X = A L_kk^{-T} (gemm_f64.cu): column block J
// (TW columns) of every listed tile is solved on the FP64 pipe against the
// TW x TW diagonal block of L_kk (launch_trsm_block), then its contribution to
// the later blocks, X_J L_{>J,J}^T, is subtracted as digit products on the
// tensor cores (launch, K = TW, output blocks of BN columns), so the FP64 pipe
// runs TW/nb of the nb^3 flops of a tile in nb/TW solve launches.
constexpr int TW = 128;
// Digits of L_kk's column blocks J < nb/TW - 1, rows r >= (J+1) TW (the rows
// the products read): exps[J nb + r] (biased), plane p of row r at arena row
// (J NS + p) nb + r of an arena with TW columns.  nb a multiple of BM.
emu_status launch_lkk_digits(emu_ctx *ctx, const double *Lkk, int nb, int *exps, uint16_t *digits);
// Column block J of the tiles d_tiles[0..ntiles) of t64 solved in place; Ls /
// rinvs are L_kk's pre-scaled 32 x 32 diagonal blocks and pivot reciprocals
// (launch_trsm64_prep).  With digits (not null), the solved block's row
// exponents and digits for the products: tile z in slot s = slot0 + z,
// exps[s nb + r], plane p of row r at arena row (s NS + p) nb + r (TW columns).
emu_status launch_trsm_block(emu_ctx *ctx, double *t64, int nb, const int *d_tiles, int ntiles, const double *Lkk,
                             int J, const double *Ls, const double *rinvs, int slot0, int *exps, uint16_t *digits);

// Implicit item sets: the items of one step of the plain FP64 factor, of the
// blocked FP64-class TRSM and of the sampler, found from the item number by
// every role of the kernel, so that no item lists are built, copied or read
// (n = 160000 would need 5 GB of them).  Rows are counted in blocks of BM,
// columns in blocks of BN (nb a multiple of BM).
struct Region {
  int NT = 0, nb = 0;
  int J = 0;                 // column block of L_kk (TRSM)
  int r_lo = 0, r_hi = 0;    // row blocks [r_lo, r_hi) (of the padded matrix; TRSM: of the listed tiles)
  int c_lo = 0, c_hi = 0;    // column blocks [c_lo, c_hi) (of the padded matrix; TRSM: of the tile)
  const int *tiles = nullptr;  // TRSM: tile indices; tile z has slot slot0 + z
  int slot0 = 0;
  int a_row0 = 0;            // TRMM: matrix row held by arena row 0 of A
  int rows_valid = 0, cols_valid = 0;  // TRMM, DENSE: rows / columns of the output that exist
  int nk = 0;                // DENSE, ANA: K (a multiple of BK)
  int div = 0;               // DENSE
  long ld2 = 0;              // DENSE
  int L = 0, T = 0, ntheta = 0;  // SYN, ANA
  int rpad = 0, cpad = 0;    // SYN, ANA: rows of A per order (SYN: exponents only), SYN: rows of B
};
// SYN operands: the orders run in blocks of 32 from m0; order m's K holds the
// degrees m0 .. L-1 (zero below m), order_k(L, m) of them (a multiple of 32),
// from K offset order_koff(L, m).
__host__ __device__ inline int order_k(int L, int m) { return (L + 31) / 32 * 32 - m / 32 * 32; }
__host__ __device__ inline int order_koff(int L, int m) {
  const int Lp = (L + 31) / 32 * 32, b = m / 32;
  return 32 * (b * Lp - 16 * b * (b - 1)) + (m % 32) * (Lp - 32 * b);
}
// ANA operands: the (m, l) pairs of even orders, then from order_odd0(L) on
// those of odd orders (the two parities are formed by different products, in
// blocks of BM rows); order m's pairs start at order_pos(L, m), l = m first.
__host__ __device__ inline int order_odd0(int L) {
  const int a = (L + 1) / 2;
  return (a * L - a * (a - 1) + 127) / 128 * 128;
}
__host__ __device__ inline int order_pos(int L, int m) {
  const int a = m / 2;
  return m % 2 == 0 ? a * L - a * (a - 1) : order_odd0(L) + a * L - a * a;
}
// SYRK: out = t64: tiles (r, c) -= A_r B_c^T for the blocks of the region on
//   or below the diagonal; A and B rows are matrix rows of a panel's digits.
// TRSM: out = t64: column block c of the listed tiles -= X_J L_cJ^T; X digits
//   per slot (launch_trsm_block), L_kk digits of block J (launch_lkk_digits).
// TRMM: out(row, col) = A_row B_col^T over K = the row's tiles 0 .. row / nb,
//   out column-major; A rows start at matrix row a_row0.
// DENSE: rows r < rows_valid (K-major digits), columns c < cols_valid, K = nk:
//   out[(r / div) * ld2 + r % div + c * ldo].
// SYN, per order m < L (of a spherical-harmonic transform): rows (s, t) = s T + t
//   (s = 0: order m, 1: order -m), columns i < ntheta, K the degrees of m's
//   block of 32 orders (order_k); out[t + T (i + ntheta (2 m + s)).
// ANA, per order m < L: rows (s, t), columns l - m for l = m .. L-1, K = nk
//   grid rings; A rows m rpad + (s, t), B rows order_pos(m) + l - m;
//   out[t ldo + l^2 + l +- m].
enum { SRC_LIST = 0, SRC_SYRK = 1, SRC_TRSM = 2, SRC_TRMM = 3, SRC_DENSE = 4, SRC_SYN = 5, SRC_ANA = 6 };
emu_status launch_region(emu_ctx *ctx, int src, const CUtensorMap &a, const CUtensorMap &b, const Region &rg,
                         int a_plane, int b_plane, const int *a_exp, const int *b_exp, double *out, long ldo,
                         int max_ctas);

// Row exponents and digits of rows [row0, row0 + nrows) of the tile columns
// [col0, ncols) (in tiles; ncols < 0: up to the row's own tile) of a packed
// FP64 matrix: exps[r - e_row0], plane p of row r at arena row
// p * plane + r - d_row0, K-major with kpad columns.  One exponent per row.
// Tiles above the diagonal are not read.  row0, nrows multiples of 32.
emu_status launch_panel_digits(emu_ctx *ctx, const double *t64, int NT, int nb, int row0, int nrows, int tcol0,
                               int tcols, int e_row0, int *exps, int d_row0, long plane, long kpad,
                               uint16_t *digits);

// Workspace of the blocked FP64-class TRSM over `slots` tiles of size nb.
struct TrsmPlan {
  int *xexp = nullptr;
  uint16_t *xdig = nullptr;   // solved blocks: slot s, plane p, row r at (s NS + p) nb + r, TW columns
  int *lexp = nullptr;        // L_kk's column blocks (launch_lkk_digits)
  uint16_t *ldig = nullptr;
  double *ls = nullptr, *rinv = nullptr;  // launch_trsm64_prep
  CUtensorMap mx, ml;
};
size_t trsm_plan_bytes(int nb, int slots);
// Lays the plan out in `base` (trsm_plan_bytes, 256-byte aligned) and encodes its maps.
emu_status trsm_plan_init(emu_ctx *ctx, TrsmPlan *P, char *base, int nb, int slots);
// Per panel, after its POTRF: the pre-scaled diagonal blocks and the digits of
// L_kk's column blocks.
emu_status trsm_plan_prep(emu_ctx *ctx, const TrsmPlan &P, const double *Lkk, int nb);
// X = A L_kk^{-T} in place for the tiles d_tiles[0 .. n) (slots slot0 ..).
emu_status trsm_plan_solve(emu_ctx *ctx, const TrsmPlan &P, double *t64, int nb, const int *d_tiles, int n,
                           const double *Lkk, int slot0);

// out64 (-= or +=) per item, K = nb per segment, on at most max_ctas persistent
// CTAs; a_plane / b_plane = arena rows between digit planes.
emu_status launch(emu_ctx *ctx, const CUtensorMap &a, const CUtensorMap &b, const Item *d_items, int nitems,
                  const Seg *d_segs, int nb, int a_plane, int b_plane, const int *a_exp, const int *b_exp, int mode,
                  double *out64, int ldo, int max_ctas);

}  // namespace gemm64
