// symm_digits.h -- S X for a symmetric covariance in packed FP64 tiles as digit
// products on the tensor cores (symm_digits.cu), for the residual of iterative
// refinement.
#pragma once
#include "emu_internal.h"

namespace symm_digits {

constexpr int NR = 16;  // right-hand sides per group

struct Plan {
  int groups = 0, nz = 0;     // groups of NR right-hand sides, column ranges per row block
  int *dexp = nullptr;        // npad: S_rr < 2^(2 dexp)
  int *dmin = nullptr;        // NT: least dexp of a tile row
  int *texp = nullptr;        // per tile: |S_rc| 2^-(dexp_r + dexp_c) < 2^texp
  int *flag = nullptr;        // set when a bound did not hold: the product is not valid
  int *xexp = nullptr;        // [chunk][NR] (biased)
  uint16_t *xdig = nullptr;   // row q NR + c: digit q of right-hand side c, npad columns
};
// Tile sizes it takes.
inline bool supports(const emu_mat *S) { return S->nb % 128 == 0; }
Plan shape(const emu_ctx *ctx, const emu_mat *S, int nrhs);
size_t bytes(const emu_mat *S);
// Lays the plan out in `base` (256-byte aligned) and enqueues the scales of S.
emu_status init(emu_ctx *ctx, Plan *P, char *base, const emu_mat *S);
// part[(group nz + z) npad + row][NR] = the partial products of S X over the
// column ranges z (X: npad x nrhs, leading dimension npad).
emu_status multiply(emu_ctx *ctx, const Plan &P, const emu_mat *S, const double *X, int nrhs, double *part);

}  // namespace symm_digits
