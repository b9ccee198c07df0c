// factor64.h -- the plain FP64 factor and its draws as digit products on the
// tensor cores (factor64.cu).
#pragma once
#include "emu_internal.h"

// Tile sizes the digit form takes: multiples of 128 (its block heights).
// Others (64, 192, ...) run on the FP64 pipe (fp64.cu).
bool factor64_digits_supports(const emu_mat *A);
// EMU_ENOMEM: the workspace does not fit and nothing was enqueued.
emu_status factor64_digits(emu_ctx *ctx, emu_mat *A);
// Y = L Z for a plain FP64 factor, Z npad x s; enqueues and returns.
// EMU_ENOMEM as above.
emu_status sample64_digits(emu_ctx *ctx, const emu_mat *L, const double *Z, long ldz, int s, double *Y, long ldy);
