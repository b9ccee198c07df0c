// sht_digits.h -- the spherical-harmonic transforms as digit products on the
// tensor cores (sht_digits.cu).  Both wait for the result and return
//   EMU_ENOMEM  the workspace does not fit, or the sizes do not: nothing was
//               written;
//   EMU_ESTATE  an operand held an infinity or a NaN: the caller runs the
//               direct sums, which carry them as floating point does.
// d_status is zero on entry.
#pragma once
#include "emu_internal.h"

emu_status isht_digits(emu_ctx *ctx, const double *dF, int L, int T, long ldf, int ntheta, int nphi, double *dZ,
                       long ldz);
emu_status sht_digits(emu_ctx *ctx, const double *dZ, int ntheta, int nphi, int T, long ldz, int L, double *dF,
                      long ldf);
