// refine_split.h -- how the residual's product is split over the chip (refine.cu).
// Host arithmetic only: every tile count, tile size and number of right-hand
// sides a matrix can have gives a split.
#pragma once
#include <stddef.h>

#include <algorithm>

constexpr int RS = 64;  // rows of a slab; tile sizes are multiples of it

// Right-hand sides per group, groups and ranges of tile columns.
struct ResidualSplit {
  int P, groups, nz;
  // FP64 partial sums of a matrix of npad rows: one range needs none (the sums
  // are the product), and several ranges are few slabs, so that 12 x 64 x 32
  // doubles per SM, 30 MB, hold them for every number of right-hand sides.
  size_t partial(long npad) const { return nz == 1 ? 0 : (size_t)groups * nz * npad * P; }
};
// P follows the right-hand sides (one of them cost sixteen columns' FP64 work),
// and the ranges fill the chip where n / 64 slabs do not (60 CTAs at n = 3840).
inline ResidualSplit residual_split(int sm_count, int nt, int nb, int nrhs) {
  ResidualSplit s;
  s.P = nrhs == 1 ? 1 : nrhs <= 4 ? 4 : nrhs <= 8 ? 8 : nrhs <= 16 ? 16 : 32;
  s.groups = (nrhs + s.P - 1) / s.P;
  const long slabs = (long)nt * (nb / RS) * s.groups;
  s.nz = (int)std::max(1l, std::min((long)nt, (6l * sm_count + slabs - 1) / slabs));
  return s;
}
