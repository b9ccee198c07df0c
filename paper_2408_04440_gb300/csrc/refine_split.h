// refine_split.h -- how the residual's product is split over the chip (refine.cu).
// Host arithmetic only: every tile count, tile size and number of right-hand
// sides a matrix can have gives a split.
#pragma once
#include <algorithm>

constexpr int RS = 64;  // rows of a slab; tile sizes are multiples of it

// Right-hand sides per group, groups and ranges of tile columns.
struct ResidualSplit {
  int P, groups, nz;
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
