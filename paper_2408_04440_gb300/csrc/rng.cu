// rng.cu -- standard normals z ~ N(0, I) for drawing emulations
// ("Generating Emulations": xi = V z).  Counter-based, so every entry depends
// only on (seed, stream id, row, column) and never on the launch shape:
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) at counter
// {p mod 2^32, p >> 32, column, stream id}, key {seed mod 2^32, seed >> 32},
// p = row / 2; two 53-bit uniforms u1 in (0,1], u2 in [0,1); Box-Muller gives
// rows 2p (cosine) and 2p+1 (sine).
#include <algorithm>

#include "emu_internal.h"
#include "rng.cuh"

namespace {

// Pairs on x, columns on y; nrows is even when `vec` (16-byte stores).
__global__ void __launch_bounds__(256)
    k_normals(uint64_t seed, uint32_t stream_id, int nrows, int s, double *__restrict__ Z, long ldz, bool vec) {
  __shared__ NormalTables T;
  T.load();
  __syncthreads();
  const int npairs = (nrows + 1) / 2;
  for (int col = blockIdx.y; col < s; col += gridDim.y)
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npairs; p += gridDim.x * blockDim.x) {
      const double2 v = normal_pair(seed, stream_id, p, col, T);
      double *z = Z + (size_t)col * ldz + 2L * p;
      if (vec) {
        *reinterpret_cast<double2 *>(z) = v;
      } else {
        z[0] = v.x;
        if (2L * p + 1 < nrows) z[1] = v.y;
      }
    }
}

// Batch: blockIdx.y = matrix b, all NT_b * nb padded rows of its block of the
// stacked Z (rows row_base ..), with its own stream id.
// The seed is read from device memory so that a captured graph can be
// replayed with another seed.
__global__ void __launch_bounds__(256)
    k_normals_batch(const uint64_t *__restrict__ seed_p, const BatchInst *__restrict__ inst, int nb,
                                int s, double *__restrict__ Z, long ldz) {
  __shared__ NormalTables T;
  T.load();
  __syncthreads();
  const uint64_t seed = *seed_p;
  const BatchInst I = inst[blockIdx.y];
  const int npairs = I.NT * nb / 2;  // nb is even
  double *Zb = Z + I.row_base;
  for (int col = blockIdx.x; col < s; col += gridDim.x)
    for (int p = threadIdx.x; p < npairs; p += blockDim.x)
      *reinterpret_cast<double2 *>(Zb + (size_t)col * ldz + 2L * p) =
          normal_pair(seed, (uint32_t)I.stream_id, p, col, T);
}
}  // namespace

emu_status launch_normals(emu_ctx *ctx, uint64_t seed, uint32_t stream_id, int nrows,
                          int s, double *Z, long ldz) {
  // about eight CTAs per SM, each with pairs enough to pay for its 11 KB of tables
  const int most = std::max(1, ((nrows + 1) / 2 + 255) / 256);
  const int gy = std::max(1, std::min(s, 8 * ctx->sm_count));
  const int gx = std::max(1, std::min(most, 8 * ctx->sm_count / gy));
  const bool vec = nrows % 2 == 0 && ldz % 2 == 0 && (reinterpret_cast<uintptr_t>(Z) & 15) == 0;
  ProfScope ps(ctx, PROF_RNG, 0.0, 8.0 * nrows * (double)s);
  k_normals<<<dim3(gx, gy), 256, 0, ctx->stream>>>(seed, stream_id, nrows, s, Z, ldz, vec);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status launch_normals_batch(emu_ctx *ctx, const uint64_t *d_seed, const BatchInst *d_inst, int count,
                                int maxNT, int nb, int s, double *Z, long ldz) {
  const int bx = std::max(1, std::min(s, 16));
  ProfScope ps(ctx, PROF_RNG, 0.0, 0.0);
  if (ldz % 2 != 0) return EMU_EINVAL;
  k_normals_batch<<<dim3(bx, count), 256, 0, ctx->stream>>>(d_seed, d_inst, nb, s, Z, ldz);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}
