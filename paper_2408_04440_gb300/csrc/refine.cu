// refine.cu -- iterative refinement for S X = B: the correction comes from the
// (possibly mixed-precision) factor, the residual R = B - S X and the update
// X += D are FP64 against the FP64 covariance tiles.  Stops when the normwise
// backward error ||r||_2 / (||S||_F ||x||_2 + ||b||_2) of every column is <= tol.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mixed.h"
#include "refine_split.h"

namespace {

// Partial sums of S X for S symmetric from its packed lower FP64 tiles, FP64 on
// the SIMT pipes: one CTA per (64-row slab of the padded matrix, range of tile
// columns, group of P right-hand sides), a loop over its tile columns j (tile
// (i, j) for j <= i, tile (j, i) read transposed for j > i), operands staged
// through shared memory in 32-wide K chunks so that every global read is
// coalesced.  part[z][row][P] of range z and group blockIdx.z; deterministic:
// one CTA owns each partial sum, k_symm_finish adds the ranges in order.  With
// one range (from 58000 rows times groups on) R = Bm - S X is written here.
//
// Bound by FP64 issue from a few right-hand sides on.  As digit products on the
// tensor cores n = 16384 with 16 columns takes 1.5 ms instead of 7.3, but that
// cuts the entries of S relative to their tile: a solution's entry that hangs on
// covariances 1e-12 of their tile's largest was off by 1.5e-6 of itself after
// refinement, where this sum, which takes every entry of S whole, leaves 5e-15.
constexpr int RK = 32;
template <int P>
__global__ void __launch_bounds__(256)
    k_symm_part(const double *__restrict__ t64, int nb, int NT, const double *__restrict__ X,
                const double *__restrict__ Bm, double *__restrict__ R, double *__restrict__ part, long npad, int nrhs) {
  constexpr int KG = P == 1 ? 4 : 1;       // thread groups that share the K chunk
  constexpr int NQ = P == 1 ? 1 : P / 4;   // right-hand sides per thread
  __shared__ double a[RK][RS + 1];
  __shared__ double x[RK][P + 1];
  const long g0 = (long)blockIdx.x * RS;
  const int i = (int)(g0 / nb), m0 = (int)(g0 % nb);
  const int c0 = blockIdx.z * P;
  const int p = min(P, nrhs - c0);
  const int tid = threadIdx.x, mm = tid & (RS - 1), q0 = tid >> 6;
  const int j0 = (int)((long)NT * blockIdx.y / gridDim.y), j1 = (int)((long)NT * (blockIdx.y + 1) / gridDim.y);
  double acc[NQ];
#pragma unroll
  for (int w = 0; w < NQ; w++) acc[w] = 0.0;
  for (int j = j0; j < j1; j++) {
    const bool lower = j <= i;
    const double *T = t64 + (size_t)(lower ? tile_index(i, j, NT) : tile_index(j, i, NT)) * nb * nb;
    for (int k0 = 0; k0 < nb; k0 += RK) {
      double v[RK * RS / 256];
#pragma unroll
      for (int u = 0; u < RK * RS / 256; u++) {
        const int e = tid + 256 * u;
        v[u] = lower ? __ldg(T + (size_t)(m0 + e % RS) + (size_t)(k0 + e / RS) * nb)
                     : __ldg(T + (size_t)(k0 + e % RK) + (size_t)(m0 + e / RK) * nb);
      }
#pragma unroll
      for (int u = 0; u < RK * RS / 256; u++) {
        const int e = tid + 256 * u;
        if (lower) a[e / RS][e % RS] = v[u];
        else a[e % RK][e / RK] = v[u];
      }
      for (int e = tid; e < RK * P; e += 256) {
        const int k = e % RK, q = e / RK;
        x[k][q] = q < p ? X[(size_t)j * nb + k0 + k + (size_t)(c0 + q) * npad] : 0.0;
      }
      __syncthreads();
      if (KG == 4) {
#pragma unroll
        for (int k = 0; k < RK / 4; k++) acc[0] = fma(a[k + q0 * (RK / 4)][mm], x[k + q0 * (RK / 4)][0], acc[0]);
      } else {
#pragma unroll 4
        for (int k = 0; k < RK; k++) {
          const double av = a[k][mm];
#pragma unroll
          for (int w = 0; w < NQ; w++) acc[w] = fma(av, x[k][q0 + 4 * w], acc[w]);
        }
      }
      __syncthreads();
    }
  }
  if (KG == 4) {
    double *red = &a[0][0];
    red[tid] = acc[0];
    __syncthreads();
    if (tid >= RS) return;
    acc[0] = (red[tid] + red[tid + 64]) + (red[tid + 128] + red[tid + 192]);
  }
  if (gridDim.y == 1) {
    // one range: the product is complete
#pragma unroll
    for (int w = 0; w < NQ; w++) {
      const size_t o = (size_t)(g0 + mm) + (size_t)(c0 + q0 + 4 * w) * npad;
      if (q0 + 4 * w < p) R[o] = Bm[o] - acc[w];
    }
  } else {
    double *o = part + (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * npad + g0 + mm) * P;
#pragma unroll
    for (int w = 0; w < NQ; w++) o[q0 + 4 * w] = acc[w];
  }
}

// R = B - the sum of the partial products' `nz` ranges, in order.
__global__ void k_symm_finish(const double *__restrict__ part, int nz, int P, const double *__restrict__ Bm,
                              double *__restrict__ R, long npad, int nrhs) {
  const long total = npad * nrhs;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const long r = e % npad;
    const int c = (int)(e / npad);
    double s = 0.0;
    for (int z = 0; z < nz; z++) s += part[(((size_t)(c / P) * nz + z) * npad + r) * P + c % P];
    R[e] = Bm[e] - s;
  }
}

// Column sums of squares of R, X and B (one CTA per column, fixed order), and
// after them whether a wait ran out in the sweeps so far.
__global__ void k_col_norms(const double *__restrict__ R, const double *__restrict__ X,
                            const double *__restrict__ Bm, long n, long ld, double *__restrict__ out, const int *st) {
  int c = blockIdx.x;
  double sr = 0, sx = 0, sb = 0;
  for (long r = threadIdx.x; r < n; r += blockDim.x) {
    double a = R[r + c * ld], b = X[r + c * ld], d = Bm[r + c * ld];
    sr += a * a;
    sx += b * b;
    sb += d * d;
  }
  __shared__ double sh[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_down_sync(0xffffffffu, sr, o);
    sx += __shfl_down_sync(0xffffffffu, sx, o);
    sb += __shfl_down_sync(0xffffffffu, sb, o);
  }
  int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    sh[0][w] = sr;
    sh[1][w] = sx;
    sh[2][w] = sb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0, d = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); k++) {
      a += sh[0][k];
      b += sh[1][k];
      d += sh[2][k];
    }
    out[3 * c] = a;
    out[3 * c + 1] = b;
    out[3 * c + 2] = d;
    if (c == 0) out[3 * gridDim.x] = st[ST_CODE] == DEV_TIMEOUT || st[ST_LATE] ? 1.0 : 0.0;
  }
}

__global__ void k_axpy(double *__restrict__ X, const double *__restrict__ D, long total) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < total; q += (long)gridDim.x * blockDim.x)
    X[q] += D[q];
}

}  // namespace

// R = B - S X (npad x nrhs each); part: the split's partial sums.
static emu_status symm_residual(emu_ctx *ctx, const emu_mat *S, const double *X, const double *Bp, double *R,
                                double *part, int nrhs) {
  const long npad = (long)S->nt * S->nb;
  const ResidualSplit sh = residual_split(ctx->sm_count, S->nt, S->nb, nrhs);
  ProfScope ps(ctx, PROF_SOLVE, 2.0 * (double)npad * npad * nrhs, 8.0 * (double)npad * npad);
  const dim3 grid((unsigned)(npad / RS), (unsigned)sh.nz, (unsigned)sh.groups);
  auto kern = sh.P == 1    ? k_symm_part<1>
              : sh.P == 4  ? k_symm_part<4>
              : sh.P == 8  ? k_symm_part<8>
              : sh.P == 16 ? k_symm_part<16>
                           : k_symm_part<32>;
  kern<<<grid, 256, 0, ctx->stream>>>(S->t64, S->nb, S->nt, X, Bp, R, part, npad, nrhs);
  EMU_LAUNCHED(ctx);
  if (sh.nz == 1) return EMU_OK;
  k_symm_finish<<<4 * ctx->sm_count, 256, 0, ctx->stream>>>(part, sh.nz, sh.P, Bp, R, npad, nrhs);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status refine_solve(emu_ctx *ctx, const emu_mat *L, const emu_mat *S, const double *dB,
                        long ldb, double *dX, long ldx, int nrhs, double tol, int maxit,
                        emu_refine_info *info) {
  if (nrhs == 0) return EMU_OK;
  EMU_CUDA_TRY(ctx, cudaSetDevice(ctx->device));
  long npad = (long)L->nt * L->nb;
  size_t blk = (size_t)npad * nrhs;
  double *buf = nullptr, *norms = nullptr;
  const ResidualSplit sh = residual_split(ctx->sm_count, S->nt, S->nb, nrhs);
  EMU_CUDA_TRY(ctx, cudaMallocAsync(&buf, (4 * blk + sh.partial(npad)) * sizeof(double), ctx->stream));
  EMU_CUDA_TRY(ctx, cudaMallocAsync(&norms, (3 * (size_t)nrhs + 1) * sizeof(double), ctx->stream));
  double *Bp = buf, *X = buf + blk, *R = buf + 2 * blk, *D = buf + 3 * blk;
  std::vector<double> hn(3 * (size_t)nrhs + 1);
  double frobS = 0.0;
  emu_status s = EMU_OK;
  int it = 0;
  double eta = INFINITY;
  float ms = 0.f;
  cudaError_t e = cudaMemsetAsync(buf, 0, 4 * blk * sizeof(double), ctx->stream);
  if (e == cudaSuccess)
    e = cudaMemcpy2DAsync(Bp, npad * sizeof(double), dB, ldb * sizeof(double), (size_t)L->n * sizeof(double),
                          nrhs, cudaMemcpyDeviceToDevice, ctx->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&frobS, S->d_frob, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaEventRecord(ctx->ev0, ctx->stream);
  if (e != cudaSuccess) s = emu_cuda_fail(ctx, e, "refine setup");
  // X0 = M^{-1} B
  if (s == EMU_OK) {
    e = cudaMemcpyAsync(X, Bp, blk * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream);
    s = (e == cudaSuccess) ? factor_potrs(ctx, L, X, npad, nrhs) : emu_cuda_fail(ctx, e, "refine x0");
  }
  while (s == EMU_OK) {
    if ((s = symm_residual(ctx, S, X, Bp, R, buf + 4 * blk, nrhs)) != EMU_OK) break;
    k_col_norms<<<nrhs, 256, 0, ctx->stream>>>(R, X, Bp, npad, npad, norms, ctx->d_status);
    ctx->launches++;
    e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(hn.data(), norms, hn.size() * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e == cudaSuccess && hn.back() != 0.0) {
      // a sweep that gave up has left X or its correction half solved
      e = cudaMemcpyAsync(ctx->h_status, ctx->d_status, ST_WORDS * sizeof(int), cudaMemcpyDeviceToHost, ctx->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
      if (e == cudaSuccess) s = status_timed_out(ctx);
    }
    if (e != cudaSuccess) s = emu_cuda_fail(ctx, e, "refine residual");
    if (s != EMU_OK) break;
    eta = 0.0;
    for (int c = 0; c < nrhs; c++) {
      double den = frobS * sqrt(hn[3 * c + 1]) + sqrt(hn[3 * c + 2]);
      double v = den > 0 ? sqrt(hn[3 * c]) / den : 0.0;
      if (!(v <= eta)) eta = v;  // NaN propagates
    }
    if (eta <= tol) break;
    if (it >= maxit) {
      s = EMU_ENOCONV;
      break;
    }
    e = cudaMemcpyAsync(D, R, blk * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream);
    if (e != cudaSuccess) {
      s = emu_cuda_fail(ctx, e, "refine copy");
      break;
    }
    s = factor_potrs(ctx, L, D, npad, nrhs);
    if (s != EMU_OK) break;
    k_axpy<<<4 * ctx->sm_count, 256, 0, ctx->stream>>>(X, D, (long)blk);
    ctx->launches++;
    it++;
  }
  cudaEventRecord(ctx->ev1, ctx->stream);
  if (s == EMU_OK || s == EMU_ENOCONV) {
    e = cudaMemcpy2DAsync(dX, ldx * sizeof(double), X, npad * sizeof(double), (size_t)L->n * sizeof(double),
                          nrhs, cudaMemcpyDeviceToDevice, ctx->stream);
    if (e != cudaSuccess) s = emu_cuda_fail(ctx, e, "refine copy-out");
  }
  cudaFreeAsync(buf, ctx->stream);
  cudaFreeAsync(norms, ctx->stream);
  cudaStreamSynchronize(ctx->stream);
  cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1);
  if (info) {
    info->iters = it;
    info->rel_resid = eta;
    info->ms = ms;
  }
  return s;
}
