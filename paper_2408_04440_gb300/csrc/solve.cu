// solve.cu -- the triangular solves L L^T X = B with a factor in packed tiles:
// emu_potrs, and the preconditioner of iterative refinement (each correction
// is M^{-1} r with M = L L^T; the FP64 residual and update live in refine.cu).
//
// Arithmetic.  A mixed factor solves in FP32: products of the stored tiles
// (FP64 tiles rounded to FP32, FP32 masters as they are; the diagonal tiles
// from their FP64 factor), accumulated in FP32 per tile in the order of the
// tile's rows and added to the FP64 right-hand sides; inside a diagonal tile
// the right-hand sides are FP32.  A plain FP64 factor solves in FP64.
//
// One launch per sweep, a dataflow over slabs of 64 rows: a CTA takes the next
// slab from a counter, subtracts the products of its blocks with the solved
// slabs, solves its own 64 x 64 triangle and publishes the result.  Slabs are
// taken in the order they are solved, so the earliest unfinished one always
// runs and only waits for finished ones; every wait is bounded.  A solved
// value is published with a tag in one 64-bit word, so that a reader polls the
// data itself: no flag, fence or second read is on the chain of n / 64 slabs
// (block product, triangle, hand-over).  The other resident CTAs read and
// convert their blocks meanwhile.  (A launch per tile for the diagonal solve
// and one for its panel cost 110 + 38 us per 256-wide tile: the diagonal solve
// was one CTA, bound by its conversions of FP64 entries, which hold the FP64
// pipe.)  A slab takes 3.5 us forward and 5.9 us backward at n = 3840 with one
// right-hand side, 7.3 and 9.6 us at n = 65536 with 16; both sweeps 4.3 -> 0.57
// and 95 -> 17 ms.  With every waiting CTA polling whole slabs they took 0.81
// and 33 ms.
#include <algorithm>

#include "convert.cuh"
#include "mixed.h"

namespace {

constexpr int SL = 64;    // rows of a slab
constexpr int LDA = 68;   // FP32 columns of a block in shared memory: 16-byte aligned, float4 reads down a column
constexpr int LDD = 66;   // FP64 columns
// default wait bound in SM clock cycles (about 2 s at 2 GHz)
constexpr long long kSweepWaitCycles = 4000000000ll;
// Published values of the groups of one launch: 16 bytes per FP32 entry of X in
// both sweeps, 32 per FP64 one, up to this much (n = 65536 with 2000 right-hand
// sides).  Every further launch is another ramp and tail of n / 64 slabs: with
// 64 MB the 1000 right-hand sides of n = 16384 ran in five launches, 66.7 ms
// instead of 56.4.
constexpr size_t kSweepWorkspace = (size_t)2 << 30;

__device__ inline bool failed(const int *st) { return *((volatile const int *)st) != DEV_OK; }

template <typename F>
__device__ inline F from_f64(double x);
template <>
__device__ inline float from_f64<float>(double x) { return f32_of(x); }
template <>
__device__ inline double from_f64<double>(double x) { return x; }

// A solved value with its tag: one 64-bit word per FP32, two per FP64 (each half
// with the tag), stored and polled as whole words.
constexpr unsigned long long kTag = 1ull << 32;
__device__ inline void put_word(unsigned long long *p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(kTag | v) : "memory");
}
__device__ inline unsigned long long get_word(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ inline void publish(unsigned long long *p, float v) { put_word(p, __float_as_uint(v)); }
__device__ inline void publish(unsigned long long *p, double v) {
  put_word(p, (unsigned)__double2loint(v));
  put_word(p + 1, (unsigned)__double2hiint(v));
}
__device__ inline float from_words(const unsigned long long (&w)[1]) { return __uint_as_float((unsigned)w[0]); }
__device__ inline double from_words(const unsigned long long (&w)[2]) {
  return __hiloint2double((int)(unsigned)w[1], (int)(unsigned)w[0]);
}

// One sweep for right-hand sides [c0, c0 + P), c0 = blockIdx.y P: forward
// X <- L^{-1} X or (BACK) X <- L^{-T} X.  ticket: the next slab per group, zero
// before the launch.  xs: the solved slabs, [group][slab][64][P] tagged values,
// zero before the launch.  cls null: every tile is FP64 (plain factor).
// wait_cycles: bound of a wait; withhold: slab that is not published (for
// tests; else -1).
template <typename F, int P, bool BACK>
__global__ void __launch_bounds__(256, sizeof(F) == 4 ? 2 : 1)
    k_sweep(const double *__restrict__ t64, const float *__restrict__ t32, const unsigned char *__restrict__ cls, int nb,
            int NT, int nslab, double *__restrict__ X, long ld, int nrhs, unsigned long long *__restrict__ xs,
            int *__restrict__ ticket, int *st, long long wait_cycles, int withhold) {
  constexpr int NQ = P / 4;                       // right-hand sides per thread
  constexpr int NW = sizeof(F) / 4;               // words per published value
  constexpr int LD = sizeof(F) == 4 ? LDA : LDD;  // block column stride
  extern __shared__ __align__(16) uint8_t smem[];
  F *a = reinterpret_cast<F *>(smem);             // two blocks [64 columns][LD]
  F *x = a + 2 * SL * LD;                         // [64][P] of the block's solved slab
  F *rinv = x + SL * P;                           // [64]
  __shared__ int s_slab;
  const int tid = threadIdx.x, row = tid & (SL - 1), g = tid >> 6, lane = tid & 31, w = tid >> 5;
  const int grp = blockIdx.y, c0 = grp * P, p = min(P, nrhs - c0);
  ticket += grp;
  xs += (size_t)grp * nslab * SL * P * NW;
  const int per = nb / SL;
  const size_t te = (size_t)nb * nb;
  if (__syncthreads_or(tid == 0 && failed(st))) return;

  // block (I, J) of the factor, I >= J, to shared memory: 16 entries per thread
  // held in registers on the way, columns cl, cl + 16, .. and rows rq .. rq + 3
  const int cl = tid >> 4, rq = (tid & 15) * 4;
  float4 vf[4];
  double2 vd[8];
  bool v64 = false;
  auto fetch = [&](int I, int J) {
    const long t = tile_index(I / per, J / per, NT);
    const size_t o = (size_t)t * te + (size_t)(I % per) * SL + rq + (size_t)((J % per) * SL + cl) * nb;
    v64 = cls == nullptr || I / per == J / per || cls[t] == EMU_CLASS_FP64;
    if (v64) {
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const double2 *s = reinterpret_cast<const double2 *>(t64 + o + (size_t)(16 * q) * nb);
        vd[2 * q] = __ldg(s);
        vd[2 * q + 1] = __ldg(s + 1);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; q++) vf[q] = __ldg(reinterpret_cast<const float4 *>(t32 + o + (size_t)(16 * q) * nb));
    }
  };
  // `flip`: transposed, as the backward sweep reads its triangle
  auto stash = [&](F *dst, bool flip) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int c = cl + 16 * q;
      F d[4];
      if (v64) {
        d[0] = from_f64<F>(vd[2 * q].x);
        d[1] = from_f64<F>(vd[2 * q].y);
        d[2] = from_f64<F>(vd[2 * q + 1].x);
        d[3] = from_f64<F>(vd[2 * q + 1].y);
      } else {
        d[0] = (F)vf[q].x;
        d[1] = (F)vf[q].y;
        d[2] = (F)vf[q].z;
        d[3] = (F)vf[q].w;
      }
#pragma unroll
      for (int i = 0; i < 4; i++) dst[flip ? (rq + i) * LD + c : c * LD + rq + i] = d[i];
    }
  };

  while (true) {
    if (tid == 0) s_slab = atomicAdd(ticket, 1);
    __syncthreads();
    const int k = s_slab;  // k-th slab of the sweep
    if (k >= nslab) break;
    const int s = BACK ? nslab - 1 - k : k, t = s / per;
    // j-th of the k solved slabs it needs, in the order of its sums: tile by
    // tile away from the sweep's start, a tile's rows ascending; then the slabs
    // of its own tile as they were solved; j = k is the slab itself
    const int noff = BACK ? nslab - (t + 1) * per : t * per;
    auto other = [&](int j) {
      if (!BACK) return j;
      return j < noff ? (NT - 1 - j / per) * per + j % per : (t + 1) * per - 1 - (j - noff);
    };
    auto block = [&](int j) {
      const int o = other(j);
      if (BACK) fetch(o, s);
      else fetch(s, o);
    };
    block(0);
    double b[NQ];
    F acc[NQ];  // a tile's sums; from the own tile on, the right-hand sides themselves
#pragma unroll
    for (int q = 0; q < NQ; q++) {
      const int c = g * NQ + q;
      b[q] = c < p ? X[(size_t)s * SL + row + (size_t)(c0 + c) * ld] : 0.0;
      acc[q] = noff == 0 ? from_f64<F>(b[q]) : (F)0;
    }
    stash(a, BACK && k == 0);
    bool bad = false;
    for (int j = 0; j < k; j++) {
      block(j + 1);
      // the solved slab's values.  The next slab in line polls them all; the
      // others, hundreds of CTAs at the sweep's front, would slow its hand-over
      // down with that: one thread polls one value, with pauses.
      const unsigned long long *xo = xs + (size_t)other(j) * SL * P * NW;
      bool early = false;
      long long t0 = 0;
      while (true) {
        int miss = 0;
        unsigned long long v[SL * P / 256][NW];
#pragma unroll
        for (int u = 0; u < SL * P / 256; u++)
#pragma unroll
          for (int h = 0; h < NW; h++) {
            v[u][h] = get_word(xo + (size_t)(tid + 256 * u) * NW + h);
            miss |= v[u][h] < kTag;
          }
#pragma unroll
        for (int u = 0; u < SL * P / 256; u++) x[tid + 256 * u] = from_words(v[u]);
        if (!__syncthreads_or(miss)) break;
        if (!early) {
          // while it waits: the next block into place
          early = true;
          stash(a + ((j + 1) & 1) * SL * LD, BACK && j + 1 == k);
          t0 = clock64();
        }
        if (tid == 0) {
          if (j + 1 < k)
            while (get_word(xo + (size_t)(P - 1) * NW) < kTag && !failed(st) && clock64() - t0 <= wait_cycles)
              __nanosleep(256);
          if (clock64() - t0 > wait_cycles) status_timeout(st, 6);
        }
        if (__syncthreads_or(tid == 0 && failed(st))) {
          bad = true;
          break;
        }
      }
      if (bad) break;
      const F *ab = a + (j & 1) * SL * LD;
      if (j < noff) {
        if (sizeof(F) == 4 && BACK) {
#pragma unroll 4
          for (int kk = 0; kk < SL; kk += 4) {
            const float4 av = *reinterpret_cast<const float4 *>(ab + row * LD + kk);
            const F a4[4] = {(F)av.x, (F)av.y, (F)av.z, (F)av.w};
#pragma unroll
            for (int u = 0; u < 4; u++)
#pragma unroll
              for (int q = 0; q < NQ; q++) acc[q] = fma(a4[u], x[(kk + u) * P + g * NQ + q], acc[q]);
          }
        } else {
#pragma unroll 8
          for (int kk = 0; kk < SL; kk++) {
            const F av = BACK ? ab[row * LD + kk] : ab[kk * LD + row];
#pragma unroll
            for (int q = 0; q < NQ; q++) acc[q] = fma(av, x[kk * P + g * NQ + q], acc[q]);
          }
        }
        if ((j + 1) % per == 0) {
          // a tile's products end: the sums go to the FP64 right-hand side
#pragma unroll
          for (int q = 0; q < NQ; q++) {
            b[q] -= (double)acc[q];
            acc[q] = j + 1 == noff ? from_f64<F>(b[q]) : (F)0;
          }
        }
      } else if (sizeof(F) == 4 && BACK) {
        // own tile: the later half of the slab's rows first
#pragma unroll 4
        for (int e = 0; e < SL; e += 4) {
          const int kk = e ^ 32;
          const float4 av = *reinterpret_cast<const float4 *>(ab + row * LD + kk);
          const F a4[4] = {(F)-av.x, (F)-av.y, (F)-av.z, (F)-av.w};
#pragma unroll
          for (int u = 0; u < 4; u++)
#pragma unroll
            for (int q = 0; q < NQ; q++) acc[q] = fma(a4[u], x[(kk + u) * P + g * NQ + q], acc[q]);
        }
      } else {
#pragma unroll 8
        for (int e = 0; e < SL; e++) {
          const int kk = BACK ? e ^ 32 : e;
          const F av = BACK ? ab[row * LD + kk] : ab[kk * LD + row];
#pragma unroll
          for (int q = 0; q < NQ; q++) acc[q] = fma(-av, x[kk * P + g * NQ + q], acc[q]);
        }
      }
      if (!early) stash(a + ((j + 1) & 1) * SL * LD, BACK && j + 1 == k);
      __syncthreads();  // x and block j are free, block j + 1 is in place
    }
    if (bad) break;
    if (k == 0) __syncthreads();
    // triangle: P / 8 right-hand sides per warp
    const F *T = a + (k & 1) * SL * LD;
#pragma unroll
    for (int q = 0; q < NQ; q++) x[row * P + g * NQ + q] = acc[q];
    if (tid < SL) rinv[tid] = (F)1 / T[tid * LD + tid];
    __syncthreads();
    unsigned long long *xo = xs + (size_t)s * SL * P * NW;
    constexpr int NR = P > 8 ? P / 8 : 1;  // right-hand sides per warp, side by side
    if (w < P) {
      F y0[NR], y1[NR];
#pragma unroll
      for (int r = 0; r < NR; r++) {
        y0[r] = x[lane * P + w + 8 * r];
        y1[r] = x[(lane + 32) * P + w + 8 * r];
      }
      if (!BACK) {
#pragma unroll 8
        for (int q = 0; q < 32; q++) {
          const F l0 = lane > q ? -T[q * LD + lane] : (F)0, l1 = -T[q * LD + lane + 32], ri = rinv[q];
#pragma unroll
          for (int r = 0; r < NR; r++) {
            const F y = __shfl_sync(0xffffffffu, y0[r], q) * ri;
            if (lane == q) y0[r] = y;
            else if (lane > q) y0[r] = fma(l0, y, y0[r]);
            y1[r] = fma(l1, y, y1[r]);
          }
        }
#pragma unroll 8
        for (int q = 32; q < 64; q++) {
          const F l1 = lane > q - 32 ? -T[q * LD + lane + 32] : (F)0, ri = rinv[q];
#pragma unroll
          for (int r = 0; r < NR; r++) {
            const F y = __shfl_sync(0xffffffffu, y1[r], q - 32) * ri;
            if (lane == q - 32) y1[r] = y;
            else if (lane > q - 32) y1[r] = fma(l1, y, y1[r]);
          }
        }
      } else {
        // L^T(r, q) = L(q, r), at T[q LD + r]
#pragma unroll 8
        for (int q = 63; q >= 32; q--) {
          const F l1 = lane < q - 32 ? -T[q * LD + lane + 32] : (F)0, ri = rinv[q];
#pragma unroll
          for (int r = 0; r < NR; r++) {
            const F y = __shfl_sync(0xffffffffu, y1[r], q - 32) * ri;
            if (lane == q - 32) y1[r] = y;
            else if (lane < q - 32) y1[r] = fma(l1, y, y1[r]);
          }
        }
#pragma unroll 8
        for (int q = 32; q < 64; q++) {
          const F l0 = -T[q * LD + lane];
#pragma unroll
          for (int r = 0; r < NR; r++) y0[r] = fma(l0, __shfl_sync(0xffffffffu, y1[r], q - 32), y0[r]);
        }
#pragma unroll 8
        for (int q = 31; q >= 0; q--) {
          const F l0 = lane < q ? -T[q * LD + lane] : (F)0, ri = rinv[q];
#pragma unroll
          for (int r = 0; r < NR; r++) {
            const F y = __shfl_sync(0xffffffffu, y0[r], q) * ri;
            if (lane == q) y0[r] = y;
            else if (lane < q) y0[r] = fma(l0, y, y0[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const int c = w + 8 * r;
        if (s != withhold) {
          publish(xo + ((size_t)lane * P + c) * NW, y0[r]);
          publish(xo + ((size_t)(lane + 32) * P + c) * NW, y1[r]);
        }
        if (c < p) {
          X[(size_t)s * SL + lane + (size_t)(c0 + c) * ld] = (double)y0[r];
          X[(size_t)s * SL + lane + 32 + (size_t)(c0 + c) * ld] = (double)y1[r];
        }
      }
    }
    __syncthreads();
  }
}

template <typename F, int P>
emu_status sweeps(emu_ctx *ctx, const emu_mat *L, double *X, long ldx, int nrhs) {
  const int nb = L->nb, NT = L->nt, nslab = NT * (nb / SL), groups = (nrhs + P - 1) / P;
  const int LD = sizeof(F) == 4 ? LDA : LDD;
  const int smem = (int)((2 * SL * LD + SL * P + SL) * sizeof(F));
  static std::atomic<uint64_t> attr_f{0}, attr_b{0};
  EMU_CUDA_TRY(ctx, smem_limit_once(attr_f, ctx->device, (const void *)k_sweep<F, P, false>, smem));
  EMU_CUDA_TRY(ctx, smem_limit_once(attr_b, ctx->device, (const void *)k_sweep<F, P, true>, smem));
  // per sweep: a group's tagged values and, in one more word, its ticket; all
  // zero.  As many groups at a time as the workspace holds, fewer where the
  // device does not have that much.
  const size_t gw = (size_t)nslab * SL * P * (sizeof(F) / 4), unit = 2 * (gw + 1) * sizeof(unsigned long long);
  int some = (int)std::max<size_t>(1, std::min<size_t>(groups, kSweepWorkspace / unit));
  unsigned long long *ws = nullptr;
  cudaError_t e = cudaMallocAsync(&ws, some * unit, ctx->stream);
  while (e == cudaErrorMemoryAllocation && some > 1) {
    cudaGetLastError();
    some = (some + 1) / 2;
    e = cudaMallocAsync(&ws, some * unit, ctx->stream);
  }
  if (e != cudaSuccess) return emu_cuda_fail(ctx, e, "triangular sweeps");
  const size_t xw = some * gw, words = some * (gw + 1);
  const unsigned char *cls = L->state == MAT_FACTOR64 ? nullptr : L->d_cls;
  const long long wait = ctx->sweep_wait > 0 ? ctx->sweep_wait : kSweepWaitCycles;
  for (int g = 0; g < groups && e == cudaSuccess; g += some) {
    const dim3 grid((unsigned)std::min(nslab, (sizeof(F) == 4 ? 2 : 1) * ctx->sm_count),
                    (unsigned)std::min(some, groups - g));
    double *Xg = X + (size_t)g * P * ldx;
    const int left = nrhs - g * P;
    e = cudaMemsetAsync(ws, 0, some * unit, ctx->stream);
    if (e != cudaSuccess) break;
    k_sweep<F, P, false><<<grid, 256, smem, ctx->stream>>>(L->t64, L->t32, cls, nb, NT, nslab, Xg, ldx, left, ws,
                                                           reinterpret_cast<int *>(ws + xw), ctx->d_status, wait,
                                                           ctx->sweep_withhold);
    k_sweep<F, P, true><<<grid, 256, smem, ctx->stream>>>(L->t64, L->t32, cls, nb, NT, nslab, Xg, ldx, left,
                                                          ws + words, reinterpret_cast<int *>(ws + words + xw),
                                                          ctx->d_status, wait, ctx->sweep_withhold);
    ctx->launches += 2;
    ctx->host_launches += 2;
    e = cudaGetLastError();
  }
  cudaFreeAsync(ws, ctx->stream);
  return e == cudaSuccess ? EMU_OK : emu_cuda_fail(ctx, e, "triangular sweeps");
}

}  // namespace

emu_status factor_potrs(emu_ctx *ctx, const emu_mat *L, double *X, long ldx, int nrhs) {
  ProfScope ps(ctx, PROF_SOLVE, 2.0 * (double)L->n * L->n * nrhs, 4.0 * (double)L->n * L->n);
  // an earlier factor's failure must not stop the solves with this one
  EMU_CUDA_TRY(ctx, status_clear(ctx));
  if (L->state == MAT_FACTOR64)
    return nrhs <= 4 ? sweeps<double, 4>(ctx, L, X, ldx, nrhs) : sweeps<double, 16>(ctx, L, X, ldx, nrhs);
  return nrhs <= 4    ? sweeps<float, 4>(ctx, L, X, ldx, nrhs)
         : nrhs <= 16 ? sweeps<float, 16>(ctx, L, X, ldx, nrhs)
                      : sweeps<float, 32>(ctx, L, X, ldx, nrhs);
}
