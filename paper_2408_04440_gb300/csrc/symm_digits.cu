// symm_digits.cu -- S X for a symmetric covariance in packed FP64 tiles, up to
// 16 right-hand sides at a time, as exact digit products on the BF16 tensor
// cores (the scheme of gemm_f64.h) with the digits of S cut on the way in.
//
// On the FP64 pipe the product of n = 65536 with 16 columns took 116 ms, all of
// it FP64 issue; its memory traffic is 5 ms (both triangles).  Digits kept in
// memory would cost 16 bytes written and read per entry and use; here eight
// warps cut them from the FP64 tile into the shared-memory operand of the MMAs;
// their integer instructions are then the bound (23 ms at n = 65536, 1.5 ms at
// n = 16384 against 7.3).  A solution refined to its limit is off by 2.9e-15 /
// 8.2e-15 (n = 2116 / 3136, extended precision), with the FP64 pipe's residual
// by 4.4e-15 / 1.6e-14.
//
// Scales.  |S_rc| <= sqrt(S_rr S_cc) < 2^(d_r + d_c), d the halved exponent of
// the diagonal rounded up, and within a tile |S_rc| is at most the tile's norm:
// entry (r, c) of tile t is cut relative to 2^(d_r + d_c + t), t <= 0 from the
// norm, so neither a graded diagonal nor a weakly correlated tile costs digits.
// X_c 2^d_c is cut relative to the largest of its chunk of 128 or 256 rows;
// chunk sums are exact, rounded once to FP64 and added in FP64.  A matrix that
// breaks the bound (not positive semidefinite, an infinity or a NaN) sets a
// flag, and the caller takes the FP64 pipe.
//
// Products with p + q <= 8 are kept, one group more than the factor's updates
// take: a row's exponent here covers a whole tile, whose other rows may be
// larger.  What is left out is the last digits' truncation.
//
// Warp roles (512 threads, one CTA per SM, persistent over row blocks x column
// ranges): warp 0 TMA loads of X's digits; warp 1 MMA issuer: digit p of S
// meets the digits q <= 8 - p of X in one MMA of N = 16 per digit, into the
// group accumulators p + q (144 TMEM columns, double-buffered by chunk); warps
// 4..7 epilogue; warps 8..15 cut S.
#include <algorithm>

#include "digits.cuh"
#include "symm_digits.h"
#include "tc.cuh"

namespace symm_digits {
namespace {

using gemm64::kExpBias;
using gemm64::kExpMin;
using gemm64::NS;

constexpr int BM = 128, BK = 32, STAGES = 3;
constexpr int A_SL = BM * BK * 2;                // one digit plane of S: 8 KB
constexpr int B_BYTES = NS * NR * BK * 2;        // X's digits: 128 rows, 8 KB
constexpr int STAGE_BYTES = NS * A_SL + B_BYTES;
constexpr int RING_BYTES = STAGES * STAGE_BYTES;
constexpr int SMEM_BYTES = RING_BYTES + 256 + 1024;
constexpr int NTHREADS = 512, EPI0 = 4, GEN0 = 8, NGEN = 8;
constexpr int NG = NS + 1;                       // groups p + q = 0 .. 8
constexpr uint32_t TMEM_COLS = 512, ACC_COLS = NG * NR;  // two buffers

struct Shared {
  uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2], done;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Shared) <= 256, "barrier block");

__device__ inline bool failed(const int *st) { return *((volatile const int *)st) != DEV_OK; }
__device__ inline void raise_timeout(Shared *sh, int *status) {
  sh->abort = 1;
  if (atomicCAS(&status[ST_CODE], DEV_OK, DEV_TIMEOUT) == DEV_OK) status[ST_AUX] = 7;
}

// Exponents d of the rows and the least one per tile row: one CTA per tile row.
__global__ void k_row_scales(const double *__restrict__ t64, int nb, int NT, int *__restrict__ dexp,
                             int *__restrict__ dmin, int *__restrict__ flag) {
  __shared__ int red[32];
  const int i = blockIdx.x;
  const double *D = t64 + (size_t)tile_index(i, i, NT) * nb * nb;
  int least = 1 << 20;
  for (int r = threadIdx.x; r < nb; r += blockDim.x) {
    const double v = D[(size_t)r * (nb + 1)];
    const unsigned long long m = gemm64::mag_bits(v);
    if (!(v > 0.0) || ((m >> 52) & 0x7ff) == 0x7ff) *flag = 1;
    const int e = m > 0 ? gemm64::biased_exp(m) - kExpBias : 0;  // v < 2^e
    const int d = (e + 1) >> 1;
    dexp[(size_t)i * nb + r] = d;
    least = min(least, d);
  }
  for (int o = 16; o > 0; o >>= 1) least = min(least, __shfl_xor_sync(0xffffffffu, least, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = least;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (int)(blockDim.x >> 5); q++) least = min(least, red[q]);
    dmin[i] = least;
  }
}
__global__ void k_tile_scales(const double *__restrict__ tnorm, int NT, long ntiles, const int *__restrict__ dmin,
                              int *__restrict__ texp) {
  const int j = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < j || i >= NT) return;
  const long t = tile_index(i, j, NT);
  const unsigned long long m = gemm64::mag_bits(tnorm[t]);
  int e = 0;
  // a diagonal tile's padding is not in its norm
  if (i > j && m > 0) e = min(0, gemm64::biased_exp(m) - kExpBias - dmin[i] - dmin[j]);
  texp[t] = e;
}

// Digits of X_c 2^d_c, one CTA per chunk of ck rows: warp w takes right-hand
// sides 2 w and 2 w + 1 of the group.
__global__ void __launch_bounds__(256)
    k_x_digits(const double *__restrict__ X, long npad, int nrhs, int c0, int ck, const int *__restrict__ dexp,
               int *__restrict__ xexp, uint16_t *__restrict__ xdig) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long r0 = (long)blockIdx.x * ck;
  for (int u = 0; u < 2; u++) {
    const int c = 2 * w + u;
    double v[8];
    unsigned long long m = 0;
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int r = lane + 32 * q;
      v[q] = 0.0;
      if (r < ck && c0 + c < nrhs) {
        const int d = dexp[r0 + r];
        v[q] = X[r0 + r + (size_t)(c0 + c) * npad] * gemm64::exp2i(max(-1000, min(1000, d)));
      }
      m = max(m, gemm64::mag_bits(v[q]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int eb = m > 0 ? gemm64::biased_exp(m) : 0;
    if (lane == 0) xexp[(size_t)blockIdx.x * NR + c] = eb;
    const int e = max(eb - kExpBias, kExpMin);
#pragma unroll
    for (int q = 0; q < 8; q++)
      if (lane + 32 * q < ck)
        gemm64::write_digits(v[q], e, xdig + (size_t)c * npad + r0 + lane + 32 * q, (size_t)NR * npad);
  }
}

__global__ void __launch_bounds__(NTHREADS, 1)
    k_symm_digits(const __grid_constant__ CUtensorMap bmap, const double *__restrict__ t64, int nb, int NT, int ck,
                  int nz, const int *__restrict__ dexp, const int *__restrict__ texp, const int *__restrict__ xexp,
                  double *__restrict__ part, long npad, int *__restrict__ flag, int *status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw), padb = ((raw + 1023u) & ~1023u) - raw, ring_addr = raw + padb;
  uint8_t *ring = smem_raw + padb;
  Shared *sh = reinterpret_cast<Shared *>(ring + RING_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblk = (int)(npad / BM), nitems = nblk * nz, nchunks = (int)(npad / ck), kst = ck / BK;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; s++) {
      tc::mbar_init(&sh->full[s], NGEN + 1);
      tc::mbar_init(&sh->empty[s], 1);
    }
    for (int b = 0; b < 2; b++) {
      tc::mbar_init(&sh->tfull[b], 1);
      tc::mbar_init(&sh->tempty[b], 128);
    }
    tc::mbar_init(&sh->done, 1);
    sh->abort = failed(status) ? 1 : 0;
    tc::fence_barrier_init();
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
  // item it: row block it / nz, chunks [q0, q1) of column range it % nz
  auto range = [&](int it, int &q0, int &q1) {
    const int z = it % nz;
    q0 = (int)((long)nchunks * z / nz);
    q1 = (int)((long)nchunks * (z + 1) / nz);
  };

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = *abort == 0;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        int q0, q1;
        range(it, q0, q1);
        for (int kc = q0 * kst; kc < q1 * kst; kc++) {
          if (!tc::mbar_wait(&sh->empty[stage], phase ^ 1u, abort)) {
            raise_timeout(sh, status);
            ok = false;
            break;
          }
          tc::mbar_arrive_expect_tx(&sh->full[stage], (uint32_t)B_BYTES);
          tc::tma_load_2d(ring + stage * STAGE_BYTES + NS * A_SL, &bmap, &sh->full[stage], kc * BK, 0);
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      // every stage's last load must have landed before the CTA exits
      for (int s = 0; s < STAGES; s++) tc::mbar_wait_inflight(&sh->full[s], (s < stage) ? phase : (phase ^ 1u));
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0, chunk = 0;
      bool ok = *abort == 0;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        int q0, q1;
        range(it, q0, q1);
        for (int q = q0; q < q1 && ok; q++, chunk++) {
          const uint32_t buf = chunk & 1u, acc = tmem + buf * ACC_COLS;
          if (!tc::mbar_wait(&sh->tempty[buf], ((chunk >> 1) & 1u) ^ 1u, abort)) {
            raise_timeout(sh, status);
            ok = false;
            break;
          }
          tc::fence_after_sync();
          for (int kc = 0; kc < kst; kc++) {
            if (!tc::mbar_wait(&sh->full[stage], phase, abort)) {
              raise_timeout(sh, status);
              ok = false;
              break;
            }
            tc::fence_after_sync();
            const uint32_t st = ring_addr + stage * STAGE_BYTES;
            const uint64_t a0 = tc::smem_desc(st, 16, 512, tc::kSwizzle64B);
            const uint64_t b0 = tc::smem_desc(st + NS * A_SL, 16, 512, tc::kSwizzle64B);
#pragma unroll
            for (int ks = 0; ks < BK / 16; ks++)
#pragma unroll
              for (int p = 0; p < NS; p++) {
                const uint64_t ad = tc::desc_add(a0, p * A_SL + ks * 32), bd = tc::desc_add(b0, ks * 32);
                const uint32_t more = kc > 0 || ks > 0 ? 1u : 0u;
                // digits q = 0 .. 8 - p of X (7 at most); digit 0 of S starts
                // groups 0 .. 7, digit 1 with X's digit 7 starts group 8
                const int nq = p == 0 ? NS : p == 1 ? NS - 1 : NG - p;
                tc::mma_f16(acc + (uint32_t)(p * NR), ad, bd, tc::idesc_f32acc(1u /*BF16*/, BM, NR * nq),
                            p > 0 ? 1u : more);
                if (p == 1)
                  tc::mma_f16(acc + (uint32_t)(NS * NR), ad, tc::desc_add(bd, (NS - 1) * NR * BK * 2),
                              tc::idesc_f32acc(1u /*BF16*/, BM, NR), more);
              }
            tc::mma_commit(&sh->empty[stage]);
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (ok) tc::mma_commit(&sh->tfull[buf]);
        }
      }
      tc::mma_commit(&sh->done);
      tc::mbar_wait_inflight(&sh->done, 0);
    }
  } else if (warp >= EPI0 && warp < GEN0) {
    const int row = (warp & 3) * 32 + lane;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t chunk = 0;
    bool ok = *abort == 0;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
      int q0, q1;
      range(it, q0, q1);
      const long gr = (long)(it / nz) * BM + row;
      const int i = (int)(gr / nb), dr = dexp[gr];
      double acc[NR];
#pragma unroll
      for (int c = 0; c < NR; c++) acc[c] = 0.0;
      for (int q = q0; q < q1; q++, chunk++) {
        const uint32_t buf = chunk & 1u;
        const int j = (int)((long)q * ck / nb);
        const int s = dr + texp[i >= j ? tile_index(i, j, NT) : tile_index(j, i, NT)];
        if (!tc::mbar_wait(&sh->tfull[buf], (chunk >> 1) & 1u, abort)) {
          raise_timeout(sh, status);
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll
        for (int h = 0; h < NR / 2; h++) {
          uint32_t r[NS][2], r8[2];
#pragma unroll
          for (int g = 0; g < NS; g++)
            tc::tmem_ld_32x32b_x2(tlane + buf * ACC_COLS + (uint32_t)(g * NR + 2 * h), r[g]);
          tc::tmem_ld_32x32b_x2(tlane + buf * ACC_COLS + (uint32_t)(NS * NR + 2 * h), r8);
          tc::tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 2; x++) {
            // group 8 in units of 2^-63 (rounded), then the others on top
            const long long t8 = (__float2int_rn(__uint_as_float(r8[x])) + 64) >> 7;
            long long hi = t8 >> 32;
            unsigned lo = (unsigned)t8;
            gemm64::fold_groups(r, x, hi, lo);
            acc[2 * h + x] += gemm64::fixed_scaled(hi, lo, s + gemm64::exp_of(xexp, (long)q * NR + 2 * h + x));
          }
        }
        tc::fence_before_sync();
        tc::mbar_arrive(&sh->tempty[buf]);
      }
      if (!ok) break;
      double2 *o = reinterpret_cast<double2 *>(part + ((size_t)(it % nz) * npad + gr) * NR);
#pragma unroll
      for (int c = 0; c < NR / 2; c++) o[c] = make_double2(acc[2 * c], acc[2 * c + 1]);
    }
  } else if (warp >= GEN0) {
    // ------------------------------------------------------- cutting S
    // row m of the block, sixteen columns (two 16-byte pieces of each plane)
    const int gw = warp - GEN0, m = (gw & 3) * 32 + lane, kg = (gw >> 2) * 2;
    int stage = 0;
    uint32_t phase = 0;
    bool ok = *abort == 0, bad = false;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
      int q0, q1;
      range(it, q0, q1);
      const long gr = (long)(it / nz) * BM + m;
      const int i = (int)(gr / nb), mr = (int)(gr % nb), dr = dexp[gr];
      double v[16], nx[16];
      auto load = [&](int kc, double (&x)[16]) {  // columns 16 (kg / 2) .. of stage kc
        const long col = (long)kc * BK + 8 * kg;
        const int j = (int)(col / nb), k = (int)(col % nb);
        if (i >= j) {
          const double *T = t64 + (size_t)tile_index(i, j, NT) * nb * nb + mr + (size_t)k * nb;
#pragma unroll
          for (int u = 0; u < 16; u++) x[u] = __ldg(T + (size_t)u * nb);
        } else {
          const double2 *T =
              reinterpret_cast<const double2 *>(t64 + (size_t)tile_index(j, i, NT) * nb * nb + k + (size_t)mr * nb);
#pragma unroll
          for (int u = 0; u < 8; u++) {
            const double2 t = __ldg(T + u);
            x[2 * u] = t.x;
            x[2 * u + 1] = t.y;
          }
        }
      };
      load(q0 * kst, v);
      for (int kc = q0 * kst; kc < q1 * kst; kc++) {
        const long col = (long)kc * BK + 8 * kg;
        const int j = (int)(col / nb);
        const int te = dr + texp[i >= j ? tile_index(i, j, NT) : tile_index(j, i, NT)];
        int dc[16];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const int4 d4 = __ldg(reinterpret_cast<const int4 *>(dexp + col) + u);
          dc[4 * u] = d4.x;
          dc[4 * u + 1] = d4.y;
          dc[4 * u + 2] = d4.z;
          dc[4 * u + 3] = d4.w;
        }
        if (kc + 1 < q1 * kst) load(kc + 1, nx);
        if (!tc::mbar_wait(&sh->empty[stage], phase ^ 1u, abort)) {
          raise_timeout(sh, status);
          ok = false;
          break;
        }
        uint8_t *st = ring + stage * STAGE_BYTES + m * 64;
#pragma unroll
        for (int g = 0; g < 2; g++) {
          uint32_t w4[NS][4];
#pragma unroll
          for (int u = 0; u < 4; u++) {
            uint32_t d0[NS], d1[NS];
            const int x0 = 8 * g + 2 * u;
            const int e0 = te + dc[x0], e1 = te + dc[x0 + 1];
            // |x| < 2^e, else the bound failed
            const unsigned long long m0 = gemm64::mag_bits(v[x0]), m1 = gemm64::mag_bits(v[x0 + 1]);
            bad |= (int)((m0 >> 52) & 0x7ff) - 1022 > e0 || (int)((m1 >> 52) & 0x7ff) - 1022 > e1;
            gemm64::field_digit_bits(gemm64::to_fixed(v[x0], e0), d0);
            gemm64::field_digit_bits(gemm64::to_fixed(v[x0 + 1], e1), d1);
#pragma unroll
            for (int p = 0; p < NS; p++) w4[p][u] = d0[p] | (d1[p] << 16);
          }
          const uint32_t off = (uint32_t)((kg + g) ^ ((m >> 1) & 3)) << 4;  // 64-byte swizzle
#pragma unroll
          for (int p = 0; p < NS; p++)
            *reinterpret_cast<uint4 *>(st + p * A_SL + off) = make_uint4(w4[p][0], w4[p][1], w4[p][2], w4[p][3]);
        }
        tc::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&sh->full[stage]);
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1u;
        }
#pragma unroll
        for (int u = 0; u < 16; u++) v[u] = nx[u];
      }
    }
    if (bad) *flag = 1;
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, TMEM_COLS);
  }
}

int chunk_of(const emu_mat *S) { return S->nb % 256 == 0 ? 256 : 128; }

struct Offsets {
  size_t dexp, dmin, texp, flag, xexp, xdig, end;
};
Offsets offsets(const emu_mat *S) {
  const size_t npad = (size_t)S->nt * S->nb;
  Offsets o;
  size_t off = 0;
  auto part = [&](size_t b) {
    const size_t q = off;
    off += (b + 255) & ~(size_t)255;
    return q;
  };
  o.dexp = part(npad * sizeof(int));
  o.dmin = part(S->nt * sizeof(int));
  o.texp = part(S->ntiles * sizeof(int));
  o.flag = part(sizeof(int));
  o.xexp = part(npad / chunk_of(S) * NR * sizeof(int));
  o.xdig = part(NS * NR * npad * sizeof(uint16_t));
  o.end = off;
  return o;
}

}  // namespace

Plan shape(const emu_ctx *ctx, const emu_mat *S, int nrhs) {
  Plan P;
  P.groups = (nrhs + NR - 1) / NR;
  const int nblk = (int)((long)S->nt * S->nb / BM), nchunks = (int)((long)S->nt * S->nb / chunk_of(S));
  P.nz = std::max(1, std::min(nchunks, (8 * ctx->sm_count + nblk - 1) / nblk));
  return P;
}

size_t bytes(const emu_mat *S) { return offsets(S).end; }

emu_status init(emu_ctx *ctx, Plan *P, char *base, const emu_mat *S) {
  const Offsets o = offsets(S);
  P->dexp = reinterpret_cast<int *>(base + o.dexp);
  P->dmin = reinterpret_cast<int *>(base + o.dmin);
  P->texp = reinterpret_cast<int *>(base + o.texp);
  P->flag = reinterpret_cast<int *>(base + o.flag);
  P->xexp = reinterpret_cast<int *>(base + o.xexp);
  P->xdig = reinterpret_cast<uint16_t *>(base + o.xdig);
  EMU_CUDA_TRY(ctx, cudaMemsetAsync(P->flag, 0, sizeof(int), ctx->stream));
  k_row_scales<<<S->nt, 256, 0, ctx->stream>>>(S->t64, S->nb, S->nt, P->dexp, P->dmin, P->flag);
  EMU_LAUNCHED(ctx);
  k_tile_scales<<<dim3((S->nt + 127) / 128, S->nt), 128, 0, ctx->stream>>>(S->d_tnorm, S->nt, S->ntiles, P->dmin,
                                                                          P->texp);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status multiply(emu_ctx *ctx, const Plan &P, const emu_mat *S, const double *X, int nrhs, double *part) {
  const long npad = (long)S->nt * S->nb;
  const int ck = chunk_of(S), items = (int)(npad / BM) * P.nz;
  CUtensorMap map;
  emu_status s = gemm64::make_map(ctx, &map, P.xdig, npad, NS * NR, NS * NR);
  if (s != EMU_OK) return s;
  static std::atomic<uint64_t> attr{0};
  EMU_CUDA_TRY(ctx, smem_limit_once(attr, ctx->device, (const void *)k_symm_digits, SMEM_BYTES));
  for (int g = 0; g < P.groups; g++) {
    k_x_digits<<<(unsigned)(npad / ck), 256, 0, ctx->stream>>>(X, npad, nrhs, g * NR, ck, P.dexp, P.xexp, P.xdig);
    EMU_LAUNCHED(ctx);
    k_symm_digits<<<std::min(items, ctx->sm_count), NTHREADS, SMEM_BYTES, ctx->stream>>>(
        map, S->t64, S->nb, S->nt, ck, P.nz, P.dexp, P.texp, P.xexp, part + (size_t)g * P.nz * npad * NR, npad, P.flag,
        ctx->d_status);
    EMU_LAUNCHED(ctx);
  }
  return EMU_OK;
}

}  // namespace symm_digits
