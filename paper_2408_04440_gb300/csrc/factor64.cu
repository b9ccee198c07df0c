// factor64.cu -- the plain FP64 tile Cholesky ("Advancements in Dense Linear
// Algebra") and its draws on the BF16 tensor cores: every product is formed
// from exact digits (gemm_f64.h), so it has FP64 accuracy relative to the
// largest entries of the two rows it multiplies, as the FP64 class of the
// mixed factor has.  For a Cholesky factor those maxima are at most
// sqrt(S_ii) and sqrt(S_jj): the error of an update is within the scaled bound
// n u sqrt(S_ii S_jj) of the factor formed in FP64 arithmetic, with 2^-56 in
// place of u.
//
// Entries of L far below that scale are less accurate relative to themselves
// than FP64 arithmetic makes them: against its own bound, n u (|L| |L|^T)_ij,
// the error reaches 1500 times that on the synthetic covariance (n = 1024, beta =
// 3; the largest relative error of an entry 1e-9 at n = 400) and far more on a
// matrix whose off-diagonal entries span fourteen decades, at the same norm of
// the error.  emu_fp64_arithmetic keeps a context on FP64 sums.
//
// Why: the FP64 pipe does 1.2 TFLOP/s, the 36 digit products of a K step run
// at 45 TFLOP/s of FP64 work.  What stays on the FP64 pipe is the diagonal
// POTRF and the 128-column block solves of the panel.
#include <algorithm>

#include "factor64.h"
#include "gemm_f64.h"
#include "mixed.h"

namespace {

// Panels whose digits may be live at once: the bulk update of panel k reads
// them while panels k + 1 and k + 2 are solved and sliced.  Panel k + 3's POTRF
// waits (through S(k + 2) and G2A(k + 1)) for the bulk stream to have passed
// G2(k), so its digits may take panel k's place.
constexpr int kRing = 3;

__global__ void k_iota(int *p, long n) {
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < n; q += (long)gridDim.x * blockDim.x) p[q] = (int)q;
}

// Stream-ordered workspace; EMU_ENOMEM when it does not fit (the caller then
// takes the FP64 pipe's kernels, which work in place).
emu_status workspace(emu_ctx *ctx, char **p, size_t bytes) {
  const cudaError_t e = cudaMallocAsync((void **)p, bytes, ctx->stream);
  if (e == cudaSuccess) return EMU_OK;
  *p = nullptr;
  if (e != cudaErrorMemoryAllocation) return emu_cuda_fail(ctx, e, "FP64 digit workspace");
  cudaGetLastError();
  return EMU_ENOMEM;
}

struct Plan {
  char *blob = nullptr;
  uint16_t *dig[kRing];
  int *exps[kRing], *tiles;
  gemm64::TrsmPlan tr[2];  // by step parity; one set of block slots, one per tile row below the panel
  CUtensorMap ma[kRing], mb[kRing];
};

emu_status plan_make(emu_ctx *ctx, const emu_mat *A, Plan *P) {
  const size_t nb = A->nb, npad = (size_t)A->nt * nb;
  size_t off = 0;
  auto part = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  };
  const int nring = std::min(kRing, A->nt);
  size_t o_dig[kRing], o_exp[kRing], o_tr[2];
  for (int q = 0; q < nring; q++) {
    o_dig[q] = part(gemm64::NS * npad * nb * sizeof(uint16_t));
    o_exp[q] = part(npad * sizeof(int));
  }
  const size_t o_t = part(A->ntiles * sizeof(int));
  for (int q = 0; q < 2; q++) o_tr[q] = part(gemm64::trsm_plan_bytes(A->nb, A->nt));
  emu_status s = workspace(ctx, &P->blob, off);
  if (s != EMU_OK) return s;
  char *b = P->blob;
  const uint64_t drows = (uint64_t)gemm64::NS * npad;
  for (int q = 0; q < kRing; q++) {
    const int r = q % nring;
    P->dig[q] = reinterpret_cast<uint16_t *>(b + o_dig[r]);
    P->exps[q] = reinterpret_cast<int *>(b + o_exp[r]);
    if (s == EMU_OK) s = gemm64::make_map(ctx, &P->ma[q], P->dig[q], nb, drows, gemm64::BM);
    if (s == EMU_OK) s = gemm64::make_map(ctx, &P->mb[q], P->dig[q], nb, drows, gemm64::BN);
  }
  P->tiles = reinterpret_cast<int *>(b + o_t);
  for (int q = 0; q < 2 && s == EMU_OK; q++) s = gemm64::trsm_plan_init(ctx, &P->tr[q], b + o_tr[q], A->nb, A->nt);
  if (s != EMU_OK) return s;
  k_iota<<<(unsigned)std::min<long>((A->ntiles + 255) / 256, 512), 256, 0, ctx->stream>>>(P->tiles, A->ntiles);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

// SMs the bulk update leaves to the panel work: a bulk CTA fills its SM's
// registers and shared memory, and the block solves are bound by the FP64
// pipes of the SMs they find.  Panel work grows as n nb, the update as n^2, so
// the best count falls with n / nb.  Factor in ms with 16 / 32 / 48 / 64:
//   n =  1600, nb =  128    1.65 / 1.65 / 1.64 / 1.63
//   n =  4096, nb =  256    4.56 / 4.58 / 4.57 / 4.57
//   n = 10000, nb =  512    21.7 / 21.4 / 21.3 / 21.3
//   n = 16384, nb =  512    62.9 / 61.4 / 60.9 / 62.7
//   n = 16384, nb = 1024    66.4 / 66.4 / 66.3 / 65.7
//   n = 40000, nb = 1024     660 /  651 /  682 /  773
//   n = 65536, nb = 1024    2380 / 2480 / 2780 / 3220
// 48 is the best up to n = 20000 or so and loses 5 % at 40000 and 17 % at 65536,
// where a count that follows the ratio of the two kinds of work would pay.
constexpr int kReserved = 48;

emu_status factor_launches(emu_ctx *ctx, emu_mat *A, Plan *P) {
  const int NT = A->nt, nb = A->nb, nJ = nb / gemm64::TW;
  const int npad = NT * nb, rb = nb / gemm64::BM, cb = nb / gemm64::BN;  // row / column blocks per tile
  const size_t te = A->tile_elems;
  const double nb3 = (double)nb * nb * nb;
  cudaStream_t user = ctx->stream;
  // streams and dependencies of the lookahead schedule (as the mixed factor's):
  //   crit: POTRF(k) -> TRSM(k+1, k) -> S(k), the update of tile (k+1, k+1)
  //   mid : TRSM(i >= k+2, k) -> G1(k), the update of column k+1 below it
  //   bulk: G2A(k), the update of column k+2, then G2(k), columns >= k+3
  const int EV = 5;
  enum { E_P = 0, E_T1 = 1, E_T = 2, E_G1 = 3, E_G2 = 4 };
  emu_status s = mixed_sched_streams(ctx, EV * NT + 2);
  if (s != EMU_OK) return s;
  auto ev = [&](int k, int w) { return ctx->sched_ev[EV * k + w]; };
  cudaEvent_t ev_start = ctx->sched_ev[EV * NT], ev_end = ctx->sched_ev[EV * NT + 1];
  EMU_CUDA_TRY(ctx, cudaEventRecord(ev_start, user));
  for (cudaStream_t q : {ctx->crit, ctx->mid, ctx->bulk}) EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(q, ev_start, 0));

  // tiles (i, k), i0 <= i < NT (count n): X = A L_kk^{-T} in place, then the digits of X
  auto trsm = [&](int k, int i0, int n) -> emu_status {
    if (n <= 0) return EMU_OK;
    const double *Lkk = A->t64 + tile_index(k, k, NT) * te;
    {
      ProfScope ps(ctx, PROF_TRSM64, n * nb3, 16.0 * n * te, 36.0 * n * nb3 * (nJ - 1) / nJ);
      emu_status e = gemm64::trsm_plan_solve(ctx, P->tr[k & 1], A->t64, nb, P->tiles + tile_index(i0, k, NT), n, Lkk,
                                             i0 - (k + 1));
      if (e != EMU_OK) return e;
    }
    return gemm64::launch_panel_digits(ctx, A->t64, NT, nb, i0 * nb, n * nb, k, 1, 0, P->exps[k % kRing], 0, npad, nb,
                                       P->dig[k % kRing]);
  };
  // update of tile columns [j0, j1), tile rows [i0, i1), lower blocks, by panel k
  auto update = [&](int k, int i0, int i1, int j0, int j1, int ctas) -> emu_status {
    if (i0 >= i1 || j0 >= j1) return EMU_OK;
    double f = 0.0;
    for (int j = j0; j < j1; j++) f += 2.0 * nb3 * (i1 - std::max(i0, j));
    ProfScope ps(ctx, PROF_UPDATE64, f, 12.0 * f / nb, 36.0 * f);
    gemm64::Region rg;
    rg.NT = NT;
    rg.nb = nb;
    rg.r_lo = i0 * rb;
    rg.r_hi = i1 * rb;
    rg.c_lo = j0 * cb;
    rg.c_hi = j1 * cb;
    const int q = k % kRing;
    return gemm64::launch_region(ctx, gemm64::SRC_SYRK, P->ma[q], P->mb[q], rg, npad, npad, P->exps[q], P->exps[q],
                                 A->t64, nb, ctas);
  };
  for (int k = 0; k < NT && s == EMU_OK; k++) {
    const long tkk = tile_index(k, k, NT);
    // ---- critical stream
    ctx->stream = ctx->crit;
    if ((s = launch_potrf64_tile(ctx, A, k)) != EMU_OK) break;
    if (k + 1 == NT) break;
    if ((s = gemm64::trsm_plan_prep(ctx, P->tr[k & 1], A->t64 + tkk * te, nb)) != EMU_OK) break;
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev(k, E_P), ctx->crit));
    if (k > 0) EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->crit, ev(k - 1, E_G1), 0));
    if ((s = trsm(k, k + 1, 1)) != EMU_OK) break;
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev(k, E_T1), ctx->crit));
    if (k > 0) EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->crit, ev(k - 1, E_G2), 0));
    if ((s = update(k, k + 1, k + 2, k + 1, k + 2, ctx->sm_count)) != EMU_OK) break;
    // ---- panel stream
    ctx->stream = ctx->mid;
    EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->mid, ev(k, E_P), 0));
    if ((s = trsm(k, k + 2, NT - k - 2)) != EMU_OK) break;
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev(k, E_T), ctx->mid));
    EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->mid, ev(k, E_T1), 0));
    if (k > 0) EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->mid, ev(k - 1, E_G2), 0));
    if ((s = update(k, k + 2, NT, k + 1, k + 2, ctx->sm_count)) != EMU_OK) break;
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev(k, E_G1), ctx->mid));
    // ---- bulk stream
    ctx->stream = ctx->bulk;
    EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->bulk, ev(k, E_T), 0));
    const int ctas = std::max(1, ctx->sm_count - kReserved);
    if ((s = update(k, k + 2, NT, k + 2, k + 3, ctas)) != EMU_OK) break;
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev(k, E_G2), ctx->bulk));
    if ((s = update(k, k + 3, NT, k + 3, NT, ctas)) != EMU_OK) break;
  }
  ctx->stream = user;
  // the context stream waits for all three, also after an error
  for (cudaStream_t q : {ctx->mid, ctx->bulk, ctx->crit}) {
    EMU_CUDA_TRY(ctx, cudaEventRecord(ev_end, q));
    EMU_CUDA_TRY(ctx, cudaStreamWaitEvent(user, ev_end, 0));
  }
  return s;
}

}  // namespace

bool factor64_digits_supports(const emu_mat *A) { return A->nb % gemm64::BM == 0 && A->nb % gemm64::TW == 0; }

emu_status factor64_digits(emu_ctx *ctx, emu_mat *A) {
  emu_status s = potrf_dag_prepare(ctx, A->nb);
  if (s != EMU_OK) return s;
  Plan P;
  s = plan_make(ctx, A, &P);
  if (s == EMU_OK) s = factor_launches(ctx, A, &P);
  if (P.blob) cudaFreeAsync(P.blob, ctx->stream);
  return s == EMU_OK ? launch_tril_diag(ctx, A) : s;
}

// Y = L Z: the rows of L in groups whose digits fit the arena, each row with
// one exponent over all its tiles, so that a row block's products with a
// sample block are summed exactly over the whole row and written once.  The
// FP64 TRMM ran (n / 64)(s / 64) CTAs over the FP64 pipe: 1.07 ms for 64
// samples at n = 1024 (16 CTAs), 22 ms for 100 at n = 10000.
emu_status sample64_digits(emu_ctx *ctx, const emu_mat *L, const double *Z, long ldz, int s, double *Y, long ldy) {
  const int NT = L->nt, nb = L->nb;
  const long npad = (long)NT * nb;
  const int s_pad = (s + gemm64::BN - 1) / gemm64::BN * gemm64::BN;
  constexpr size_t kArena = (size_t)2 << 30;
  const int g = (int)std::max<size_t>(1, std::min<size_t>(NT, kArena / (gemm64::NS * sizeof(uint16_t) * npad * nb)));
  const long grows = (long)g * nb;
  size_t off = 0;
  auto part = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  };
  const size_t o_a = part(gemm64::NS * grows * npad * sizeof(uint16_t)),
               o_z = part((size_t)gemm64::NS * s_pad * npad * sizeof(uint16_t)), o_ae = part(grows * sizeof(int)),
               o_ze = part(s_pad * sizeof(int));
  char *b = nullptr;
  emu_status st = workspace(ctx, &b, off);
  if (st != EMU_OK) return st;
  uint16_t *ad = reinterpret_cast<uint16_t *>(b + o_a), *zd = reinterpret_cast<uint16_t *>(b + o_z);
  int *ae = reinterpret_cast<int *>(b + o_ae), *ze = reinterpret_cast<int *>(b + o_ze);
  CUtensorMap ma, mz;
  st = gemm64::make_map(ctx, &ma, ad, npad, (uint64_t)gemm64::NS * grows, gemm64::BM);
  if (st == EMU_OK) st = gemm64::make_map(ctx, &mz, zd, npad, (uint64_t)gemm64::NS * s_pad, gemm64::BN);
  if (st == EMU_OK) st = gemm64::launch_slice_cols(ctx, Z, ldz, s, s_pad, (int)npad, ze, zd);
  for (int i0 = 0; i0 < NT && st == EMU_OK; i0 += g) {
    const int i1 = std::min(NT, i0 + g);
    st = gemm64::launch_panel_digits(ctx, L->t64, NT, nb, i0 * nb, (i1 - i0) * nb, 0, -1, i0 * nb, ae, i0 * nb, grows,
                                     npad, ad);
    if (st != EMU_OK) break;
    const double f = ((double)i1 * (i1 + 1) - (double)i0 * (i0 + 1)) * nb * nb * s;
    ProfScope ps(ctx, PROF_TRMM64, f, 0.0, 36.0 * f);
    gemm64::Region rg;
    rg.NT = NT;
    rg.nb = nb;
    rg.r_lo = i0 * (nb / gemm64::BM);
    rg.r_hi = (std::min(i1 * nb, L->n) + gemm64::BM - 1) / gemm64::BM;
    rg.c_lo = 0;
    rg.c_hi = s_pad / gemm64::BN;
    rg.a_row0 = i0 * nb;
    rg.rows_valid = L->n;
    rg.cols_valid = s;
    st = gemm64::launch_region(ctx, gemm64::SRC_TRMM, ma, mz, rg, (int)grows, s_pad, ae, ze, Y, ldy, ctx->sm_count);
  }
  cudaFreeAsync(b, ctx->stream);
  return st;
}
