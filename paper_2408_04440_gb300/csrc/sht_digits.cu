// sht_digits.cu -- the inverse and forward spherical-harmonic transforms of
// emulate.cu with their sums as exact digit products on the tensor cores
// (gemm_f64.h).  On the FP64 pipe (1.2 TFLOP/s) the sums of the inverse
// transform at L = 128 (256 steps, 129 x 256 grid) took 4.6 ms, those of the
// forward one at L = 90 (100 steps, 181 x 360) 5.4 ms; a digit product does 45.
//
// Inverse: per order m the Legendre sums A_m, B_m as one product over the
// degrees for all time steps and rings, then one product with the table of
// cos / sin (m p_j).
// Forward: one product with that table over the longitudes; then, as the
// coefficient is linear in the ring values v of its order,
//   f_lm = sum_i G_lm(i) v(i),  G_lm(i) = sum_i' W(i, i') lam_lm(i'),
// W = the quadratic form Re sum_q sum_q' kappa_q(i) I(q + q') kappa_q'(i') of
// the circle coefficients kappa (|q| < L) and I(k) = int_0^pi e^{ikt} sin t dt,
// which depends on the parity of m only.  G is one product per parity, the
// coefficients one per order.  (Forming S_lmq and contracting it with the
// circle coefficients of every step and order took two FP64 passes of
// Q = 2 L - 1 terms per ring and degree.)
#include <climits>
#include <cmath>

#include "digits.cuh"
#include "sht_digits.h"

namespace {

using gemm64::NS;

// Coefficients of the normalised Legendre recursion (k_legendre, emulate.cu):
// ca = a_lm, cr = a_lm / a_{l-1,m} at the pair's place, cq[q] = -sqrt((2q+1)/(2q)).
__global__ void k_leg_coef(int L, double *__restrict__ ca, double *__restrict__ cr, double *__restrict__ cq) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
  if (l >= L) return;
  if (m == 0) cq[l] = l > 0 ? -sqrt((2.0 * l + 1.0) / (2.0 * l)) : 1.0;
  if (l < m + 2) return;
  const double a = sqrt((4.0 * l * l - 1.0) / ((double)l * l - (double)m * m)), l1 = l - 1.0;
  const double ap = l == m + 2 ? sqrt(2.0 * m + 3.0) : sqrt((4.0 * l1 * l1 - 1.0) / (l1 * l1 - (double)m * m));
  const size_t p = (size_t)m * L - (size_t)m * (m - 1) / 2 + (l - m);
  ca[p] = a;
  cr[p] = a / ap;
}

// lam[pos * ntheta + i], pos the pair's place: order by order, or (parity)
// order_pos.  One thread per (order, ring); a step of the recursion is two
// dependent FP64 operations (with a division and a square root in the loop the
// table took 330 us at L = 128).
__global__ void k_legendre_fast(int L, int ntheta, int parity, const double *__restrict__ ca,
                                const double *__restrict__ cr, const double *__restrict__ cq,
                                double *__restrict__ lam) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
  if (i >= ntheta) return;
  double s, c;
  sincos(M_PI * (double)i / (double)(ntheta - 1), &s, &c);
  double pmm = 0.28209479177387814;  // 1 / sqrt(4 pi)
  for (int q = 1; q <= m; q++) pmm *= cq[q] * s;
  if (m > 0) pmm *= 1.4142135623730951;
  const size_t p = (size_t)m * L - (size_t)m * (m - 1) / 2;
  const double *a = ca + p - m, *r = cr + p - m;
  double *out = lam + (size_t)ntheta * (parity ? gemm64::order_pos(L, m) : p) + i;
  out[0] = pmm;
  if (m + 1 >= L) return;
  double p0 = pmm, p1 = sqrt(2.0 * m + 3.0) * c * pmm;
  out[ntheta] = p1;
#pragma unroll 4
  for (int l = m + 2; l < L; l++) {
    const double v = fma(a[l], c * p1, -(r[l] * p0));
    out[(size_t)(l - m) * ntheta] = v;
    p0 = p1;
    p1 = v;
  }
}

// Digits of scale * cos / sin (m p_j), p_j = 2 pi j / nphi.  BYJ: row j, K =
// 2 m + {0, 1} (kpad columns); else rows 2 m + {0, 1}, K = j.  All rows carry
// the exponent e (scale < 2^e).
template <bool BYJ>
__global__ void k_trig_digits(int L, int nphi, double scale, int e, int kpad, size_t plane, uint16_t *__restrict__ d,
                              int *__restrict__ exps) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  const int m = BYJ ? x : y, j = BYJ ? y : x;
  if (x >= (BYJ ? kpad / 2 : kpad)) return;
  double s = 0.0, c = 0.0;
  if (m < L && j < nphi) {
    sincospi(2.0 * (double)(((long)m * j) % nphi) / (double)nphi, &s, &c);
    s *= scale;
    c *= scale;
  }
  if (BYJ) {
    gemm64::write_digits2(c, s, e, d + (size_t)j * kpad + 2 * m, plane);
    if (m == 0) exps[j] = e + gemm64::kExpBias;
  } else {
    gemm64::write_digits(c, e, d + (size_t)(2 * m) * kpad + j, plane);
    gemm64::write_digits(s, e, d + (size_t)(2 * m + 1) * kpad + j, plane);
    if (j == 0) exps[2 * m] = exps[2 * m + 1] = e + gemm64::kExpBias;
  }
}

struct SrcBase {
  uint16_t *digits;
  int *exps, *flag;
  size_t plane;
};
// Coefficients: batch (time step, sign, block of 32 orders), rows = its orders,
// K = the degrees from the block's first.
struct CoefSrc : SrcBase {
  const double *f;
  long ldf, ktot;
  int L, T, MB, rpad;
  __device__ int m0(int b) const { return b % MB * 32; }
  __device__ int sgn(int b) const { return b / MB % 2; }
  __device__ int rows(int b) const { return min(32, L - m0(b)); }
  __device__ int nk(int b) const { return L - m0(b); }
  __device__ int kpad(int b) const { return gemm64::order_k(L, m0(b)); }
  __device__ double load(int b, int r, int k) const {
    const int m = m0(b) + r;
    const long l = m0(b) + k;
    if (l < m || (sgn(b) && m == 0)) return 0.0;
    return f[(long)(b / MB / 2) * ldf + l * l + l + (sgn(b) ? -m : m)];
  }
  __device__ int row(int b) const { return sgn(b) * T + b / MB / 2; }
  __device__ size_t dst(int b, int r) const { return (size_t)row(b) * ktot + gemm64::order_koff(L, m0(b) + r); }
  __device__ size_t e(int b, int r) const { return (size_t)(m0(b) + r) * rpad + row(b); }
};
// Legendre table, order by order: batch m, rows = rings, K = the degrees from
// the block's first.
struct LamSrc : SrcBase {
  const double *lam;
  long ktot;
  int L, ntheta, cpad;
  __device__ int rows(int) const { return ntheta; }
  __device__ int nk(int m) const { return L - m / 32 * 32; }
  __device__ int kpad(int m) const { return gemm64::order_k(L, m); }
  __device__ double load(int m, int r, int k) const {
    const int l = m / 32 * 32 + k;
    return l < m ? 0.0 : lam[((size_t)m * L - (size_t)m * (m - 1) / 2 + (l - m)) * ntheta + r];
  }
  __device__ size_t dst(int m, int r) const { return (size_t)r * ktot + gemm64::order_koff(L, m); }
  __device__ size_t e(int m, int r) const { return (size_t)m * cpad + r; }
};
// x[b * sb + r * sr + k * sk] to row b * db + r * dr.
struct StridedSrc : SrcBase {
  const double *x;
  long sb, sr, sk, db, dr;
  int nrows, k, kp;
  __device__ int rows(int) const { return nrows; }
  __device__ int nk(int) const { return k; }
  __device__ int kpad(int) const { return kp; }
  __device__ double load(int b, int r, int q) const { return x[b * sb + r * sr + q * sk]; }
  __device__ size_t e(int b, int r) const { return (size_t)(b * db + r * dr); }
  __device__ size_t dst(int b, int r) const { return e(b, r) * kp; }
};
// Ring sums by order: batch m, rows (sign, time step), K = rings.
struct RingSrc : SrcBase {
  const double *cs;
  long R;
  int T, ntheta, kp, rpad;
  __device__ int rows(int) const { return 2 * T; }
  __device__ int nk(int) const { return ntheta; }
  __device__ int kpad(int) const { return kp; }
  __device__ double load(int m, int r, int q) const {
    const int s = r / T, t = r - s * T;
    return cs[(long)t * ntheta + q + R * (2 * m + s)];
  }
  __device__ size_t e(int m, int r) const { return (size_t)m * rpad + r; }
  __device__ size_t dst(int m, int r) const { return e(m, r) * kp; }
};
// Rows of the pairs, even orders (b = 0) or odd ones: x[r * sr + k * sk].
struct PairSrc : SrcBase {
  const double *x;
  long sr, sk;
  int odd0, n0, n1, ntheta, kp;
  __device__ int rows(int b) const { return b ? n1 : n0; }
  __device__ int nk(int) const { return ntheta; }
  __device__ int kpad(int) const { return kp; }
  __device__ double load(int b, int r, int q) const { return x[(b * odd0 + r) * sr + q * sk]; }
  __device__ size_t e(int b, int r) const { return (size_t)b * odd0 + r; }
  __device__ size_t dst(int b, int r) const { return e(b, r) * kp; }
};

// W of the forward transform.  With M = 2 N, N = ntheta - 1, the circle
// coefficients of ring i are (even orders) w_i cos(2 pi q i / M) / M, w = 2
// inside and 1 at the poles, and (odd orders) -i 2 sin(2 pi q i / M) / M inside
// and cos(2 pi q i / M) / M at the poles.  Folding q and q' to q, q' >= 0 with
// Re I(k) = 2 / (1 - k^2) for even k:
//   even:  J(q, q') = 2 I(q+q') + 2 I(q-q') (half of it where one is 0, a quarter where both are)
//   odd, inside x inside: 2 I(q-q') - 2 I(q+q') on the sines;
//   odd, pole x pole: as even; odd, pole x inside: only Im I(+-1) = +-pi/2 is
//   left and telescopes to (2 pi / M^2) sin(2 pi (L-1) i' / M), times (-1)^L at
//   the south pole.
__global__ void k_w_tables(int M, int L, double *__restrict__ cm, double *__restrict__ ir) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < M) {
    double s, c;
    sincospi(2.0 * (double)r / (double)M, &s, &c);
    cm[2 * r] = c;
    cm[2 * r + 1] = s;
  }
  if (r < 2 * L) ir[r] = r % 2 ? 0.0 : 2.0 / (1.0 - (double)r * r);
}
// P[p][q][i] = sum_q' J(q, q') kappa_q'(i), q' of q's parity (kappa without its 1 / M).
__global__ void k_w_left(int L, int ntheta, int M, const double *__restrict__ cm, const double *__restrict__ ir,
                         double *__restrict__ P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y, odd = blockIdx.z;
  if (i >= ntheta) return;
  double acc = 0.0;
  const int step = (int)(2L * i % M);
  int q2 = q & 1, r = q2 ? i % M : 0;
  for (; q2 < L; q2 += 2) {
    const double jp = ir[q + q2], jm = ir[abs(q - q2)];
    double J = odd ? 2.0 * (jm - jp) : 2.0 * (jp + jm);
    if (!odd) J *= (q == 0 ? 0.5 : 1.0) * (q2 == 0 ? 0.5 : 1.0);
    acc = fma(J, cm[2 * r + odd], acc);
    r += step;
    if (r >= M) r -= M;
  }
  P[((size_t)odd * L + q) * ntheta + i] = acc * (i == 0 || i == ntheta - 1 ? 1.0 : 2.0);
}
__global__ void k_w(int L, int ntheta, int M, const double *__restrict__ cm, const double *__restrict__ P,
                    double *__restrict__ W) {
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y, odd = blockIdx.z, N = ntheta - 1;
  if (i2 >= ntheta) return;
  const bool pole = i == 0 || i == N, pole2 = i2 == 0 || i2 == N;
  const double invM = 1.0 / (double)M;
  double v;
  if (odd && pole != pole2) {
    const int in = pole ? i2 : i, at = pole ? i : i2;
    v = L < 2 ? 0.0
              : 6.283185307179586 * invM * invM * cm[2 * (int)((long)(L - 1) * in % M) + 1] *
                    (at == 0 || L % 2 == 0 ? 1.0 : -1.0);
  } else {
    const int par = odd && !pole ? 1 : 0;  // poles of odd orders: the cosine form
    const double *p = P + (size_t)par * L * ntheta + i2;
    double acc = 0.0;
    int r = 0;
    for (int q = 0; q < L; q++) {
      acc = fma(cm[2 * r + par], p[(size_t)q * ntheta], acc);
      r += i;
      if (r >= M) r -= M;
    }
    v = acc * (pole ? 1.0 : 2.0) * invM * invM;
  }
  W[((size_t)odd * ntheta + i) * ntheta + i2] = v;
}

int pad(long x, int m) { return (int)((x + m - 1) / m * m); }

struct Parts {
  size_t off = 0;
  size_t add(size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  }
};

template <bool KFAST, class S>
emu_status digits(emu_ctx *ctx, const S &s, int batches, int rows) {
  gemm64::k_source_digits<S, KFAST><<<dim3((unsigned)batches, (unsigned)((rows + 31) / 32)), 256, 0, ctx->stream>>>(s);
  EMU_LAUNCHED(ctx);
  return EMU_OK;
}

emu_status alloc(emu_ctx *ctx, char **p, size_t bytes) {
  const cudaError_t e = cudaMallocAsync((void **)p, bytes, ctx->stream);
  if (e == cudaSuccess) return EMU_OK;
  *p = nullptr;
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? EMU_ENOMEM : emu_cuda_fail(ctx, e, "transform workspace");
}

#define TRY(expr)                     \
  do {                                \
    const emu_status _s = (expr);     \
    if (_s != EMU_OK) return _s;      \
  } while (0)

// Time steps per pass: operands of one pass within 1 GB.
int steps_per_pass(int T, double bytes_per_step) {
  const int most = (int)std::max(1.0, std::min<double>(T, 1073741824.0 / bytes_per_step));
  const int passes = (T + most - 1) / most;
  return (T + passes - 1) / passes;
}

emu_status isht_passes(emu_ctx *ctx, const double *dF, int L, int T, long ldf, int ntheta, int nphi, double *dZ,
                       long ldz, char *b, int Tc, const size_t (&o)[16]) {
  cudaStream_t st = ctx->stream;
  const int Lp = pad(L, 32), MB = Lp / 32, ktot = gemm64::order_koff(L, Lp - 32) + 32 * 32, Kq = pad(2L * L, 32);
  const int cpad = pad(ntheta, gemm64::BN), npj = pad(nphi, gemm64::BN), rpad = pad(2L * Tc, gemm64::BM);
  const long Rp = pad((long)Tc * ntheta, gemm64::BM);
  auto D = [&](int k) { return reinterpret_cast<double *>(b + o[k]); };
  auto U = [&](int k) { return reinterpret_cast<uint16_t *>(b + o[k]); };
  auto I = [&](int k) { return reinterpret_cast<int *>(b + o[k]); };
  double *ca = D(0), *cr = D(1), *cq = D(2), *lam = D(3), *ab = D(4);
  uint16_t *ld = U(5), *fd = U(6), *ad = U(7), *td = U(8);
  int *le = I(9), *fe = I(10), *ae = I(11), *te = I(12), *flag = ctx->d_status + ST_FLAG;
  CUtensorMap ml, mf, ma, mt;
  TRY(gemm64::make_map(ctx, &ml, ld, ktot, (uint64_t)NS * cpad, gemm64::BN));
  TRY(gemm64::make_map(ctx, &mf, fd, ktot, (uint64_t)NS * rpad, gemm64::BM));
  TRY(gemm64::make_map(ctx, &ma, ad, Kq, (uint64_t)NS * Rp, gemm64::BM));
  TRY(gemm64::make_map(ctx, &mt, td, Kq, (uint64_t)NS * npj, gemm64::BN));
  k_leg_coef<<<dim3((L + 127) / 128, L), 128, 0, st>>>(L, ca, cr, cq);
  EMU_LAUNCHED(ctx);
  k_legendre_fast<<<dim3((ntheta + 31) / 32, L), 32, 0, st>>>(L, ntheta, 0, ca, cr, cq, lam);
  EMU_LAUNCHED(ctx);
  k_trig_digits<true><<<dim3((Kq / 2 + 127) / 128, nphi), 128, 0, st>>>(L, nphi, 1.0, 1, Kq, (size_t)npj * Kq, td, te);
  EMU_LAUNCHED(ctx);
  LamSrc ls;
  ls.digits = ld, ls.exps = le, ls.flag = nullptr, ls.plane = (size_t)cpad * ktot;
  ls.lam = lam, ls.ktot = ktot, ls.L = L, ls.ntheta = ntheta, ls.cpad = cpad;
  TRY((digits<false>(ctx, ls, L, ntheta)));
  for (int t0 = 0; t0 < T; t0 += Tc) {
    const int nt = std::min(Tc, T - t0);
    CoefSrc fs;
    fs.digits = fd, fs.exps = fe, fs.flag = flag, fs.plane = (size_t)rpad * ktot;
    fs.f = dF + (long)t0 * ldf, fs.ldf = ldf, fs.ktot = ktot, fs.L = L, fs.T = nt, fs.MB = MB, fs.rpad = rpad;
    TRY((digits<false>(ctx, fs, 2 * nt * MB, 32)));
    gemm64::Region rg;
    rg.L = L, rg.T = nt, rg.ntheta = ntheta, rg.rpad = rpad, rg.cpad = cpad;
    TRY(gemm64::launch_region(ctx, gemm64::SRC_SYN, mf, ml, rg, rpad, cpad, fe, le, ab, nt, ctx->sm_count));
    StridedSrc as;
    as.digits = ad, as.exps = ae, as.flag = flag, as.plane = (size_t)Rp * Kq;
    as.x = ab, as.sb = nt, as.sr = 1, as.sk = (long)nt * ntheta, as.db = 1, as.dr = ntheta;
    as.nrows = nt, as.k = 2 * L, as.kp = Kq;
    TRY((digits<false>(ctx, as, ntheta, nt)));
    gemm64::Region rd;
    rd.rows_valid = nt * ntheta, rd.cols_valid = nphi, rd.nk = Kq, rd.div = ntheta, rd.ld2 = ldz;
    TRY(gemm64::launch_region(ctx, gemm64::SRC_DENSE, ma, mt, rd, (int)Rp, npj, ae, te, dZ + (long)t0 * ldz, ntheta,
                              ctx->sm_count));
  }
  return EMU_OK;
}

emu_status sht_passes(emu_ctx *ctx, const double *dZ, int ntheta, int nphi, int T, long ldz, int L, double *dF,
                      long ldf, char *b, int Tc, const size_t (&o)[24]) {
  cudaStream_t st = ctx->stream;
  const int M = 2 * ntheta - 2, Kj = pad(nphi, 32), Ki = pad(ntheta, 32), nq = pad(2L * L, gemm64::BN);
  const int odd0 = gemm64::order_odd0(L), n0 = ((L + 1) / 2) * L - ((L + 1) / 2) * ((L + 1) / 2 - 1),
            n1 = L * (L + 1) / 2 - n0;
  const int np = odd0 + pad(n1, gemm64::BM), wpad = pad(ntheta, gemm64::BN), rpad = pad(2L * Tc, gemm64::BM);
  const long Rp = pad((long)Tc * ntheta, gemm64::BM);
  auto D = [&](int k) { return reinterpret_cast<double *>(b + o[k]); };
  auto U = [&](int k) { return reinterpret_cast<uint16_t *>(b + o[k]); };
  auto I = [&](int k) { return reinterpret_cast<int *>(b + o[k]); };
  double *ca = D(0), *cr = D(1), *cq = D(2), *lam = D(3), *cm = D(4), *ir = D(5), *P = D(6), *W = D(7), *G = D(8),
         *cs = D(9);
  uint16_t *ld = U(10), *wd = U(11), *gd = U(12), *zd = U(13), *td = U(14), *rd = U(15);
  int *le = I(16), *we = I(17), *ge = I(18), *ze = I(19), *te = I(20), *re = I(21), *flag = ctx->d_status + ST_FLAG;
  CUtensorMap mg, mz, mt, mr;
  TRY(gemm64::make_map(ctx, &mg, gd, Ki, (uint64_t)NS * np, gemm64::BN));
  TRY(gemm64::make_map(ctx, &mz, zd, Kj, (uint64_t)NS * Rp, gemm64::BM));
  TRY(gemm64::make_map(ctx, &mt, td, Kj, (uint64_t)NS * nq, gemm64::BN));
  TRY(gemm64::make_map(ctx, &mr, rd, Ki, (uint64_t)NS * L * rpad, gemm64::BM));
  k_leg_coef<<<dim3((L + 127) / 128, L), 128, 0, st>>>(L, ca, cr, cq);
  EMU_LAUNCHED(ctx);
  k_legendre_fast<<<dim3((ntheta + 31) / 32, L), 32, 0, st>>>(L, ntheta, 1, ca, cr, cq, lam);
  EMU_LAUNCHED(ctx);
  k_w_tables<<<(std::max(M, 2 * L) + 127) / 128, 128, 0, st>>>(M, L, cm, ir);
  EMU_LAUNCHED(ctx);
  k_w_left<<<dim3((ntheta + 63) / 64, L, 2), 64, 0, st>>>(L, ntheta, M, cm, ir, P);
  EMU_LAUNCHED(ctx);
  k_w<<<dim3((ntheta + 63) / 64, ntheta, 2), 64, 0, st>>>(L, ntheta, M, cm, P, W);
  EMU_LAUNCHED(ctx);
  const double wphi = 6.283185307179586 / (double)nphi;
  const int we2 = std::ilogb(wphi) + 1;  // wphi < 2^we2
  k_trig_digits<false><<<dim3((Kj + 127) / 128, L), 128, 0, st>>>(L, nphi, wphi, we2, Kj, (size_t)nq * Kj, td, te);
  EMU_LAUNCHED(ctx);
  PairSrc lp;
  lp.digits = ld, lp.exps = le, lp.flag = nullptr, lp.plane = (size_t)np * Ki;
  lp.x = lam, lp.sr = ntheta, lp.sk = 1, lp.odd0 = odd0, lp.n0 = n0, lp.n1 = n1, lp.ntheta = ntheta, lp.kp = Ki;
  TRY((digits<true>(ctx, lp, 2, n0)));
  // W: rows i of both parities, parity p's digit planes from row p NS wpad on
  for (int p = 0; p < 2; p++) {
    StridedSrc wsrc;
    wsrc.digits = wd + (size_t)p * NS * wpad * Ki, wsrc.exps = we + p * wpad, wsrc.flag = nullptr;
    wsrc.plane = (size_t)wpad * Ki;
    wsrc.x = W + (size_t)p * ntheta * ntheta, wsrc.sb = 0, wsrc.sr = ntheta, wsrc.sk = 1, wsrc.db = 0, wsrc.dr = 1;
    wsrc.nrows = ntheta, wsrc.k = ntheta, wsrc.kp = Ki;
    TRY((digits<true>(ctx, wsrc, 1, ntheta)));
    CUtensorMap mwp;
    TRY(gemm64::make_map(ctx, &mwp, wd + (size_t)p * NS * wpad * Ki, Ki, (uint64_t)NS * wpad, gemm64::BN));
    CUtensorMap mlp;  // the parity's rows: planes are np rows apart
    TRY(gemm64::make_map(ctx, &mlp, ld + (size_t)(p ? odd0 : 0) * Ki, Ki, (uint64_t)NS * np - (p ? odd0 : 0), gemm64::BM));
    gemm64::Region rw;
    rw.rows_valid = p ? n1 : n0, rw.cols_valid = ntheta, rw.nk = Ki, rw.div = INT_MAX, rw.ld2 = 0;
    if (rw.rows_valid > 0)
      TRY(gemm64::launch_region(ctx, gemm64::SRC_DENSE, mlp, mwp, rw, np, wpad, le + (p ? odd0 : 0), we + p * wpad,
                                G + (p ? odd0 : 0), np, ctx->sm_count));
  }
  PairSrc gp = lp;
  gp.digits = gd, gp.exps = ge, gp.x = G, gp.sr = 1, gp.sk = np;
  TRY((digits<false>(ctx, gp, 2, n0)));
  for (int t0 = 0; t0 < T; t0 += Tc) {
    const int nt = std::min(Tc, T - t0);
    const long R = (long)nt * ntheta;
    StridedSrc zs;
    zs.digits = zd, zs.exps = ze, zs.flag = flag, zs.plane = (size_t)Rp * Kj;
    zs.x = dZ + (long)t0 * ldz, zs.sb = ldz, zs.sr = 1, zs.sk = ntheta, zs.db = ntheta, zs.dr = 1;
    zs.nrows = ntheta, zs.k = nphi, zs.kp = Kj;
    TRY((digits<false>(ctx, zs, nt, ntheta)));
    gemm64::Region rf;
    rf.rows_valid = (int)R, rf.cols_valid = 2 * L, rf.nk = Kj, rf.div = INT_MAX, rf.ld2 = 0;
    TRY(gemm64::launch_region(ctx, gemm64::SRC_DENSE, mz, mt, rf, (int)Rp, nq, ze, te, cs, R, ctx->sm_count));
    RingSrc rs;
    rs.digits = rd, rs.exps = re, rs.flag = flag, rs.plane = (size_t)L * rpad * Ki;
    rs.cs = cs, rs.R = R, rs.T = nt, rs.ntheta = ntheta, rs.kp = Ki, rs.rpad = rpad;
    TRY((digits<true>(ctx, rs, L, 2 * nt)));
    gemm64::Region ra;
    ra.L = L, ra.T = nt, ra.nk = Ki, ra.rpad = rpad;
    TRY(gemm64::launch_region(ctx, gemm64::SRC_ANA, mr, mg, ra, L * rpad, np, re, ge, dF + (long)t0 * ldf, ldf,
                              ctx->sm_count));
  }
  return EMU_OK;
}

// Waits for the transform: EMU_ESTATE when an operand held an infinity or a NaN.
emu_status finish(emu_ctx *ctx, char *blob, emu_status s) {
  cudaError_t e = cudaSuccess;
  if (s == EMU_OK)
    e = cudaMemcpyAsync(ctx->h_status, ctx->d_status, ST_WORDS * sizeof(int), cudaMemcpyDeviceToHost, ctx->stream);
  cudaFreeAsync(blob, ctx->stream);
  if (s != EMU_OK) return s;
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return emu_cuda_fail(ctx, e, "transform");
  s = status_timed_out(ctx);
  return s != EMU_OK ? s : ctx->h_status[ST_FLAG] ? EMU_ESTATE : EMU_OK;
}

}  // namespace

emu_status isht_digits(emu_ctx *ctx, const double *dF, int L, int T, long ldf, int ntheta, int nphi, double *dZ,
                       long ldz) {
  const size_t npair = (size_t)L * (L + 1) / 2, Lp = pad(L, 32), Kq = pad(2L * L, 32), cpad = pad(ntheta, gemm64::BN),
               npj = pad(nphi, gemm64::BN);
  const double ktot_d = 16.0 * Lp * (Lp + 32.0) / 32.0;  // sum over orders of order_k
  // rings in blocks of 32, and longitudes, count on the second axis of a grid
  if (ntheta > 32 * 65535 || nphi > 65535) return EMU_ENOMEM;
  if (npair * ntheta > (size_t)1 << 31 || 32.0 * ktot_d > 2147483647.0) return EMU_ENOMEM;
  const size_t ktot = (size_t)gemm64::order_koff(L, (int)Lp - 32) + 32 * 32;
  const int Tc = steps_per_pass(T, 2.0 * NS * ((double)ntheta * Kq + 2.0 * ktot) + 16.0 * L * ntheta);
  const size_t rpad = pad(2L * Tc, gemm64::BM), Rp = pad((long)Tc * ntheta, gemm64::BM);
  Parts p;
  size_t o[16] = {};
  o[0] = p.add(npair * 8);
  o[1] = p.add(npair * 8);
  o[2] = p.add((size_t)L * 8);
  o[3] = p.add(npair * ntheta * 8);
  o[4] = p.add((size_t)2 * L * ntheta * Tc * 8);
  o[5] = p.add(NS * cpad * ktot * 2);
  o[6] = p.add(NS * rpad * ktot * 2);
  o[7] = p.add(NS * Rp * Kq * 2);
  o[8] = p.add(NS * npj * Kq * 2);
  o[9] = p.add(L * cpad * 4);
  o[10] = p.add(L * rpad * 4);
  o[11] = p.add(Rp * 4);
  o[12] = p.add(npj * 4);
  char *b = nullptr;
  TRY(alloc(ctx, &b, p.off));
  const emu_status s = isht_passes(ctx, dF, L, T, ldf, ntheta, nphi, dZ, ldz, b, Tc, o);
  return finish(ctx, b, s);
}

emu_status sht_digits(emu_ctx *ctx, const double *dZ, int ntheta, int nphi, int T, long ldz, int L, double *dF,
                      long ldf) {
  const size_t Kj = pad(nphi, 32), Ki = pad(ntheta, 32), nq = pad(2L * L, gemm64::BN), M = 2 * ntheta - 2;
  const size_t npair = (size_t)L * (L + 1) / 2, np = npair + 3 * gemm64::BM, wpad = pad(ntheta, gemm64::BN);
  const int Tc = steps_per_pass(T, 2.0 * NS * ((double)ntheta * Kj + 2.0 * L * Ki) + 16.0 * L * ntheta);
  const size_t rpad = pad(2L * Tc, gemm64::BM), Rp = pad((long)Tc * ntheta, gemm64::BM);
  Parts p;
  size_t o[24] = {};
  o[0] = p.add(npair * 8);
  o[1] = p.add(npair * 8);
  o[2] = p.add((size_t)L * 8);
  o[3] = p.add(np * ntheta * 8);
  o[4] = p.add(2 * M * 8);
  o[5] = p.add(2 * (size_t)L * 8);
  o[6] = p.add(2 * (size_t)L * ntheta * 8);
  o[7] = p.add(2 * (size_t)ntheta * ntheta * 8);
  o[8] = p.add(np * ntheta * 8);
  o[9] = p.add((size_t)2 * L * ntheta * Tc * 8);
  o[10] = p.add(NS * np * Ki * 2);
  o[11] = p.add(2 * NS * wpad * Ki * 2);
  o[12] = p.add(NS * np * Ki * 2);
  o[13] = p.add(NS * Rp * Kj * 2);
  o[14] = p.add(NS * nq * Kj * 2);
  o[15] = p.add(NS * L * rpad * Ki * 2);
  o[16] = p.add(np * 4);
  o[17] = p.add(2 * wpad * 4);
  o[18] = p.add((np + gemm64::BN) * 4);
  o[19] = p.add(Rp * 4);
  o[20] = p.add(nq * 4);
  o[21] = p.add(L * rpad * 4);
  char *b = nullptr;
  TRY(alloc(ctx, &b, p.off));
  const emu_status s = sht_passes(ctx, dZ, ntheta, nphi, T, ldz, L, dF, ldf, b, Tc, o);
  return finish(ctx, b, s);
}
