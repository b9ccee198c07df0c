"""Timed workloads of the library, each one pass through the public Python API.

A case is a dict of plain values whose "kind" says which part of the emulator
it stands for:

  fp64      covariance build, plain FP64 tile Cholesky, draws; the factor is exported
  mixed     covariance build, adaptive-precision Cholesky, draws (norm rule or a band map)
  fit       empirical covariance of residual vectors, adaptive Cholesky, both exported
  classfmt  class-format covariance build, factor, draws
  sample    draws from a factor in hand
  refine    refined solve against a covariance and a factor in hand
  emulate   draws -> VAR recursion -> inverse SHT -> emulations on the grid
  analyse   forward SHT of gridded fields
  batch     many covariances of uneven bandlimit factored and sampled in one call

``exact`` is the same result from plain torch in 64 bits (no code of this
library).
"""
import math

import torch

import paper_2408_04440_gb300 as E

MASKS = (0b01011, 0b11011, 0b01111)  # FP64/FP32/BF16, with E4M3, with TF32
SIGMA_EXP, NUGGET = 1.5, 1e-8


def listed():
    return [
        # the small plain FP64 configuration (n = 1024, 128-wide tiles): launches and latency count
        dict(name="fp64_L32", kind="fp64", L=32, nb=128, beta=4.0, samples=64),
        # plain FP64 reference factor of a ragged n = 10000 covariance, as users check mixed results with
        dict(name="fp64_L100", kind="fp64", L=100, nb=512, beta=8.0, samples=100),
        # the headline step: n = 16384 at eps = 1e-8, 256 draws
        dict(name="mixed_L128", kind="mixed", L=128, nb=512, beta=8.0, eps=1e-8, mask=0b01011, band=0, samples=256),
        # the large configuration with all formats: n = 65536 at eps = 1e-6
        dict(name="mixed_L256", kind="mixed", L=256, nb=1024, beta=12.0, eps=1e-6, mask=0b11011, band=0, samples=16),
        # fitting from data: residuals of an odd bandlimit (n = 5041, ragged tiles) and fewer residuals than a multiple
        dict(name="fit_L71", kind="fit", L=71, nb=256, beta=5.0, m=6001, eps=1e-6, mask=0b11011),
        # class-format storage of covariances too large for FP64 tiles, here at n = 22500
        dict(name="classfmt_L150", kind="classfmt", L=150, nb=1024, beta=10.0, eps=1e-6, mask=0b11011, samples=64),
        # repeated use of one factor: a large ensemble of draws
        dict(name="sample_L128", kind="sample", L=128, nb=512, beta=8.0, eps=1e-8, mask=0b01011, samples=1024),
        # one right-hand side against a small ragged covariance (kriging, likelihoods), default tolerance
        dict(name="refine_L60", kind="refine", L=60, nb=256, beta=5.0, eps=1e-8, mask=0b01011, nrhs=1, tol=1e-14),
        # the large refined solve: n = 65536, 16 right-hand sides to 1e-12
        dict(name="refine_L256", kind="refine", L=256, nb=1024, beta=12.0, eps=1e-6, mask=0b11011, nrhs=16, tol=1e-12),
        # monthly emulations, 256 steps on a 129 x 256 grid
        dict(name="emulate_L128", kind="emulate", L=128, T=256, ntheta=129, nphi=256, P=3, K=3, tau=12.0),
        # forward transform of 100 fields on the one-degree grid
        dict(name="analyse_L90", kind="analyse", L=90, T=100, ntheta=181, nphi=360),
        # a batch of small regional covariances, bandlimits 8..64
        dict(name="batch_256", kind="batch", count=256, lmin=8, lmax=64, draws=3, nb=256, eps=1e-8, samples=256),
    ]


def _logint(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(("fp64", "mixed", "fit", "classfmt", "sample", "refine", "emulate", "analyse", "batch"))
    if kind == "fp64":
        return dict(kind=kind, L=_logint(rng, 12, 100), nb=rng.choice((128, 192, 256, 512)),
                    beta=round(rng.uniform(3.0, 9.0), 2), samples=_logint(rng, 1, 300))
    if kind in ("mixed", "sample"):
        L = _logint(rng, 24, 160)
        c = dict(kind=kind, L=L, nb=rng.choice((256, 512)) if L < 100 else rng.choice((512, 1024)),
                 beta=round(rng.uniform(4.0, 12.0), 2), eps=rng.choice((1e-6, 1e-8)), mask=rng.choice(MASKS),
                 samples=_logint(rng, 1, 1024))
        if kind == "mixed":
            c["band"] = rng.choice((0, 0, 0, 1, 2, 3))
        return c
    if kind == "fit":
        L = _logint(rng, 16, 90)
        return dict(kind=kind, L=L, nb=rng.choice((256, 512)), beta=round(rng.uniform(3.0, 6.0), 2),
                    m=L * L + _logint(rng, 100, 6000), eps=rng.choice((1e-6, 1e-8)), mask=rng.choice(MASKS))
    if kind == "classfmt":
        L = _logint(rng, 48, 150)
        return dict(kind=kind, L=L, nb=rng.choice((256, 512)) if L < 100 else rng.choice((512, 1024)),
                    beta=round(rng.uniform(4.0, 12.0), 2), eps=rng.choice((1e-6, 1e-8)), mask=rng.choice(MASKS[:2]),
                    samples=_logint(rng, 1, 256))
    if kind == "refine":
        L = _logint(rng, 20, 128)
        return dict(kind=kind, L=L, nb=rng.choice((256, 512)), beta=round(rng.uniform(3.0, 8.0), 2),
                    eps=rng.choice((1e-6, 1e-8)), mask=rng.choice(MASKS), nrhs=_logint(rng, 1, 40), tol=1e-14)
    if kind == "emulate":
        L = _logint(rng, 12, 128)
        return dict(kind=kind, L=L, T=_logint(rng, 1, 300), ntheta=L + rng.randint(1, L), nphi=2 * L + rng.randint(0, L),
                    P=rng.randint(0, 3), K=rng.randint(0, 4), tau=rng.choice((12.0, 365.0)))
    if kind == "analyse":
        L = _logint(rng, 12, 110)
        return dict(kind=kind, L=L, T=_logint(rng, 1, 200), ntheta=L + rng.randint(1, L), nphi=2 * L + rng.randint(0, 2 * L))
    lmin = rng.randint(4, 12)
    return dict(kind="batch", count=_logint(rng, 8, 200), lmin=lmin, lmax=rng.randint(lmin + 10, 64),
                draws=rng.randint(10, 10000), nb=256, eps=rng.choice((0.0, 1e-6, 1e-8)), samples=_logint(rng, 1, 256))


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _beta(case, seed):
    """The correlation length, a little different for each seed."""
    return case["beta"] * (1.0 + 0.02 * (((seed * 2654435761) % 4093) / 4093.0 - 0.5))


def _colmajor(t):
    return t.t().contiguous().t()


def _degrees(L):
    l = torch.arange(L, device="cuda").repeat_interleave(2 * torch.arange(L, device="cuda") + 1)
    return l, torch.arange(L * L, device="cuda") - l * l - l


def _residuals(case, seed):
    """m residual vectors whose spread falls with the degree and whose neighbouring orders are correlated."""
    L, m = case["L"], case["m"]
    l, _ = _degrees(L)
    x = torch.randn(m, L * L, dtype=torch.float64, device="cuda", generator=_gen(seed))
    x = x + 0.6 * torch.roll(x, 1, 1) + 0.3 * torch.roll(x, 2, 1)
    return (x * (1.0 + l.double()) ** -SIGMA_EXP).t()


def _field(case, seed):
    """Band-limited fields plus a little unresolved noise on the grid, one column per time step."""
    L, T, nth, nph = case["L"], case["T"], case["ntheta"], case["nphi"]
    g = _gen(seed)
    l, _ = _degrees(L)
    F = torch.randn(L * L, T, dtype=torch.float64, device="cuda", generator=g) * ((1.0 + l.double()) ** -1.5)[:, None]
    Z = _synthesis(F, L, nth, nph)
    return _colmajor(Z + 0.01 * torch.randn(Z.shape, dtype=torch.float64, device="cuda", generator=g))


def _emulation_inputs(case, seed):
    L, T, P, K = case["L"], case["T"], case["P"], case["K"]
    G = case["ntheta"] * case["nphi"]
    g = _gen(seed)

    def u(*shape):
        return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)

    l, _ = _degrees(L)
    Xi = torch.randn(T, L * L, dtype=torch.float64, device="cuda", generator=g) * (1.0 + l.double()) ** -SIGMA_EXP
    Phi = ((u(P, L * L) * torch.tensor([0.6, 0.2, 0.1], dtype=torch.float64, device="cuda")[:P, None]).t()
           if P else None)
    nyears = max(1, math.ceil(T / case["tau"]))
    return dict(Xi=Xi.t(), Phi=Phi, beta0=270.0 + 30.0 * u(G), beta1=u(G), beta2=u(G), rho=0.9 * u(G),
                A=u(K, G) if K else None, B=u(K, G) if K else None, x=torch.cumsum(0.1 * u(nyears + 1), 0),
                sigma=0.5 + u(G), v=0.1 * u(G))


def _batch_params(case, seed):
    """Bandlimits fixed by the case, correlation lengths by the seed."""
    import random

    r, q = random.Random(case["draws"]), random.Random(seed)
    return [(r.randint(case["lmin"], case["lmax"]), q.uniform(2.0, 8.0)) for _ in range(case["count"])]


class _State(dict):
    """What a program holds between calls; its context is closed with it."""

    def __del__(self):
        try:
            self["ctx"].close()
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    st = _State(case=case, seed=seed, ctx=E.Context(0))
    if kind == "fit":
        st["Xi"] = _residuals(case, seed)
    elif kind in ("sample", "refine"):
        ctx, beta = st["ctx"], _beta(case, seed)
        A = E.emu_cov_build(ctx, case["L"], beta, case["nb"])
        if kind == "refine":
            st["S"] = A
            A = E.emu_mat_clone(ctx, A)
            st["B"] = torch.randn(case["nrhs"], case["L"] ** 2, dtype=torch.float64, device="cuda",
                                  generator=_gen(seed)).t()
        E.emu_potrf_mp(ctx, A, eps=case["eps"], prec_mask=case["mask"])
        st["A"] = A
    elif kind == "emulate":
        st.update(_emulation_inputs(case, seed))
    elif kind == "analyse":
        st["Z"] = _field(case, seed)
    elif kind == "batch":
        st["params"] = _batch_params(case, seed)
        s = case["samples"]
        sizes = [p[0] ** 2 for p in st["params"]]
        st["flat"] = torch.empty(sum(sizes) * s, dtype=torch.float64, device="cuda")
        st["Y"] = [q.view(s, n).t() for n, q in zip(sizes, st["flat"].split([n * s for n in sizes]))]
    return st


def run(st):
    case, ctx, seed = st["case"], st["ctx"], st["seed"]
    kind = case["kind"]
    if kind == "fp64":
        A = E.emu_cov_build(ctx, case["L"], _beta(case, seed), case["nb"])
        E.emu_potrf_mp(ctx, A)
        return {"L": E.emu_mat_export(ctx, A), "Y": E.emu_sample(ctx, A, case["samples"], seed)}
    if kind == "mixed":
        A = E.emu_cov_build(ctx, case["L"], _beta(case, seed), case["nb"])
        E.emu_potrf_mp(ctx, A, eps=case["eps"], prec_mask=case["mask"], band=case["band"])
        return E.emu_sample(ctx, A, case["samples"], seed)
    if kind == "fit":
        A, _ = E.emu_cov_from_residuals(ctx, st["Xi"], case["nb"])
        U = E.emu_mat_export(ctx, A)
        E.emu_potrf_mp(ctx, A, eps=case["eps"], prec_mask=case["mask"])
        return {"U": U, "L": E.emu_mat_export(ctx, A)}
    if kind == "classfmt":
        A = E.emu_cov_build_classfmt(ctx, case["L"], _beta(case, seed), case["nb"], eps=case["eps"],
                                     prec_mask=case["mask"])
        E.emu_potrf_mp(ctx, A, eps=case["eps"], prec_mask=case["mask"])
        return E.emu_sample(ctx, A, case["samples"], seed)
    if kind == "sample":
        return E.emu_sample(ctx, st["A"], case["samples"], seed)
    if kind == "refine":
        X, _ = E.emu_solve_refine(ctx, st["A"], st["S"], st["B"], tol=case["tol"], raise_on_error=False)
        return X
    if kind == "emulate":
        F = E.emu_var_recursion(ctx, st["Xi"], st["Phi"])
        Zs = E.emu_isht(ctx, F, case["L"], case["ntheta"], case["nphi"])
        Y = E.emu_emulate_grid(ctx, Zs, case["tau"], st["beta0"], st["beta1"], st["beta2"], st["rho"], st["A"], st["B"],
                               st["x"], st["sigma"], st["v"], seed)
        return {"F": F, "Zs": Zs, "Y": Y}
    if kind == "analyse":
        return E.emu_sht(ctx, st["Z"], case["L"], case["ntheta"], case["nphi"])
    E.emu_batch_potrf_sample(ctx, st["params"], nb=case["nb"], eps=case["eps"], nsamples=case["samples"], seed=seed,
                             out_Y=st["Y"])
    return st["flat"]


# --------------------------------------------------------------------- work
def work(case):
    """Algorithmic bytes (inputs read once, results written once) and flops of one pass."""
    kind = case["kind"]
    if kind == "batch":
        ns = [p[0] ** 2 for p in _batch_params(case, 0)]
        return {"bytes": 8.0 * case["samples"] * sum(ns),
                "flops": sum(n**3 / 3.0 + float(n) * n * case["samples"] for n in ns)}
    L = case["L"]
    n = float(L * L)
    if kind == "fp64":
        return {"bytes": 8.0 * (n * n + n * case["samples"]), "flops": n**3 / 3 + n * n * case["samples"]}
    if kind in ("mixed", "classfmt"):
        return {"bytes": 8.0 * n * case["samples"], "flops": n**3 / 3 + n * n * case["samples"]}
    if kind == "fit":
        return {"bytes": 8.0 * (n * case["m"] + 2 * n * n), "flops": n * n * case["m"] + n**3 / 3}
    if kind == "sample":
        # the factor is kept in tiles of 2 to 8 bytes per entry: at least 2 bytes of its lower triangle
        return {"bytes": n * n + 8.0 * n * case["samples"], "flops": n * n * case["samples"]}
    if kind == "refine":
        # one residual against the FP64 lower triangle and one solve with the factor, at least
        return {"bytes": 4.0 * n * n + n * n + 16.0 * n * case["nrhs"], "flops": 4.0 * n * n * case["nrhs"]}
    T, G = case["T"], float(case["ntheta"] * case["nphi"])
    # per time step: Legendre sums over l for every order and ring, then one FFT per ring
    transform = T * (2.0 * n * case["ntheta"] + 2.5 * G * math.log2(case["nphi"]))
    if kind == "emulate":
        return {"bytes": 8.0 * T * (2 * n + 2 * G), "flops": transform + 2.0 * n * T * case["P"] + 30.0 * G * T}
    return {"bytes": 8.0 * T * (n + G), "flops": transform}


# -------------------------------------------------------------------- exact
def _covariance(L, beta):
    l, m = _degrees(L)
    l, m = l.double(), m.double()
    s = (1.0 + l) ** -SIGMA_EXP
    S = (l[:, None] - l[None, :]).square_()
    S += (m[:, None] - m[None, :]).square_()
    S.sqrt_().div_(-beta).exp_()
    S.mul_(s[:, None]).mul_(s[None, :])
    S.diagonal().add_(NUGGET * float(S.diagonal().max()))
    return S


def _normals(n, cols, seed, stream=0):
    """Standard normals of Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) and Box-Muller, rows 2p and 2p+1 a pair."""
    M32 = (1 << 32) - 1

    def mul(a, c):  # (high, low) words of the product of two 32-bit values, in 64-bit integers
        lo = a * (c & 0xFFFF)
        hi = a * (c >> 16)
        low = (lo + ((hi & 0xFFFF) << 16))
        return (hi >> 16) + (low >> 32), low & M32

    p = torch.arange((n + 1) // 2, device="cuda")[:, None].expand(-1, cols)
    c = [p & M32, p >> 32, torch.arange(cols, device="cuda")[None, :].expand(p.shape), torch.full_like(p, stream)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    a = (c[0] << 21) | (c[1] >> 11)
    b = (c[2] << 21) | (c[3] >> 11)
    r = torch.sqrt(-2.0 * torch.log((a.double() + 1.0) * 2.0**-53))
    th = (2.0 * math.pi) * (b.double() * 2.0**-53)
    return torch.stack((r * torch.cos(th), r * torch.sin(th)), 1).reshape(-1, cols)[:n]


def _legendre(L, ntheta, m):
    """Real orthonormal Y_lm without its longitude factor at the ntheta colatitudes, rows l = m .. L-1."""
    th = math.pi * torch.arange(ntheta, dtype=torch.float64, device="cuda") / (ntheta - 1)
    s, c = torch.sin(th), torch.cos(th)
    pmm = torch.full_like(th, 0.5 / math.sqrt(math.pi))
    for q in range(1, m + 1):
        pmm = pmm * (-math.sqrt((2 * q + 1) / (2 * q))) * s
    rows = [pmm]
    if m + 1 < L:
        rows.append(math.sqrt(2 * m + 3) * c * pmm)
    prev = math.sqrt(2 * m + 3)
    for l in range(m + 2, L):
        a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
        rows.append(a * (c * rows[-1] - rows[-2] / prev))
        prev = a
    return torch.stack(rows) * (math.sqrt(2.0) if m else 1.0)


def _angles(nphi, m):
    j = (torch.arange(nphi, device="cuda") * m) % nphi
    a = 2.0 * math.pi * j.double() / nphi
    return torch.cos(a), torch.sin(a)


def _synthesis(F, L, ntheta, nphi):
    """Grid values (i + j ntheta, t) of real-form coefficients F[l^2 + l + m, t]."""
    T = F.shape[1]
    Z = torch.zeros(nphi, ntheta, T, dtype=torch.float64, device="cuda")
    for m in range(L):
        lam = _legendre(L, ntheta, m)
        l = torch.arange(m, L, device="cuda")
        c, s = _angles(nphi, m)
        Z += c[:, None, None] * (lam.t() @ F[l * l + l + m])[None]
        if m:
            Z += s[:, None, None] * (lam.t() @ F[l * l + l - m])[None]
    return Z.reshape(nphi * ntheta, T)


def _analysis(Z, L, ntheta, nphi):
    """Coefficients by longitude DFT, extension of each order to the circle in colatitude, |q| < L Fourier terms."""
    T = Z.shape[1]
    Z = Z.reshape(nphi, ntheta, T)
    M, Q = 2 * ntheta - 2, 2 * L - 1
    i = torch.arange(M, device="cuda")
    src = torch.where(i < ntheta, i, M - i)
    q = torch.arange(-(L - 1), L, device="cuda")
    ang = 2.0 * math.pi * ((q[:, None] * i[None, :]) % M).double() / M
    four = torch.complex(torch.cos(ang), -torch.sin(ang)) / M  # Q x M
    k = (q[:, None] + q[None, :]).double()
    even = (k.long() % 2) == 0
    I = torch.complex(torch.where(even, 2.0 / (1.0 - k * k), torch.zeros_like(k)),
                      torch.where(k.abs() == 1, 0.5 * math.pi * k, torch.zeros_like(k)))
    F = torch.empty(L * L, T, dtype=torch.float64, device="cuda")
    for m in range(L):
        ext = torch.where((i >= ntheta) & bool(m % 2), -1.0, 1.0).double()
        c, s = _angles(nphi, m)
        lam = (_legendre(L, ntheta, m)[:, src] * ext).to(torch.complex128)
        S = (lam @ four.t()) @ I  # (L - m) x Q
        l = torch.arange(m, L, device="cuda")
        for trig, sign in ((c, 1), (s, -1))[: 2 if m else 1]:
            g = torch.einsum("j,jit->it", trig, Z) * (2.0 * math.pi / nphi)
            K = four @ (g[src] * ext[:, None]).to(torch.complex128)
            F[l * l + l + sign * m] = (S @ K).real
    return F


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for b, (L, beta) in enumerate(_batch_params(case, seed)):
            Y = torch.linalg.cholesky(_covariance(L, beta)) @ _normals(L * L, case["samples"], seed, b)
            out.append(Y.t().reshape(-1))
        return torch.cat(out)
    L = case["L"]
    if kind == "emulate":
        x = _emulation_inputs(case, seed)
        T, P, tau = case["T"], case["P"], case["tau"]
        F = x["Xi"].clone()
        for t in range(T):
            for p in range(min(P, t)):
                F[:, t] += x["Phi"][:, p] * F[:, t - 1 - p]
        Zs = _synthesis(F, L, case["ntheta"], case["nphi"])
        Y = torch.empty_like(Zs)
        e = _normals(Zs.shape[0], T, seed)
        D, year = x["x"][0].expand(Zs.shape[0]), 1
        for t in range(1, T + 1):
            while year < math.ceil(t / tau):
                D = (1.0 - x["rho"]) * x["x"][year] + x["rho"] * D
                year += 1
            mt = x["beta0"] + x["beta1"] * x["x"][year] + x["beta2"] * D
            for h in range(case["K"]):
                w = 2.0 * math.pi * t * (h + 1) / tau
                mt = mt + x["A"][h] * math.cos(w) + x["B"][h] * math.sin(w)
            Y[:, t - 1] = mt + x["sigma"] * (Zs[:, t - 1] + x["v"] * e[:, t - 1])
        return {"F": F, "Zs": Zs, "Y": Y}
    if kind == "analyse":
        return _analysis(_field(case, seed), L, case["ntheta"], case["nphi"])
    if L > 165:
        return None  # minutes of 64-bit Cholesky
    if kind == "fit":
        X = _residuals(case, seed)
        U = X @ X.t() / X.shape[1]
        return {"U": torch.tril(U), "L": torch.linalg.cholesky(U)}
    if kind == "refine":
        C = torch.linalg.cholesky(_covariance(L, _beta(case, seed)))
        B = torch.randn(case["nrhs"], L * L, dtype=torch.float64, device="cuda", generator=_gen(seed)).t()
        return torch.cholesky_solve(B.contiguous(), C)
    C = torch.linalg.cholesky(_covariance(L, _beta(case, seed)))
    Y = C @ _normals(L * L, case["samples"], seed)
    return {"L": C, "Y": Y} if kind == "fp64" else Y
