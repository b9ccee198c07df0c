"""Refined solves entry by entry: the residual takes every entry of the covariance whole, so a solution's entry that hangs
on covariances far below their tile's largest is as accurate, relative to itself, as the others.  And the smallest
matrices, one 64-wide tile among them."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    return E


@pytest.fixture(scope="module")
def ctx(E):
    c = E.Context(0)
    yield c
    c.close()


def _dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t()


@pytest.mark.parametrize("n,nb,r", [(2304, 256, 4), (2048, 256, 2), (3100, 512, 17)])
@pytest.mark.parametrize("small", [1e-9, 1e-12])
def test_small_covariances_beside_a_large_one(E, ctx, n, nb, r, small):
    """The unit matrix but for tile (5, 1) = M: one entry 0.5, the others about `small`.  With b zero outside tile row 1,
    x_5 = -M x_1 and x_1 = b_1 + M^T M x_1, here in extended precision.  Errors of x_5 relative to |M| |x_1|: n u of the
    FP64 residual, plus what the FP32 factor leaves after a correction, the square of nb 2^-24; four times that."""
    rng = np.random.default_rng(n + r)
    M = small * rng.standard_normal((nb, nb))
    M[7, :] = 0.0
    M[:, 9] = 0.0
    M[7, 9] = 0.5
    lo, hi = slice(nb, 2 * nb), slice(5 * nb, 6 * nb)
    C = np.eye(n)
    C[hi, lo], C[lo, hi] = M, M.T
    B = np.zeros((n, r))
    B[lo] = rng.standard_normal((nb, r))
    S = E.emu_mat_import(ctx, _dev(C), nb)
    A = E.emu_mat_clone(ctx, S)
    E.emu_potrf_mp(ctx, A, eps=1e-10, prec_mask=0b00011)
    X, info = E.emu_solve_refine(ctx, A, S, _dev(B), tol=1e-15, raise_on_error=False)
    assert info.iters >= 1
    X = X.cpu().numpy()
    Ml, x1 = M.astype(np.longdouble), B[lo].astype(np.longdouble)
    for _ in range(60):  # the norm of M^T M is a quarter
        x1 = B[lo] + Ml.T @ (Ml @ x1)
    off = np.abs(X[hi] + Ml @ x1) / np.maximum(np.abs(Ml) @ np.abs(x1), 1e-300)
    assert off[np.arange(nb) != 7].max() <= 4 * (n * 2.0**-53 + (nb * 2.0**-24) ** 2)


@pytest.mark.parametrize("L,nb,r", [(1, 64, 1), (5, 64, 2), (8, 64, 17), (9, 64, 3), (8, 192, 1), (15, 192, 5)])
def test_smallest_matrices(E, ctx, L, nb, r):
    import torch

    n = L * L
    S = E.emu_cov_build(ctx, L, 4.0, nb)
    A = E.emu_mat_clone(ctx, S)
    E.emu_potrf_mp(ctx, A)
    B = torch.from_numpy(np.random.default_rng(n + r).standard_normal((r, n))).cuda().t()
    X, info = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
    X, B, C = X.cpu().numpy(), B.cpu().numpy(), O.cov_build(L, 4.0)
    back = np.linalg.norm(B - C @ X, axis=0) / (np.linalg.norm(C) * np.linalg.norm(X, axis=0) + np.linalg.norm(B, axis=0))
    assert info.status == E.EMU_OK and back.max() <= 1e-14 + 2 * n * 2.0**-53
