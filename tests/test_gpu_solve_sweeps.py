"""Triangular sweeps and refined solves at the edges of their slabs (64 rows), right-hand-side groups (1, 4, 16, 32) and
tile sizes, against the oracle's factor: the plain FP64 factor to 1e-12 of its condition-free residual, the mixed factor as
a preconditioner (refinement converges), and repeated solves give the same bits."""
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


def _rhs(n, r):
    import torch

    return torch.from_numpy(np.random.default_rng(n + r).standard_normal((r, n))).cuda().t()


def _backward(S, X, B):
    return np.max(np.linalg.norm(B - S @ X, axis=0) / (np.linalg.norm(S) * np.linalg.norm(X, axis=0)))


# a slab alone, two slabs, ragged tiles, tile sizes from 64 to 2048
@pytest.mark.parametrize("L,nb,r", [(8, 64, 1), (9, 64, 4), (11, 192, 5), (20, 256, 16), (23, 128, 17), (33, 1024, 3)])
def test_fp64_sweeps(E, ctx, L, nb, r):
    A = E.emu_cov_build(ctx, L, 4.0, nb)
    E.emu_potrf_mp(ctx, A)
    B = _rhs(L * L, r)
    X = E.emu_potrs(ctx, A, B)
    # backward stable: n u, with a factor 4 for the two sweeps and the check's own product
    assert _backward(O.cov_build(L, 4.0), X.cpu().numpy(), B.cpu().numpy()) <= 4 * L * L * 2.0**-53
    assert (E.emu_potrs(ctx, A, B) == X).all()


@pytest.mark.parametrize("L,nb,r,eps", [(16, 256, 1, 1e-8), (23, 256, 4, 1e-6), (23, 256, 16, 1e-8), (30, 256, 33, 1e-6),
                                        (33, 1024, 2, 1e-8), (46, 2048, 5, 1e-8)])
def test_refined_solves(E, ctx, L, nb, r, eps):
    S = E.emu_cov_build(ctx, L, 4.0, nb)
    A = E.emu_mat_clone(ctx, S)
    E.emu_potrf_mp(ctx, A, eps=eps, prec_mask=0b11011)
    B = _rhs(L * L, r)
    X, info = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
    assert info.status == E.EMU_OK
    assert _backward(O.cov_build(L, 4.0), X.cpu().numpy(), B.cpu().numpy()) <= 1e-14 + 2 * L * L * 2.0**-53
    again, _ = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
    assert (again == X).all()


@pytest.mark.parametrize("L,nb,r", [(46, 128, 2), (46, 256, 16), (46, 512, 17), (47, 384, 33)])
def test_residuals_as_digit_products(E, ctx, L, nb, r):
    """From 2048 rows on: chunks of 128 and 256, ragged tiles, groups of 16; a matrix whose rows are scaled by powers of
    two over 2^-40 .. 2^40 converges as it does unscaled, and one that is not positive semidefinite is solved too."""
    import torch

    n = L * L
    S0 = O.cov_build(L, 4.0)
    d = 2.0 ** np.random.default_rng(L).integers(-20, 21, n)
    for kind in ("plain", "scaled", "indefinite"):
        M = S0 * d[:, None] * d[None, :] if kind == "scaled" else S0.copy()
        A = E.emu_mat_import(ctx, torch.from_numpy(M).cuda(), nb)
        E.emu_potrf_mp(ctx, A)
        if kind == "indefinite":  # refine against another matrix: one entry above its rows' diagonals
            M[1500, 1400] = M[1400, 1500] = 1e-5
        S = E.emu_mat_import(ctx, torch.from_numpy(M).cuda(), nb)
        B = _rhs(n, r)
        X, info = E.emu_solve_refine(ctx, A, S, B, tol=1e-14, raise_on_error=False)
        X, Bn = X.cpu().numpy(), B.cpu().numpy()
        if kind != "indefinite":
            assert info.status == E.EMU_OK
        # the residual the call reports is the one its iterate has
        have = np.max(np.linalg.norm(Bn - M @ X, axis=0)
                      / (np.linalg.norm(M) * np.linalg.norm(X, axis=0) + np.linalg.norm(Bn, axis=0)))
        assert abs(have - info.rel_resid) <= 1e-6 * have + 2 * n * 2.0**-53
