"""Sizes at which what the plain FP64 factor and the sweeps keep in rotation comes round: more tile rows than the factor
keeps panels' digits for (three) and than its two sets of block solves, and more slabs than the sweeps have CTAs, so that
a CTA takes several slabs.  Bounds as in the tests of one or two tiles: 2 (n + 2) u sqrt(S_ii S_jj) of the factor, 4 n u of
the solves' normwise backward error."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
u = 2.0**-53


@pytest.fixture(scope="module")
def E():
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    return E


@pytest.mark.parametrize("L,nb", [(23, 128), (46, 128), (50, 256), (61, 512)])
def test_factor_of_many_tile_rows(E, L, nb):
    n = L * L
    with E.Context(0) as ctx:
        A = E.emu_cov_build(ctx, L, 4.0, nb)
        E.emu_potrf_mp(ctx, A)
        G = E.emu_mat_export(ctx, A).cpu().numpy()
        S = O.cov_build(L, 4.0)
        d = np.sqrt(np.diag(S))
        assert np.max(np.abs(G @ G.T - S) / np.outer(d, d)) <= 2 * (n + 2) * u
        # the same factor whatever the streams' timing
        for _ in range(3):
            B = E.emu_cov_build(ctx, L, 4.0, nb)
            E.emu_potrf_mp(ctx, B)
            assert (E.emu_mat_export(ctx, B).cpu().numpy() == G).all()


# 156 FP64 slabs on 152 CTAs at most, 308 FP32 ones on 304; one, several and two groups of right-hand sides
@pytest.mark.parametrize("L,nb,r,eps", [(99, 256, 1, 0.0), (99, 256, 18, 0.0), (140, 512, 3, 1e-8)])
def test_sweeps_of_more_slabs_than_ctas(E, L, nb, r, eps):
    import torch

    n = L * L
    B = torch.from_numpy(np.random.default_rng(r).standard_normal((r, n))).cuda().t()
    with E.Context(0) as ctx:
        S = E.emu_cov_build(ctx, L, 4.0, nb)
        norm = float(torch.linalg.norm(E.emu_mat_export(ctx, S))) * 2**0.5  # the lower triangle: at most that much
        A = E.emu_mat_clone(ctx, S)
        E.emu_potrf_mp(ctx, A, eps=eps)
        if eps == 0.0:
            X = E.emu_potrs(ctx, A, B)
            assert (E.emu_potrs(ctx, A, B) == X).all()
            bound = 4 * n * u
        else:
            X, info = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
            bound = 1e-14 + 4 * n * u
    X, B = X.cpu().numpy(), B.cpu().numpy()
    rows = np.unique(np.r_[0, 63, 64, n // 2, n - 65, n - 1, np.random.default_rng(n).integers(0, n, 40)])
    off = np.abs(O.cov_rows(L, 4.0, rows) @ X - B[rows])
    assert off.max() <= bound * (norm * np.linalg.norm(X, axis=0).max() + np.linalg.norm(B, axis=0).max())
