"""Plain FP64 factor and draws as digit products on the tensor cores, at the edges of their tiles and blocks.

The factor's error against S is bounded entry by entry by (n + 2) u sqrt(S_ii S_jj) (the bound of a Cholesky factor
formed in FP64 arithmetic; the check's own product adds as much again), the draws' by (n + 2) u (|L| |Z|)."""
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


@pytest.fixture(scope="module")
def ctx(E):
    c = E.Context(0)
    yield c
    c.close()


def _factor_error(G, S):
    d = np.sqrt(np.diag(S))
    return np.max(np.abs(G @ G.T - S) / np.outer(d, d))


# one tile, two tiles, ragged last tiles of a few rows, several panels, 128 .. 1024 wide tiles
@pytest.mark.parametrize("L,nb", [(11, 128), (12, 128), (17, 128), (16, 256), (23, 256), (25, 384), (33, 512), (33, 1024)])
def test_fp64_factor_and_draws(E, ctx, L, nb):
    n = L * L
    A = E.emu_cov_build(ctx, L, 4.0, nb)
    S = O.cov_build(L, 4.0)
    E.emu_potrf_mp(ctx, A)
    G = E.emu_mat_export(ctx, A).cpu().numpy()
    assert np.all(np.triu(G, 1) == 0.0)
    assert _factor_error(G, S) <= 2 * (n + 2) * u
    for s in (1, 63, 65):
        Y, Z = E.emu_sample(ctx, A, s, seed=4, return_z=True)
        Y, Z = Y.cpu().numpy(), Z.cpu().numpy()
        assert np.all(np.abs(Y - G @ Z) <= 2 * (n + 2) * u * (np.abs(G) @ np.abs(Z)))


@pytest.mark.parametrize("nb", [128, 256])
def test_fp64_factor_of_a_badly_scaled_matrix(E, ctx, nb):
    """Rows and columns scaled by powers of two over 2^-300 .. 2^300: the factor's error scales with them."""
    import torch

    L = 21
    n = L * L
    rng = np.random.default_rng(5)
    d = 2.0 ** rng.integers(-300, 301, n)
    S = O.cov_build(L, 4.0) * d[:, None] * d[None, :]
    A = E.emu_mat_import(ctx, torch.from_numpy(S).cuda(), nb)
    E.emu_potrf_mp(ctx, A)
    G = E.emu_mat_export(ctx, A).cpu().numpy()
    assert _factor_error(G / d[:, None], O.cov_build(L, 4.0)) <= 2 * (n + 2) * u


@pytest.mark.parametrize("nb,eps", [(128, 0.0), (256, 0.0), (256, 1e-8)])
@pytest.mark.parametrize("row,col,bad,pivot", [(300, 40, np.nan, 301), (400, 400, np.nan, 401), (290, 289, np.nan, 291),
                                               (300, 40, np.inf, 301), (40, 40, np.inf, 0)])
def test_fp64_class_factor_with_an_infinity_or_a_nan_is_refused(E, ctx, nb, eps, row, col, bad, pivot):
    """It reaches the diagonal of its row through the digit products and is reported there, as FP64 arithmetic reports
    it (an infinite variance: at the first row of the next tile)."""
    import torch

    S = O.cov_build(21, 4.0)
    S[row, col] = S[col, row] = bad
    A = E.emu_mat_import(ctx, torch.from_numpy(S).cuda(), nb)
    info = E.emu_potrf_mp(ctx, A, eps=eps, prec_mask=1, raise_on_error=False)
    assert info.status == E.EMU_ENOTPD and info.pivot == (pivot or nb + 1)
