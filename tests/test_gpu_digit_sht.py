"""Spherical-harmonic transforms as digit products: bandlimits, ring counts, longitudes and step counts at the edges of
their blocks of 32 orders, 64 columns and 128 rows, against the oracle (1e-12 of the largest value, the direct sums'
tolerance), and operands with an infinity or a NaN against the direct sums."""
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


def _col(x):
    import torch

    return torch.from_numpy(np.asfortranarray(x)).cuda().t().contiguous().t()


# L below, at and above multiples of 32 and 64; fewer rings than degrees; one and several row blocks of steps
@pytest.mark.parametrize("L,nt,nph,T", [(40, 41, 79, 1), (63, 33, 40, 2), (64, 65, 20, 3), (65, 30, 33, 2),
                                        (40, 12, 9, 65), (41, 7, 70, 129)])
def test_transforms_match_the_oracle(E, ctx, L, nt, nph, T):
    rng = np.random.default_rng(L + T)
    F = rng.standard_normal((L * L, T))
    Z = E.emu_isht(ctx, _col(F), L, nt, nph).cpu().numpy()
    want = O.isht(F, L, nt, nph)
    assert np.abs(Z - want).max() <= 1e-12 * np.abs(want).max()
    G = rng.standard_normal((nt * nph, T))
    F2 = E.emu_sht(ctx, _col(G), L, nt, nph).cpu().numpy()
    want = O.sht(G, L, nt, nph)
    assert np.abs(F2 - want).max() <= 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_operands_as_the_direct_sums(E, ctx, bad):
    """One column alone is small enough for the direct sums; among others it runs as digit products."""
    L, nt, nph, T = 24, 36, 60, 150
    rng = np.random.default_rng(3)
    F = rng.standard_normal((L * L, T))
    F[200, 7] = bad
    many = E.emu_isht(ctx, _col(F), L, nt, nph).cpu().numpy()
    one = E.emu_isht(ctx, _col(F[:, 7:8]), L, nt, nph).cpu().numpy()
    np.testing.assert_array_equal(many[:, 7:8], one)
    assert np.isfinite(np.delete(many, 7, 1)).all()
    G = rng.standard_normal((nt * nph, T))
    G[300, 9] = bad
    many = E.emu_sht(ctx, _col(G), L, nt, nph).cpu().numpy()
    one = E.emu_sht(ctx, _col(G[:, 9:10]), L, nt, nph).cpu().numpy()
    np.testing.assert_array_equal(many[:, 9:10], one)
    assert np.isfinite(np.delete(many, 9, 1)).all()
