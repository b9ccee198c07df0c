"""The plain FP64 factor, its draws and the transforms in FP64 arithmetic by choice (emu_fp64_arithmetic), which is also
where they go when their digits do not fit the device: entry by entry within the bounds of FP64 sums, 2 (n + 2) u
(|L| |L|^T) with the check's own product, and switched off the digit form's bits again."""
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


def _dev(x):
    import torch

    return torch.from_numpy(np.ascontiguousarray(x.T)).cuda().t()


def _uneven(n, nb):
    """Unit matrix plus tiles whose entries span 1e-14 .. 1e-1."""
    rng = np.random.default_rng(n)
    C = np.eye(n)
    E = np.tril(rng.choice((-1.0, 1.0), (n, n)) * 10.0 ** rng.uniform(-14, -1, (n, n)), -1) / n**0.5
    E *= rng.random((n, n)) < 0.1
    return C + E + E.T


@pytest.mark.parametrize("n,nb", [(512, 128), (700, 256), (1025, 512)])
@pytest.mark.parametrize("kind", ["uneven", "covariance"])
def test_factor_and_draws_entry_by_entry(E, kind, n, nb):
    if kind == "covariance":
        L = int(n**0.5)
        S = O.cov_build(L, 3.0)
    else:
        S = _uneven(n, nb)
    n = S.shape[0]
    with E.Context(0) as ctx:
        ctx.fp64_arithmetic()
        A = E.emu_mat_import(ctx, _dev(S), nb)
        E.emu_potrf_mp(ctx, A)
        G = E.emu_mat_export(ctx, A).cpu().numpy()
        assert np.all(np.abs(G @ G.T - S) <= 2 * (n + 2) * u * (np.abs(G) @ np.abs(G).T))
        Y, Z = E.emu_sample(ctx, A, 65, seed=4, return_z=True)
        Y, Z = Y.cpu().numpy(), Z.cpu().numpy()
        assert np.all(np.abs(Y - G @ Z) <= 2 * (n + 2) * u * (np.abs(G) @ np.abs(Z)))


def test_transforms_are_the_direct_sums(E):
    """A column of a transform of many is the one that a transform small enough for the direct sums gives alone."""
    rng = np.random.default_rng(3)
    L, nt, nph, T = 24, 36, 60, 150
    F, G = rng.standard_normal((L * L, T)), rng.standard_normal((nt * nph, T))
    with E.Context(0) as ctx:
        digits = E.emu_isht(ctx, _dev(F), L, nt, nph), E.emu_sht(ctx, _dev(G), L, nt, nph)
        one = E.emu_isht(ctx, _dev(F[:, 7:8]), L, nt, nph), E.emu_sht(ctx, _dev(G[:, 7:8]), L, nt, nph)
        ctx.fp64_arithmetic()
        many = E.emu_isht(ctx, _dev(F), L, nt, nph), E.emu_sht(ctx, _dev(G), L, nt, nph)
        for d, m, o in zip(digits, many, one):
            assert (m[:, 7:8] == o).all()
            assert float((m - d).abs().max()) <= 1e-12 * float(d.abs().max())
        L, nt, nph = 48, 50, 97
        F, G = rng.standard_normal((L * L, 2)), rng.standard_normal((nt * nph, 2))
        for have, want in ((E.emu_isht(ctx, _dev(F), L, nt, nph), O.isht(F, L, nt, nph)),
                           (E.emu_sht(ctx, _dev(G), L, nt, nph), O.sht(G, L, nt, nph))):
            assert np.abs(have.cpu().numpy() - want).max() <= 1e-12 * np.abs(want).max()


def test_off_again(E):
    L, nb = 24, 128

    def run(ctx):
        A = E.emu_cov_build(ctx, L, 4.0, nb)
        E.emu_potrf_mp(ctx, A)
        return E.emu_mat_export(ctx, A).cpu(), E.emu_sample(ctx, A, 9, 2).cpu()

    with E.Context(0) as ctx:
        first = run(ctx)
        ctx.fp64_arithmetic()
        fp64 = run(ctx)
        ctx.fp64_arithmetic(False)
        again = run(ctx)
    for a, b, c in zip(first, again, fp64):
        assert (a == b).all() and not (a == c).all()
        assert float((a - c).norm()) <= 1e-13 * float(a.norm())
