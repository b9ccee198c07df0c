"""Digit products of operands near the lower end of the FP64 range.  The transforms are linear, and a power of two scales
every exact step of theirs: scaled inputs give the scaled result but for values that become denormal on the way, which are
off by 2^-1074 each, below 2^-60 of the largest result at these scales."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    return E


@pytest.mark.parametrize("k", [-940, -970, -990, -1000])
def test_transforms_scale_with_their_input(E, k):
    import torch

    L, nt, nph, T = 48, 64, 100, 3
    g = torch.Generator("cuda").manual_seed(5)
    F = torch.randn(T, L * L, dtype=torch.float64, device="cuda", generator=g)
    with E.Context(0) as ctx:
        for call, X in ((lambda x: E.emu_isht(ctx, x, L, nt, nph), F),
                        (lambda x: E.emu_sht(ctx, x, L, nt, nph), E.emu_isht(ctx, F.t(), L, nt, nph).t().contiguous())):
            want = call(X.t())
            have = call((X * 2.0**k).t()) * 2.0**-k
            assert float((have - want).abs().max()) <= 2.0**-60 * float(want.abs().max())


def test_denormal_rows(E):
    """Rows of residuals whose every entry is denormal beside rows of size one: their products with those keep all bits
    that the result can hold (the diagonal perturbation is off)."""
    import torch

    n, m = 300, 128
    x = torch.randn(m, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    x[:, 40] *= 2.0**-1030
    x = x.contiguous()
    with E.Context(0) as ctx:
        A, _ = E.emu_cov_from_residuals(ctx, x.t(), 256, nugget_rel=0.0)
        U = E.emu_mat_export(ctx, A).cpu().numpy()
    X = x.cpu().numpy().astype(np.longdouble)
    want = (X[:, 41:].T @ X[:, 40]) / m
    # m roundings of FP64 (the scaling by 1 / m), and the denormal spacing of the result
    assert np.abs(U[41:, 40] - want).max() <= 4 * 2.0**-1074
