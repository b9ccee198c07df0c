"""Inverse transforms of more rings, or longitudes, than the digit form's grids take: the direct sums take them, as they do
smaller ones, against the closed forms of degree 1."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nt,nph", [(2, 32 * 65535 + 1, 1), (2, 2200001, 2), (2, 40, 65536)])
def test_isht_of_a_long_grid(L, nt, nph):
    import torch

    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    F = torch.tensor([[0.5, -0.25, 1.5, 0.75]], dtype=torch.float64, device="cuda").t()
    T = 8 if nt * nph < 4000000 else 1
    with E.Context(0) as ctx:
        Z = E.emu_isht(ctx, F.repeat(1, T), L, nt, nph)[:, T - 1].reshape(nph, nt)
    t = math.pi * torch.arange(nt, dtype=torch.float64, device="cuda") / (nt - 1)
    p = 2 * math.pi * torch.arange(nph, dtype=torch.float64, device="cuda") / nph
    c0, c1 = math.sqrt(1 / (4 * math.pi)), math.sqrt(3 / (4 * math.pi))
    # real basis of degree 1: -sqrt(3 / 4 pi) sin t {sin p, cos p} (Condon-Shortley phase), sqrt(3 / 4 pi) cos t
    want = 0.5 * c0 + c1 * (1.5 * torch.cos(t)[None] - torch.sin(t)[None] * (-0.25 * torch.sin(p) + 0.75 * torch.cos(p))[:, None])
    # the arguments of sine and cosine carry a rounding of pi i / (nt - 1): a few units
    assert float((Z - want).abs().max()) <= 1e-14
