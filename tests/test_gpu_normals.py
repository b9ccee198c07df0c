"""The normal generator's own logarithm, sine and square root (table and Taylor polynomial, table entries recomputed here
with 60 digits) and the draws built on it, against 64-bit references, at odd sizes."""
import os
import re
from decimal import Decimal, getcontext

import numpy as np
import pytest

import oracle as O

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_2408_04440_gb300", "csrc", "rng_tables.h")


def _table(name):
    src = open(HEADER).read()
    body = src[src.index("double " + name):]
    body = body[body.index("= {") + 3:body.index("};")]
    return [[float.fromhex(x) for x in re.findall(r"-?0x[0-9a-f.]+p[+-]?\d+", row)] for row in re.findall(r"\{([^{}]*)\}", body)]


def test_logarithm_tables():
    getcontext().prec = 60
    log = _table("kLogTab")
    assert len(log) == 257
    ln2 = Decimal(2).ln()
    for j, (inv, hi, lo) in enumerate(log):
        assert inv == 1.0 / (1.0 + j / 256.0)
        want = 2 * Decimal(inv).ln() + (2 * ln2 if j >= 128 else 0)
        assert (hi * 2.0**40).is_integer()
        assert abs(Decimal(hi) + Decimal(lo) - want) <= Decimal(2) ** -94
    for k, (hi, lo) in enumerate(_table("kLogExp")):
        assert (hi * 2.0**40).is_integer()
        assert abs(Decimal(hi) + Decimal(lo) - 2 * k * ln2) <= Decimal(2) ** -92
    # the ends meet 1 without cancellation
    assert log[0] == [1.0, 0.0, 0.0] and log[256] == [0.5, 0.0, 0.0]


def _cos_sin(x):
    """Taylor sums of cos x and sin x, |x| < 7, with the context's digits."""
    out = []
    for term, n in ((Decimal(1), 0), (x, 1)):
        total = Decimal(0)
        while abs(term) > Decimal(10) ** -50:
            total += term
            term *= -x * x / ((n + 1) * (n + 2))
            n += 2
        out.append(total)
    return out


def test_trigonometric_table():
    getcontext().prec = 60
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494")
    tab = _table("kTrigTab")
    assert len(tab) == 256
    for j, (c, s) in enumerate(tab):
        for got, want in zip((c, s), _cos_sin(2 * pi * j / 256)):
            assert abs(Decimal(got) - want) <= Decimal(2) ** -54
            assert got in (0.0, 1.0, -1.0) or j % 64
    assert [r[0] for r in tab[::64]] == [1, 0, -1, 0] and [r[1] for r in tab[::64]] == [0, 1, 0, -1]


@pytest.mark.gpu
@pytest.mark.parametrize("L,nb,s", [(7, 64, 1), (9, 128, 3), (33, 64, 65), (20, 256, 700)])
def test_normals_match_the_oracle(L, nb, s):
    """Every normal within 4 ulp of its pair's radius (at most 8.6) of the oracle's, which takes them from libm."""
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    with E.Context(0) as ctx:
        A = E.emu_cov_build(ctx, L, 4.0, nb)
        E.emu_potrf_mp(ctx, A)
        _, Z = E.emu_sample(ctx, A, s, seed=(5 << 40) + 11, stream_id=3, return_z=True)
        Z = Z.cpu().numpy()
    want = O.normal_matrix((5 << 40) + 11, 3, L * L, s)
    assert np.abs(Z - want).max() <= 8.6 * 4 * 2.0**-52
