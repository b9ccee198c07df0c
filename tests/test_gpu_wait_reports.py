"""Waits of the triangular sweeps that run out are reported (failure detection without a GPU fault): the test hook keeps
one solved slab unpublished and bounds the wait at 2e5 cycles, so the sweep that needs it gives up and returns.  A refined
solve reports it itself; emu_potrs returns before its device work ends, and the context's next call that reads the device
status reports it, once.  The context then works as before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L, NB = 32, 256


@pytest.fixture(scope="module")
def E():
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    return E


@pytest.fixture()
def ctx(E):
    c = E.Context(0)
    yield c
    c.close()


def _factor(E, ctx, eps):
    S = E.emu_cov_build(ctx, L, 4.0, NB)
    A = E.emu_mat_clone(ctx, S)
    E.emu_potrf_mp(ctx, A, eps=eps)
    return S, A


def _rhs(r):
    import torch

    return torch.from_numpy(np.random.default_rng(r).standard_normal((r, L * L))).cuda().t()


def _times_out(E, call):
    with pytest.raises(E.EmuError) as err:
        call()
    assert err.value.status == E.EMU_ETIMEOUT


@pytest.mark.parametrize("slab", [0, 5, 15])
@pytest.mark.parametrize("eps,r", [(0.0, 1), (0.0, 17), (1e-8, 1), (1e-8, 33)])
def test_refined_solve_reports_it(E, ctx, eps, r, slab):
    S, A = _factor(E, ctx, eps)
    B = _rhs(r)
    want, _ = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
    ctx.test_sweep_hook(200000, slab)
    _times_out(E, lambda: E.emu_solve_refine(ctx, A, S, B, tol=1e-14))
    ctx.test_sweep_hook()
    have, _ = E.emu_solve_refine(ctx, A, S, B, tol=1e-14)
    assert (have == want).all()


@pytest.mark.parametrize("eps", [0.0, 1e-8])
@pytest.mark.parametrize("reader", ["factor", "residuals", "refine", "sample_host", "isht", "batch"])
def test_the_next_reader_reports_what_a_solve_left(E, ctx, eps, reader):
    import torch

    S, A = _factor(E, ctx, eps)
    B = _rhs(2)
    want = E.emu_potrs(ctx, A, B)
    ctx.test_sweep_hook(200000, 3)
    E.emu_potrs(ctx, A, B)
    ctx.test_sweep_hook()
    # another solve clears the status words of its own, and not what the first one left
    assert (E.emu_potrs(ctx, A, B) == want).all()
    xi = torch.randn(3000, L * L, dtype=torch.float64, device="cuda").t()
    F = torch.randn(2, 48 * 48, dtype=torch.float64, device="cuda").t()
    call = {"factor": lambda: E.emu_potrf_mp(ctx, E.emu_mat_clone(ctx, S), eps=eps),
            "residuals": lambda: E.emu_cov_from_residuals(ctx, xi, NB),
            "refine": lambda: E.emu_solve_refine(ctx, A, S, B, tol=1e-14),
            "sample_host": lambda: E.emu_sample_host(ctx, A, 4, 1),
            "isht": lambda: E.emu_isht(ctx, F, 48, 60, 100),
            "batch": lambda: E.emu_batch_potrf_sample(ctx, [(8, 3.0), (12, 3.0)], nb=NB, eps=1e-8, nsamples=4, seed=1),
            }[reader]
    _times_out(E, call)
    call()
    assert (E.emu_potrs(ctx, A, B) == want).all()
