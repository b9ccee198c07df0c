"""Draws from a good factor after another matrix of the same context was refused: the refusal's status word does not stop
them, for every storage of the factor, and what the sampler prepares on its first call is sound."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    return E


@pytest.mark.parametrize("kind", ["fp64", "mixed", "classfmt"])
def test_a_refused_matrix_does_not_stop_draws(E, kind):
    import torch

    L, nb, eps = 23, 256, 1e-8

    def factor(ctx):
        if kind == "classfmt":
            A = E.emu_cov_build_classfmt(ctx, L, 4.0, nb, eps=eps)
        else:
            A = E.emu_cov_build(ctx, L, 4.0, nb)
        E.emu_potrf_mp(ctx, A, eps=0.0 if kind == "fp64" else eps)
        return A

    with E.Context(0) as ctx:
        want = E.emu_sample(ctx, factor(ctx), 40, 3).cpu()
    with E.Context(0) as ctx:
        A = factor(ctx)
        bad = E.emu_mat_import(ctx, -torch.eye(300, dtype=torch.float64, device="cuda"), nb)
        assert E.emu_potrf_mp(ctx, bad, eps=eps, raise_on_error=False).status == E.EMU_ENOTPD
        for _ in range(2):
            assert (E.emu_sample(ctx, A, 40, 3).cpu() == want).all()
