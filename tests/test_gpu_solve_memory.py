"""Device memory of solves with many right-hand sides: beside the blocks of X's size that they keep, a bounded workspace
whatever their number.  The high-water mark is the device's memory pool's, from which the library allocates.  The columns
that end up in different launches are those of solves of their own, bit for bit."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L, NB, R = 32, 256, 200000
BLOCK = 8 * L * L * R  # bytes of X
USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


class _Pool:
    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.pool = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def peak(self, call):
        v = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0  # to what is in use
        assert self.cu.cuMemPoolGetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        before = v.value
        out = call()
        assert self.cu.cuMemPoolGetAttribute(self.pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
        return v.value - before, out


@pytest.mark.parametrize("eps", [0.0, 1e-8])
def test_many_right_hand_sides(eps):
    import torch

    import paper_2408_04440_gb300 as E
    from paper_2408_04440_gb300 import build

    build.build()
    with E.Context(0) as ctx:
        S = E.emu_cov_build(ctx, L, 4.0, NB)
        A = E.emu_mat_clone(ctx, S)
        E.emu_potrf_mp(ctx, A, eps=eps)
        B = torch.randn(R, L * L, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).t()
        torch.cuda.synchronize()
        pool = _Pool()
        # a padded copy of B, and the sweeps' workspace of 2 GB (allocations are rounded up)
        used, X = pool.peak(lambda: E.emu_potrs(ctx, A, B))
        assert used <= BLOCK + (2048 + 16 << 20)
        for c in (0, 130000, R - 33):
            assert (X[:, c:c + 33] == E.emu_potrs(ctx, A, B[:, c:c + 33])).all()
        # right-hand side, X, residual and correction; that workspace; the partial sums of few slabs
        used, (X, info) = pool.peak(lambda: E.emu_solve_refine(ctx, A, S, B, tol=1e-14))
        assert used <= 4 * BLOCK + (2048 + 64 << 20)
        assert info.status == E.EMU_OK
        Bn, Xn = B[:, -50:].cpu().numpy(), X[:, -50:].cpu().numpy()
        import oracle as O

        C = O.cov_build(L, 4.0)
        back = np.linalg.norm(Bn - C @ Xn, axis=0) / (np.linalg.norm(C) * np.linalg.norm(Xn, axis=0))
        assert back.max() <= 1e-14 + 2 * L * L * 2.0**-53
