"""The lagged recursion f_t = sum_p phi_p f_{t-p} + xi_t against NumPy: every
number of lags (the kernel is compiled per lag count up to four), sizes around
a warp and the sixteen steps read ahead, and values that are not finite."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _recursion(xi, phi):
    n, T = xi.shape
    c = np.zeros((n, 8))
    c[:, :phi.shape[1]] = phi
    f = np.zeros((n, T + 8))
    with np.errstate(all="ignore"):
        for t in range(T):
            v = np.zeros(n)
            for p in range(8):
                v = v + c[:, p] * f[:, t + 7 - p]
            f[:, t + 8] = v + xi[:, t]
    return f[:, 8:]


def _case(P, n, T, seed):
    rng = np.random.default_rng(seed)
    phi = rng.uniform(-1, 1, (n, P))
    phi *= 0.5 / np.maximum(np.abs(phi).sum(axis=1, keepdims=True), 1e-30)
    return rng.standard_normal((n, T)), phi


def _run(xi, phi):
    import paper_2408_04440_gb300 as E
    ctx = E.Context(0)
    X = torch.from_numpy(np.asfortranarray(xi)).cuda()
    Ph = torch.from_numpy(np.asfortranarray(phi)).cuda()
    return E.emu_var_recursion(ctx, X, Ph).cpu().numpy()


@pytest.mark.parametrize("P", range(1, 9))
@pytest.mark.parametrize("n,T", [(1, 1), (31, 7), (33, 8), (1000, 9), (64, 41), (65, 15), (5, 16), (32, 17), (3, 33)])
def test_matches_numpy(P, n, T):
    xi, phi = _case(P, n, T, 100 * P + T)
    ref = _recursion(xi, phi)
    # sum |phi| = 1/2: roundings of a step (at most 3 P + 2 of half a unit on both
    # sides together, each of a term below max |f|) at most double along the chain
    tol = 2 * (3 * P + 2) * 2.0 ** -52 * np.abs(ref).max()
    assert np.abs(_run(xi, phi) - ref).max() <= tol


@pytest.mark.parametrize("P", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_values_not_finite(P, bad):
    xi, phi = _case(P, 40, 30, P)
    phi[::3] = 0.0  # a zero factor times an infinity is NaN
    for k in range(40):
        xi[k, k % 30] = bad
    ref, got = _recursion(xi, phi), _run(xi, phi)
    assert np.array_equal(np.isnan(ref), np.isnan(got))
    assert np.array_equal(np.isinf(ref), np.isinf(got))
    assert np.array_equal(np.sign(ref[np.isinf(ref)]), np.sign(got[np.isinf(ref)]))
