"""Top eigenpairs of matrices whose tridiagonal form decouples (diagonal, and
diagonal in blocks of two), with repeated and dyadic entries, and with one
entry on a point of the first bisection grid followed by entries just below
it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _grid_point(t):
    """Point t of the 512 between -2^-21 and 1 + 2^-21 (diagonal entries
    between 0 and 1), in FP32 as the kernel forms it, and the spacing."""
    f = np.float32
    lo, hi = f(0) - f(2.0 ** -21), f(1) + f(2.0 ** -21)
    step = f(hi - lo) * (f(1) / f(513))
    return f(np.float64(t) * np.float64(step) + np.float64(lo)), step


def _matrix(kind, k):
    rng = np.random.default_rng(k)
    if kind == "dyadic":
        return np.diag(rng.integers(-8, 9, k) / 8.0)
    if kind == "blocks":
        H = np.diag(rng.integers(-4, 5, k) / 4.0)
        for i in range(0, k - 1, 2):
            H[i, i + 1] = H[i + 1, i] = rng.integers(0, 3) / 4.0
        return H
    if kind == "identity":
        return np.eye(k)
    x, step = _grid_point(int(kind))
    d = np.zeros(k)
    d[:5] = [1.0, x, x - 0.4 * step, x - 0.5 * step, x - 0.6 * step]
    return np.diag(d)


@pytest.mark.parametrize("kind", ["dyadic", "blocks", "identity", "100", "256", "300", "411"])
@pytest.mark.parametrize("k,r", [(8, 5), (33, 5), (64, 16), (150, 20)])
def test_decoupled_matrices(kind, k, r):
    import paper_2308_01480_gb300 as tt
    H = torch.from_numpy(_matrix(kind, k).astype(np.float32)).cuda()
    V, lam = (t.cpu().double().numpy() for t in tt.sym_eig_top(H, r))
    Hd = H.cpu().double().numpy()
    # the bisection stops at 5e-8 of the span, FP32 vectors at 1e-6 of the norm
    assert np.abs(lam - np.linalg.eigvalsh(Hd)[::-1][:r]).max() <= 1e-6
    assert np.abs(V.T @ V - np.eye(r)).max() <= 1e-5
    assert np.abs(Hd @ V - V * lam).max() <= 1e-5
