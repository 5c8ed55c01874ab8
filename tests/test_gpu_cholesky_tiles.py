"""Cholesky and solve at the edges of the 32-wide panels and 64-row solve
blocks, and on both sides of the line between 64 x 64 and 32 x 32 update tiles
(about 1,570 rows left); right-hand sides beyond one per warp.  Tolerances as
in test_gpu_metric.py: 1e-13 of the factor's largest element, and 20 kappa eps
for the solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as m
    return m


def spd(n, seed):
    rng = np.random.default_rng(seed)
    M = rng.standard_normal((n, n))
    return M @ M.T / n + np.eye(n)


@pytest.mark.parametrize("n,nrhs", [(2, 1), (31, 2), (32, 1), (33, 9), (127, 17), (1567, 1), (1633, 3)])
def test_factor_and_solve(lx, n, nrhs):
    A = spd(n, 3 * n)
    lda = n + 3  # rows padded: the factor keeps to its n columns
    buf = torch.full((n, lda), 7.0, dtype=torch.float64, device="cuda")
    buf[:, :n] = torch.tensor(A, device="cuda")
    view = buf[:, :n]
    _, info = lx.cholesky(view)
    assert info == 0 and bool((buf[:, n:] == 7.0).all())
    L = view.cpu().numpy()
    Lr = np.linalg.cholesky(A)
    assert np.abs(np.tril(L) - Lr).max() <= 1e-13 * np.abs(Lr).max()
    iu = np.triu_indices(n, 1)
    assert np.array_equal(L[iu], A[iu])
    B = np.random.default_rng(n).standard_normal((n, nrhs))
    X = lx.cholesky_solve(view, torch.tensor(B, device="cuda")).cpu().numpy()
    Xr = np.linalg.solve(A, B)
    assert np.abs(X - Xr).max() <= 20 * np.linalg.cond(A) * 2.2e-16 * np.abs(Xr).max()


def test_small_and_large_diagonals(lx):
    """Pivots outside the range of the reciprocal root's single-precision seed."""
    for scale in (1e-80, 1e-40, 1e40, 1e80):
        A = spd(70, 5) * scale
        At = torch.tensor(A, device="cuda")
        _, info = lx.cholesky(At)
        Lr = np.linalg.cholesky(A)
        assert info == 0 and np.abs(np.tril(At.cpu().numpy()) - Lr).max() <= 1e-13 * np.abs(Lr).max()
