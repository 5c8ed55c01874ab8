"""cholesky_solve with many right-hand sides (V^-1 itself, or L^-1 (P|ab)):
values at widths on both sides of a block's eight columns, and 256 columns in
well under the time of 32 solves of eight."""
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


def factored(lx, n, seed):
    rng = np.random.default_rng(seed)
    M = rng.standard_normal((n, n))
    A = M @ M.T / n + np.eye(n)
    At = torch.tensor(A, device="cuda")
    lx.cholesky(At)
    return A, At


@pytest.mark.parametrize("n,nrhs", [(64, 8), (65, 9), (200, 64), (130, 255), (129, 256), (33, 257), (300, 300)])
def test_many_right_hand_sides(lx, n, nrhs):
    A, At = factored(lx, n, 7 * n + nrhs)
    B = np.random.default_rng(n).standard_normal((n, nrhs))
    X = lx.cholesky_solve(At, torch.tensor(B, device="cuda")).cpu().numpy()
    Xr = np.linalg.solve(A, B)
    assert np.abs(X - Xr).max() <= 20 * np.linalg.cond(A) * 2.2e-16 * np.abs(Xr).max()


def test_columns_side_by_side(lx):
    """One block's columns are independent: 256 of them fill the chip where
    eight use one block, so they take less than half of 32 times as long."""
    _, At = factored(lx, 1024, 3)

    def ms(nrhs):
        B = torch.randn(1024, nrhs, dtype=torch.float64, device="cuda")
        best = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            lx.cholesky_solve(At, B)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    assert ms(256) < 16 * ms(8)
