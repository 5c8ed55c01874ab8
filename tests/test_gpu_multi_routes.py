"""Several densities on (s s|C) and (p s|C) launches: the register-resident
kernels from two warps per SM on, at every width of a tile (each density as by
itself, 1e-13: only the order of sums differs), and small launches in less time
than a warp takes to run its tiles one after another."""
import numpy as np
import pytest

from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as m
    return m


def basis(rng, recipe, box, lo, hi):
    return W.concat(*[W.random_shells(rng, n, l, K, box, lo, hi) for l, n, K in recipe])


@pytest.mark.parametrize("count,nd", [(1, 8), (2, 3), (3, 5), (7, 2), (16, 1), (33, 8)])
def test_register_kernels_with_full_launches(lx, count, nd):
    """9,870 (s s| and 9,800 (p s| pairs: 304 warps and more even with one ket
    shell of a kind (32 pairs a warp)."""
    rng = np.random.default_rng(700 + count)
    orb = basis(rng, [(0, 140, 1), (1, 70, 1)], 3.0, 0.1, 3.0)
    aux = basis(rng, [(0, count, 2), (2, count, 1), (4, 1, 1), (6, 1, 1)], 3.0, 0.2, 3.0)
    plan = lx.DFJPlan(orb, aux, 0.0)
    D = torch.tensor(np.stack([W.density(rng, plan.nao) for _ in range(nd)]), device="cuda")
    c = torch.tensor(rng.standard_normal((nd, plan.naux_ao)), device="cuda")
    g, J = plan.execute_multi(D, c)
    for k in range(nd):
        g1, J1 = plan.execute(D[k].contiguous(), c[k].contiguous())
        assert (g[k] - g1).abs().max() <= 1e-13 * g1.abs().max()
        assert (J[k] - J1).abs().max() <= 1e-13 * J1.abs().max()


def test_small_launches_are_not_one_warp_long(lx):
    """One (s s| pair of 100 primitives over 32 d kets: 218 us a build when one
    warp runs them and eight densities one after another, 140 when the tile
    kernel shares them among its threads."""
    rng = np.random.default_rng(3)
    orb = basis(rng, [(0, 1, 10)], 1.0, 0.1, 3.0)
    aux = basis(rng, [(2, 32, 1)], 1.0, 0.2, 3.0)
    plan = lx.DFJPlan(orb, aux, 0.0)
    D = torch.tensor(np.stack([W.density(rng, plan.nao) for _ in range(8)]), device="cuda")
    c = torch.tensor(rng.standard_normal((8, plan.naux_ao)), device="cuda")
    best = 1e30
    for _ in range(10):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(10):
            plan.execute_multi(D, c)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) / 10)
    assert best < 0.18, best
