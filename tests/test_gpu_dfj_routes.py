"""Strongly contracted classes of low angular momentum: their DF-J build forms
and digests integrals, in about the time the several-density build (which always
does) takes for one density; gamma and J agree with it to rounding."""
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


def best_ms(f):
    f()
    best = 1e30
    for _ in range(6):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        f()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("recipe,lc", [([(1, 60, 6)], 0), ([(1, 40, 4)], 0), ([(0, 60, 6), (2, 20, 6)], 0),
                                       ([(0, 60, 6), (3, 20, 6)], 2), ([(2, 40, 1)], 3), ([(1, 60, 2)], 2)])
def test_route(lx, recipe, lc):
    rng = np.random.default_rng(5)
    orb = W.concat(*[W.random_shells(rng, n, l, K, 6.0, 0.1, 30.0) for l, n, K in recipe])
    aux = W.random_shells(rng, 256, lc, 1, 6.0, 0.1, 30.0)
    plan = lx.DFJPlan(orb, aux, 1e-12)
    D = torch.tensor(W.density(rng, plan.nao), device="cuda")
    c = torch.tensor(rng.standard_normal(plan.naux_ao), device="cuda")
    D1, c1 = D[None].contiguous(), c[None].contiguous()
    g, J = plan.execute(D, c)
    g1, J1 = plan.execute_multi(D1, c1)
    assert (g - g1[0]).abs().max() <= 1e-13 * g.abs().max()
    assert (J - J1[0]).abs().max() <= 1e-13 * J.abs().max()
    assert torch.equal(plan.execute(D, c, outputs="gamma")[0], g)
    assert torch.equal(plan.execute(D, c, outputs="J")[1], J)
    single, several = best_ms(lambda: plan.execute(D, c)), best_ms(lambda: plan.execute_multi(D1, c1))
    assert single < 1.2 * several, (single, several)
