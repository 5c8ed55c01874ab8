"""The per-pair kernels of the Hermite-basis DF-J build (densities before, J
blocks and forces after) on strongly contracted pairs, whose primitives are cut
into ranges: values at ragged ranges (tolerances as in test_gpu_hermite.py),
and a single pair of 256 primitives in a fraction of the time that one warp
takes to run them one after another (3.2 ms a build, 5.3 a gradient)."""
import numpy as np
import pytest

import oracle
from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as m
    return m


def problem(seed, recipe, auxr):
    rng = np.random.default_rng(seed)
    make = lambda r: W.concat(*[W.random_shells(rng, n, l, K, 2.5, 0.2, 20.0) for l, n, K in r])  # noqa: E731
    orb, aux = make(recipe), make(auxr)
    for b in (orb, aux):
        b.atom[:] = np.arange(b.nshell) % 2
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    return orb, aux, W.density(rng, n), rng.standard_normal(na)


@pytest.mark.parametrize("recipe", [[(1, 1, 5), (2, 1, 1)], [(2, 1, 5), (1, 2, 3)], [(0, 1, 7), (3, 1, 3)]])
def test_ranges_of_primitives(lx, recipe):
    orb, aux, D, c = problem(11, recipe, [(0, 3, 1), (2, 2, 2), (5, 1, 1)])
    plan = lx.DFJPlan(orb, aux, 0.0, gradient=True)
    Dt, ct = torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")
    g, J = (x.cpu().numpy() for x in plan.execute(Dt, ct))
    go, Jo = oracle.dfj(orb, aux, D, c, tasks=plan.tasks(), mode="quad")
    assert np.abs(g - go).max() <= 1e-12 * np.abs(go).max()
    assert np.abs(J - Jo).max() <= 1e-12 * np.abs(Jo).max()
    G = plan.gradient(Dt, ct).cpu().numpy()
    Go = oracle.dfj_grad(orb, aux, D, c, plan.natom, tasks=plan.tasks(), mode="quad")
    assert np.abs(G - Go).max() <= 1e-11 * np.abs(Go).max()


def test_one_pair_of_many_primitives(lx):
    orb, aux, D, c = problem(5, [(1, 1, 16)], [(2, 32, 1)])
    plan = lx.DFJPlan(orb, aux, 0.0, gradient=True)
    Dt, ct = torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")

    def ms(f):
        best = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            f()
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best
    assert ms(lambda: plan.execute(Dt, ct)) < 0.6
    assert ms(lambda: plan.gradient(Dt, ct)) < 1.0
