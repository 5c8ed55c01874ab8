"""DF-J with orbital l = 5 and 6 over ket lists of one and two shells of their
own (l, K): a tile of one or two kets would hold the densities of 32 or 16
primitive pairs side by side, more than shared memory takes at Hermite degrees
11 and 12.  Tolerances as in test_gpu_hermite.py (1e-12 of the largest
element, binary128 oracle)."""
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


@pytest.mark.parametrize("lc", [0, 5, 6])
@pytest.mark.parametrize("la,lb,count", [(6, 6, 1), (6, 6, 2), (6, 5, 1), (6, 5, 2)])
def test_short_ket_lists(lx, la, lb, lc, count):
    rng = np.random.default_rng(100 * la + 10 * lc + count)
    at = np.array([[0.0, 0.0, 0.0], [1.2, 0.3, -0.5]])
    orb = W.make_basis([la, lb], [1, 1], at, rng.uniform(0.2, 1.5, 2), rng.uniform(0.1, 1.0, 2), [0, 1])
    aux = W.make_basis([lc] * count, [1] * count, at[:count], rng.uniform(0.3, 2.0, count), rng.uniform(0.1, 1.0, count),
                       list(range(count)))
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    D, c = W.density(rng, n), rng.standard_normal(na)
    plan = lx.DFJPlan(orb, aux, 0.0)
    g, J = (x.cpu().numpy() for x in plan.execute(torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")))
    go, Jo = oracle.dfj(orb, aux, D, c, tasks=plan.tasks(), mode="quad")
    assert np.abs(g - go).max() <= 1e-12 * np.abs(go).max()
    assert np.abs(J - Jo).max() <= 1e-12 * np.abs(Jo).max()
