"""Primitive pairs whose share of a block is below rounding are left out of
the class launches (csrc/primitives.h), and a shell pair whose Gaussian
products all underflow has zero blocks.  Checked where the rule can go wrong:
pairs with all, some and no primitive pairs left, one and many kets, the
tile kernel and the register-resident ones, B-oriented and split pairs, the
planned, host and allocation-free paths, into buffers that hold NaN."""
import numpy as np
import pytest

from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity import assert_parity  # noqa: E402
from test_zz_no_alloc import launch_noalloc  # noqa: E402


@pytest.fixture(scope="module")
def lx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as m
    return m


def mixed_problem(la, lb, lc, npair, naux, ka, kb, kc, seed):
    """A third of the pairs far apart with compact primitives only (products
    underflow to 0), a third with one diffuse primitive on each shell, a
    third as drawn."""
    p = W.class_problem(la, lb, lc, npair, naux, ka, kb, kc, box=12.0, exp_lo=0.05, exp_hi=1e4, seed=seed)
    rng = np.random.default_rng(seed + 1)
    for i, (a, b) in enumerate(p.pairs):
        if i % 3 == 2:
            continue
        for s in (a, b):
            e = p.orb.exps[p.orb.off[s]:p.orb.off[s] + p.orb.k[s]]
            e[:] = np.exp(rng.uniform(np.log(300.0), np.log(1e4), len(e)))
            if i % 3 == 1:
                e[0] = 0.08
        p.orb.xyz[b] = p.orb.xyz[a] + np.array([4.0, -3.0, 2.5])
    return p


@pytest.mark.parametrize("cls", [(0, 0, 3), (1, 0, 2), (0, 1, 2), (1, 0, 6), (2, 1, 1), (1, 3, 2), (3, 3, 0)])
@pytest.mark.parametrize("ka,kb,kc,naux", [(1, 1, 1, 1), (3, 2, 2, 37)])
def test_screened_primitives(lx, cls, ka, kb, kc, naux):
    p = mixed_problem(*cls, 9, naux, ka, kb, kc, seed=sum(cls) * 7 + ka)
    plan = lx.Eri3cPlan(p.orb, p.aux, p.pairs, p.auxs)
    out = torch.full(plan.shape, float("nan"), dtype=torch.float64, device="cuda")
    g = plan.execute(out).cpu().numpy()
    assert_parity(g, p)
    assert (g[0::3] == 0.0).all() and (np.abs(g[2::3]) > 0).any()
    h = lx.eri3c_host(p.orb, p.aux, p.pairs, p.auxs, out=np.full(plan.shape, np.nan))
    assert np.array_equal(h, g)
    n, keep = launch_noalloc(lx, p)
    torch.cuda.synchronize()
    assert_parity(n.cpu().numpy(), p)
