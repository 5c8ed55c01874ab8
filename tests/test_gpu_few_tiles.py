"""The tile shape of plans with fewer tiles a launch than two for each SM: wide
tiles keep the primitives that two CTAs per SM hold side by side, as a third
CTA would find no tile; larger plans keep the planner's default.  Values
against the oracle, per element."""
import pytest

from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity import assert_parity  # noqa: E402


@pytest.mark.parametrize("la,lb,lc,kc", [(1, 1, 1, 2), (1, 1, 2, 2), (1, 2, 0, 2), (2, 0, 2, 2)])
def test_few_and_many_tiles(la, lb, lc, kc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as lx
    seen = {}
    for npair in (60, 2400):
        p = W.class_problem(la, lb, lc, npair, 60, 3, 2, kc, box=3.0, exp_lo=0.2, exp_hi=5.0, seed=31)
        plan = lx.Eri3cPlan(p.orb, p.aux, p.pairs, p.auxs, False)
        for s in plan.shapes:
            if s["nsub"]:
                tiles = s["nsub"] * -(-60 // s["T"])
                seen.setdefault(npair, set()).add((s["T"], s["G"], tiles <= 304))
        if npair == 60:
            assert_parity(plan.execute().cpu().numpy(), p, bra_pure=False)
    few, many = ({(t, g) for t, g, f in seen[n] if f == (n == 60)} for n in (60, 2400))
    assert {t for t, _ in few} == {64} == {t for t, _ in many}
    assert min(g for _, g in few) > min(g for _, g in many)
