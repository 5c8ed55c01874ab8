"""A second device in one process (skipped with one): plans made on it run the
same kernels to the same bits, tiles above the 48 KB that a kernel gets
unasked among them."""
import numpy as np
import pytest

from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_plans_on_two_devices():
    if not torch.cuda.is_available() or torch.cuda.device_count() < 2:
        pytest.skip("needs two CUDA devices")
    import paper_2210_03192_gb300 as lx
    problems = [W.class_problem(la, lb, lc, 4, 40, 2, 2, 1, box=6.0, exp_lo=0.1, exp_hi=50.0, seed=5)
                for la, lb, lc in ((1, 1, 2), (3, 3, 4), (4, 4, 6))]
    outs = []
    for dev in (0, 1):
        with torch.cuda.device(dev):
            outs.append([lx.eri3c(p.orb, p.aux, p.pairs, p.auxs).cpu().numpy() for p in problems])
    for a, b in zip(*outs):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
