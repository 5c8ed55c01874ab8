"""No one-off measurement of bench.py replaces a key of its JSON line: the name
of the benchmark stays beside the fitting metric's figures."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_extras_leave_the_contract_keys_alone():
    sys.path.insert(0, ROOT)
    import bench

    class A:
        npair, naux, steps, warmup = 4096, 512, 1, 3
    res = dict(ms=1000.0, total_int=1e9, total_flops=1e12, table=[], clocks={}, launches=7, roofline={}, l3_frac={},
               e2e=dict(value=1.0))
    plain = bench.make_line(A, res, [(1, 1, 1, 1)], 1, None, {})
    fit = dict(naux_ao=27136, cholesky_ms=5660.0)
    line = bench.make_line(A, res, [(1, 1, 1, 1)], 1, None, dict(metric=fit, dfj=dict(fused_s=22.4), unit="x"))
    assert {k: line[k] for k in plain} == plain
    assert line["metric"] == "3c-ERI Gints/s FP64 per (La,Lb,Lc,K)"
    assert line["dfj"] == dict(fused_s=22.4) and fit in line.values()
