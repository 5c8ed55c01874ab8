"""The shipped tile hints: one line per class and contraction.  (A tile line
takes precedence over a CTAs-per-SM line, which would never act beside it.)"""
import paper_2210_03192_gb300 as lx


def test_one_line_per_class():
    seen = []
    with open(lx.HINTS_GB300) as f:
        for line in f:
            fields = line.split("#", 1)[0].split()
            if fields:
                seen.append(tuple(int(x) for x in fields[:6]))
    assert len(seen) == len(set(seen)), sorted(k for k in set(seen) if seen.count(k) > 1)
