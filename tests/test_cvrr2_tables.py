"""The values of the planner's (a 0|C) tables (VRR1 items, harmonic weights,
accumulators, gather), evaluated on the host for one primitive triple, against
Eq. vrr1 taken one quantum at a time and the closed n-quantum form on a
Cartesian ket followed by the oracle's solid-harmonic transform.  The
geometry's numbers are drawn independently: the identity is algebraic.

Tolerance: both sides are sums of at most a few hundred terms in FP64, each
term a product of at most 2 (la + lb) + lc + 4 factors, so they agree to that
many roundings of the terms' magnitudes: 1e-13 of the sum with every term
taken positive."""
import ctypes
from functools import lru_cache
from math import comb, factorial

import numpy as np
import pytest

from oracle.solid import cart_list, solid_matrix
from paper_2210_03192_gb300 import _lib


def evaluate(la, lb, lc, geom, base):
    L = _lib.load()
    cap = sum((l + 1) * (l + 2) // 2 for l in range(la + lb + 1))
    out, rows, n = np.zeros((cap, 2 * lc + 1)), np.zeros((cap, 3), np.int32), ctypes.c_int32()
    g, b = np.ascontiguousarray(geom), np.ascontiguousarray(base)
    rc = L.lx3c_cvrr2_tables_eval(la, lb, lc, g.ctypes.data, b.ctypes.data, cap, out.ctypes.data, rows.ctypes.data,
                                  ctypes.addressof(n))
    assert rc == 0, L.lx3c_last_error()
    return [tuple(int(x) for x in r) for r in rows[:n.value]], out[:n.value]


def reference(lc, geom, base, a):
    """(a 0|C) and the same sum of magnitudes."""
    PA, f, rg, h, X, Y = geom[:3], geom[3:6], geom[6], geom[7], geom[8:11], geom[11]

    @lru_cache(None)
    def v(e, m):  # [e 0|0]^(lc+m), magnitude
        if sum(e) == 0:
            return base[m], abs(base[m])
        i = next(x for x in range(3) if e[x])
        lo = tuple(e[x] - (x == i) for x in range(3))
        (p, pm), (q, qm) = v(lo, m), v(lo, m + 1)
        s, t = PA[i] * p - f[i] * q, abs(PA[i]) * pm + abs(f[i]) * qm
        if lo[i]:
            lo2 = tuple(lo[x] - (x == i) for x in range(3))
            (p, pm), (q, qm) = v(lo2, m), v(lo2, m + 1)
            s, t = s + lo[i] * h * (p - rg * q), t + lo[i] * h * (pm + rg * qm)
        return s, t

    T = solid_matrix(lc)
    val, mag = np.zeros(len(T)), np.zeros(len(T))
    for ic, c in enumerate(cart_list(lc)):
        s = t = 0.0
        for u in np.ndindex(*(min(a[i], c[i]) + 1 for i in range(3))):
            k = Y ** sum(u)
            for i in range(3):
                k *= comb(a[i], u[i]) * comb(c[i], u[i]) * factorial(u[i]) * X[i] ** (c[i] - u[i])
            e, em = v(tuple(a[i] - u[i] for i in range(3)), 0)
            s, t = s + k * e, t + abs(k) * em
        val += T[:, ic] * s
        mag += np.abs(T[:, ic]) * t
    return val, mag


CLASSES = ([(la, lb, lc) for la in range(4) for lb in range(la + 1) for lc in range(7)] +
           [(4, 4, 6), (4, 2, 5), (2, 4, 6), (0, 3, 6), (5, 1, 4), (6, 0, 6), (6, 6, 6)])


@pytest.mark.parametrize("la,lb,lc", CLASSES)
def test_targets(la, lb, lc):
    rng = np.random.default_rng(100 * la + 10 * lb + lc)
    geom = rng.uniform(-1.3, 1.3, 12)
    geom[6:8] = rng.uniform(0.2, 0.9, 2)
    geom[11] = rng.uniform(0.1, 0.7)
    base = rng.uniform(0.1, 1.0, la + lb + 1)
    rows, out = evaluate(la, lb, lc, geom, base)
    assert len(set(rows)) == len(rows) and {sum(r) for r in rows} <= set(range(la, la + lb + 1))
    assert set(cart_list(la)) <= set(rows)
    for a, got in zip(rows, out):
        ref, mag = reference(lc, geom, base, a)
        assert np.all(np.abs(got - ref) <= 1e-13 * mag.max()), (a, np.abs(got - ref).max(), mag.max())


def test_bad_arguments():
    L = _lib.load()
    assert L.lx3c_cvrr2_tables_eval(7, 0, 0, None, None, 0, None, None, None) == -1
