"""lx3c_class_flops of the classes on the register-resident kernels, (s s|C)
and (p s|C) with lc <= 4, which accumulate Cartesian ket monomials: counted
here from the exponents.  And, of the others, the harmonic weights' powers of
x + i y once."""
import pytest

import paper_2210_03192_gb300 as lx
from oracle.solid import cart_list, solid_matrix


def per_primitive(la, lb, lc):
    return lx.class_flops(la, lb, lc, 2) - lx.class_flops(la, lb, lc, 1)


def products(factors):
    return max(0, factors - 1)


@pytest.mark.parametrize("lc", range(7))
def test_ss(lc):
    mono = [sum(x > 0 for x in c) for c in cart_list(lc)]
    # geometry without (rho/gamma) PC, powers, Boys function, monomials, sums
    prim = 29 + (4 * (lc - 1) if lc else 0) + 16 + sum(products(n) for n in mono) + 2 * len(mono)
    assert per_primitive(0, 0, lc) == prim
    # targets (one term each), ket transform
    assert lx.class_flops(0, 0, lc, 1) - prim == 2 * len(mono) + 2 * int((solid_matrix(lc) != 0).sum())


@pytest.mark.parametrize("lc", range(5))
def test_ps(lc):
    mono = [sum(x > 0 for x in c) for c in cart_list(lc)]
    less = [sum(x > 0 for x in c) for c in cart_list(lc - 1)] if lc else []
    prim = 32 + (4 * (lc - 1) if lc else 0) + 35 + 3 * 3  # Boys and one order down; the VRR1 step
    prim += sum(products(n) for n in mono) + sum(products(n + 1) for n in less)  # X^c, Y X^n
    prim += 2 * (3 * len(mono) + len(less))
    assert per_primitive(1, 0, lc) == prim


def test_harmonic_weights_counted_once():
    """(p p|i) against (p p|h): one more power of x + i y is 6 flops, not six
    times as many as lanes that form it."""
    def weights(lc, lab):  # X: r^2, powers, Q recursions, products with Y^k and the power
        k = min(lab, lc)
        return (5 + 6 * (lc - 1) + sum(4 * max(0, lc - m - 1) for m in range(lc + 1)) +
                sum((j > 0) + (2 if m else 0) for m in range(lc + 1) for j in range(min(k, lc - m) + 1)))

    def accumulators(lc):  # (e, k) for e of degree 2 (k = 0), 1 (k <= 1), 0 (k <= 2)
        pairs = {(tuple(a[i] - u[i] for i in range(3)), sum(u))
                 for l in (1, 2) for a in cart_list(l)
                 for u in ((x, y, z) for x in range(a[0] + 1) for y in range(a[1] + 1) for z in range(a[2] + 1))
                 if sum(u) <= lc}
        return sum(2 * (lc - k) + 1 for _, k in pairs)

    diff = per_primitive(1, 1, 6) - per_primitive(1, 1, 5)
    assert diff == weights(6, 2) - weights(5, 2) + 2 * (accumulators(6) - accumulators(5))
