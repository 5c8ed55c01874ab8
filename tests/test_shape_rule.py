"""The planner's default tile against its rule, worked out here from the sizes
that lx3c_tile_hint makes visible: the largest T, then the largest balanced G
up to 8, that two CTAs per SM hold, T >= 64 only with three primitives side by
side; three CTAs where they take no fewer triples a tile, or still 32, with
two primitives (three for T >= 128)."""
import pytest

import paper_2210_03192_gb300 as lx

SM = 233472  # shared memory of an SM, 1 KB of it reserved per CTA


def balanced(K):
    """G for ever more chunks, the largest first."""
    out = []
    for chunks in range(1, K + 1):
        G = -(-K // chunks)
        if G <= 8 and G not in out:
            out.append(G)
    return out


def rule(la, lb, lc, K, naux):
    size = {}

    def bytes_of(T, G):
        if (T, G) not in size:
            lx.tile_hint(la, lb, lc, K, 1, T, G)
            try:
                q = lx.shape_query(la, lb, lc, K, 1, naux, 0)
            finally:
                lx.tile_hint(la, lb, lc, K, 1, 0, 0)
            size[T, G] = q[3] if q[:2] == (T, G) else 1 << 30  # does not fit one CTA: ignored
        return size[T, G]

    def fit(ctas, least):
        for T in (512, 256, 128, 64, 32, 16, 8, 4, 2, 1):
            if T > 1 and T >= 2 * naux:
                continue
            G = next((g for g in balanced(K) if bytes_of(T, g) <= (SM // ctas - 1024) // 8 * 8), 0)
            if G >= min(K, least(T)):
                return T, G, 0 if T >= 32 else 1, bytes_of(T, G)
        return None

    two = fit(2, lambda T: 3 if T >= 64 else 1)
    if two is None:
        return fit(1, lambda T: 1)
    three = fit(3, lambda T: 3 if T >= 128 else 2)
    return three if three and three[0] >= min(two[0], 32) else two


@pytest.mark.parametrize("K", [1, 2, 3, 6, 9, 36])
@pytest.mark.parametrize("la,lb,lc", [(1, 0, 5), (1, 1, 1), (1, 1, 2), (2, 0, 6), (2, 1, 2), (2, 2, 3), (3, 1, 0),
                                      (3, 2, 3), (3, 3, 2), (4, 0, 2), (4, 3, 0), (4, 4, 1), (4, 4, 6)])
def test_default_shape_is_the_rules(la, lb, lc, K):
    for naux in (1, 7, 33, 512):
        assert lx.shape_query(la, lb, lc, K, 1, naux, 0) == rule(la, lb, lc, K, naux), naux
