"""The Hermite-basis DF-J build and gradient (csrc/hermite.cu) at the edges of
its tiles: one ket shell, one more and one less than a tile's 32, contracted
ket shells, s to h orbitals with every auxiliary l, pairs whose ket lists end
at different places, gamma alone and J alone.  Tolerances as for the other
DF-J and gradient tests: normwise 1e-12 (values) and 1e-11 of max|F| against
the binary128 oracle over the same screened triples."""
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


def shells(rng, recipe, coords, exp_lo, exp_hi):
    """(l, count, K) shells over the atoms in turn."""
    ls, ks, xyz, ex, co, at = [], [], [], [], [], []
    for l, count, K in recipe:
        for i in range(count):
            ia = i % len(coords)
            ls.append(l); ks.append(K); xyz.append(coords[ia]); at.append(ia)
            ex.append(np.exp(rng.uniform(np.log(exp_lo), np.log(exp_hi), K)))
            co.append(rng.uniform(0.1, 1.0, K))
    return W.make_basis(ls, ks, np.array(xyz), np.concatenate(ex), np.concatenate(co), at)


CASES = {
    "one_ket": ([(1, 2, 2), (2, 1, 1)], [(2, 1, 1)]),
    "tile_less_one": ([(1, 2, 2), (2, 2, 1)], [(0, 31, 1), (1, 31, 1), (5, 1, 1)]),
    "tile_plus_one": ([(1, 1, 3), (2, 1, 2), (3, 1, 1)], [(0, 33, 1), (3, 33, 1), (6, 3, 1)]),
    "contracted_kets": ([(0, 1, 2), (1, 1, 2), (2, 1, 1), (3, 1, 1)], [(0, 5, 3), (2, 3, 2), (4, 2, 2), (6, 1, 3)]),
    "high_l": ([(0, 1, 1), (4, 1, 1), (5, 1, 1)], [(l, 2, 1) for l in range(7)]),
}


def problem(name, hi):
    rng = np.random.default_rng(sorted(CASES).index(name) + 10)
    coords = np.array([[0.0, 0.0, 0.0], [1.7, 0.4, -0.6], [-0.9, 1.5, 7.0]])
    orb, aux = CASES[name]
    return shells(rng, orb, coords, 0.1, hi), shells(rng, aux, coords, 0.1, hi), rng


@pytest.mark.parametrize("name", sorted(CASES))
def test_gamma_and_J(lx, name):
    orb, aux, rng = problem(name, 300.0)
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    D, c = W.density(rng, n), rng.standard_normal(na)
    plan = lx.DFJPlan(orb, aux, 1e-10)  # some ket lists end early
    Dt, ct = torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")
    g, J = plan.execute(Dt, ct)
    go, Jo = oracle.dfj(orb, aux, D, c, tasks=plan.tasks(), mode="quad")
    assert np.abs(g.cpu().numpy() - go).max() <= 1e-12 * np.abs(go).max()
    assert np.abs(J.cpu().numpy() - Jo).max() <= 1e-12 * np.abs(Jo).max()
    g1, _ = plan.execute(Dt, ct, outputs="gamma")
    _, J1 = plan.execute(Dt, ct, outputs="J")
    assert torch.equal(g1, g) and torch.equal(J1, J)


@pytest.mark.parametrize("name", ["one_ket", "tile_plus_one", "contracted_kets"])
def test_gradient(lx, name):
    orb, aux, rng = problem(name, 100.0)
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    D, c = W.density(rng, n), rng.standard_normal(na)
    plan = lx.DFJPlan(orb, aux, 1e-10, gradient=True)
    G = plan.gradient(torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")).cpu().numpy()
    Go = oracle.dfj_grad(orb, aux, D, c, plan.natom, tasks=plan.tasks(), mode="quad")
    assert np.abs(G - Go).max() <= 1e-11 * np.abs(Go).max()


@pytest.mark.parametrize("count", [1, 2, 3, 5, 17, 31, 32, 33, 65])
def test_register_kernels_ket_widths(lx, count):
    """(s s|C) and (p s|C) ket lists of every width that shares a warp, the
    last group of a launch partly empty, primitives of unequal number."""
    rng = np.random.default_rng(100 + count)
    coords = np.array([[0.0, 0.0, 0.0], [1.7, 0.4, -0.6], [-0.9, 1.5, 3.0]])
    orb = shells(rng, [(0, 3, 1), (0, 2, 3), (1, 2, 2), (1, 1, 1)], coords, 0.1, 300.0)
    aux = shells(rng, [(0, count, 1), (2, count, 1), (3, 1, 2), (6, 2, 1)], coords, 0.1, 300.0)
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    D, c = W.density(rng, n), rng.standard_normal(na)
    plan = lx.DFJPlan(orb, aux, 1e-10)
    g, J = (x.cpu().numpy() for x in plan.execute(torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")))
    go, Jo = oracle.dfj(orb, aux, D, c, tasks=plan.tasks(), mode="quad")
    assert np.abs(g - go).max() <= 1e-12 * np.abs(go).max()
    assert np.abs(J - Jo).max() <= 1e-12 * np.abs(Jo).max()


@pytest.mark.parametrize("lc", range(7))
@pytest.mark.parametrize("la,lb", [(1, 0), (1, 1), (2, 1), (2, 2), (3, 2), (3, 3)])
def test_unrolled_classes(lx, la, lb, lc):
    """Every class of the unrolled kernel, and its neighbours on the table
    kernel: one shell more than half a tile, contracted and plain kets, values
    and gradient."""
    rng = np.random.default_rng(1000 + 100 * la + 10 * lb + lc)
    coords = np.array([[0.0, 0.0, 0.0], [1.7, 0.4, -0.6], [-0.9, 1.5, 3.0]])
    orb = shells(rng, [(la, 1, 2), (lb, 2, 1)], coords, 0.1, 100.0)
    aux = shells(rng, [(lc, 17, 1), (lc, 2, 2)], coords, 0.1, 100.0)
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    D, c = W.density(rng, n), rng.standard_normal(na)
    Dt, ct = torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")
    plan = lx.DFJPlan(orb, aux, 1e-10, gradient=True)
    g, J = plan.execute(Dt, ct)
    go, Jo = oracle.dfj(orb, aux, D, c, tasks=plan.tasks(), mode="quad")
    assert np.abs(g.cpu().numpy() - go).max() <= 1e-12 * np.abs(go).max()
    assert np.abs(J.cpu().numpy() - Jo).max() <= 1e-12 * np.abs(Jo).max()
    assert torch.equal(plan.execute(Dt, ct, outputs="gamma")[0], g)
    assert torch.equal(plan.execute(Dt, ct, outputs="J")[1], J)
    G = plan.gradient(Dt, ct).cpu().numpy()
    Go = oracle.dfj_grad(orb, aux, D, c, plan.natom, tasks=plan.tasks(), mode="quad")
    assert np.abs(G - Go).max() <= 1e-11 * np.abs(Go).max()


@pytest.mark.parametrize("nd", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("count", [1, 2, 3, 7, 16, 33])
def test_register_kernels_several_densities(lx, count, nd):
    """(s s|C) and (p s|C) for several densities at every width of a tile:
    each density as by itself (1e-13, only the order of sums differs)."""
    rng = np.random.default_rng(500 + 10 * count + nd)
    coords = np.array([[0.0, 0.0, 0.0], [1.7, 0.4, -0.6], [-0.9, 1.5, 3.0]])
    orb = shells(rng, [(0, 3, 1), (0, 2, 3), (1, 2, 2), (1, 1, 1)], coords, 0.1, 300.0)
    aux = shells(rng, [(0, count, 1), (2, count, 1), (4, 1, 2), (6, 2, 1)], coords, 0.1, 300.0)
    n, na = int(oracle.ao_offsets(orb)[-1]), int(oracle.ao_offsets(aux)[-1])
    plan = lx.DFJPlan(orb, aux, 1e-10)
    D = torch.tensor(np.stack([W.density(rng, n) for _ in range(nd)]), device="cuda")
    c = torch.tensor(rng.standard_normal((nd, na)), device="cuda")
    g, J = plan.execute_multi(D, c)
    for k in range(nd):
        g1, J1 = plan.execute(D[k].contiguous(), c[k].contiguous())
        assert (g[k] - g1).abs().max() <= 1e-13 * g1.abs().max()
        assert (J[k] - J1).abs().max() <= 1e-13 * J1.abs().max()
    assert (plan.execute_multi(D, None, outputs="gamma")[0] - g).abs().max() <= 1e-13 * g.abs().max()
    assert (plan.execute_multi(None, c, outputs="J")[1] - J).abs().max() <= 1e-13 * J.abs().max()
