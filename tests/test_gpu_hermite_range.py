"""J and forces from unit-normalised shells, l = 4 to 6, exponents from 0.01 to
1e4 on one centre and one beside it: the Hermite potentials behind them span
h^-6 (h = 1/(2 gamma)) where J itself is of the size of c, for coefficients c
of 1e-8, 1 and 1e8.  Tolerances as for the other DF-J and gradient tests, with
the absolute term at the scale of c: J and gamma sampled_against_oracle's
1e-12 sum |I||w| + 1e-14 sum |w|, gradient 1e-11 of max|F|, in binary128."""
import math
from types import SimpleNamespace

import numpy as np
import pytest

import oracle
from dfj_sampling import sampled_against_oracle
from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ATOMS = np.array([[0.0, 0.0, 0.0], [1.1, 0.4, -0.7]])


@pytest.fixture(scope="module")
def lx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as m
    return m


def normalised(l, z):
    """Coefficient of a unit-normalised solid-harmonic shell (Racah S_l)."""
    a = 2.0 * z
    return math.sqrt((2 * l + 1) / (4 * math.pi) * 2.0 * a ** (l + 1.5) / math.gamma(l + 1.5))


def problem(l):
    shells = [(l, 0.01, 0), (l, 0.3, 0), (l, 30.0, 0), (l, 1e4, 0), (l, 0.8, 1), (0, 0.5, 1)]
    orb = W.make_basis([s[0] for s in shells], [1] * len(shells), ATOMS[[s[2] for s in shells]],
                       [s[1] for s in shells], [normalised(s[0], s[1]) for s in shells], [s[2] for s in shells])
    kets = [(0, 0.02, 1), (0, 1e4, 0), (2, 1.0, 0), (3, 40.0, 1)]
    ones = W.make_basis([k[0] for k in kets], [1] * len(kets), ATOMS[[k[2] for k in kets]], [k[1] for k in kets],
                        [1.0] * len(kets), [k[2] for k in kets])
    d = np.diag(oracle.metric(ones))[oracle.ao_offsets(ones)[:-1]]
    aux = W.make_basis(ones.l, ones.k, ones.xyz, ones.exps, 1.0 / np.sqrt(d), ones.atom)
    return orb, aux


def density_and_c(orb, aux, l, scale):
    rng = np.random.default_rng(40 + l)
    return (W.density(rng, int(oracle.ao_offsets(orb)[-1])),
            scale * rng.standard_normal(int(oracle.ao_offsets(aux)[-1])))


@pytest.mark.parametrize("scale", [1e-8, 1.0, 1e8])
@pytest.mark.parametrize("l", [4, 5, 6])
def test_J_of_normalised_shells(lx, l, scale):
    orb, aux = problem(l)
    D, c = density_and_c(orb, aux, l, scale)
    plan = lx.DFJPlan(orb, aux, 0.0)
    g, J = (x.cpu().numpy() for x in plan.execute(torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")))
    npair = orb.nshell * (orb.nshell + 1) // 2
    sampled_against_oracle(SimpleNamespace(orb=orb, aux=aux), plan, D, c, g, J, npair, aux.nshell, 1, "quad", 1e-12)


@pytest.mark.parametrize("scale", [1e-8, 1.0, 1e8])
@pytest.mark.parametrize("l", [4, 5])
def test_gradient_of_normalised_shells(lx, l, scale):
    orb, aux = problem(l)
    D, c = density_and_c(orb, aux, l, scale)
    plan = lx.DFJPlan(orb, aux, 0.0, gradient=True)
    G = plan.gradient(torch.tensor(D, device="cuda"), torch.tensor(c, device="cuda")).cpu().numpy()
    Go = oracle.dfj_grad(orb, aux, D, c, 2, tasks=plan.tasks(), mode="quad")
    assert np.abs(G - Go).max() <= 1e-11 * np.abs(Go).max()
