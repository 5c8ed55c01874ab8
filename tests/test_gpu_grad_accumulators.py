"""The bound of the contributions to one atom's force accumulators, by which a
gradient plan is refused at 2^32, is that atom's own: twice the atoms, each as
far from the others as before, take it up by their own pairs and kets only, not
by every tile of the plan."""
import ctypes

import numpy as np
import pytest

from paper_2210_03192_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bound(lx, natom):
    """natom atoms 60 bohr apart, tight shells: no pair or triple between them
    passes the screen but those of the Coulomb tail."""
    rng = np.random.default_rng(2)
    xyz = np.repeat(60.0 * np.arange(natom)[:, None] * np.array([[1.0, 0.0, 0.0]]), 3, axis=0)
    at = np.repeat(np.arange(natom), 3)
    orb = W.make_basis(np.tile([0, 1, 2], natom), np.ones(3 * natom, int), xyz, rng.uniform(1.0, 3.0, 3 * natom),
                       np.ones(3 * natom), at)
    aux = W.make_basis(np.tile([0, 1, 2], natom), np.ones(3 * natom, int), xyz, rng.uniform(1.0, 3.0, 3 * natom),
                       np.ones(3 * natom), at)
    plan = lx.DFJPlan(orb, aux, 1e-12, gradient=True)
    info = np.zeros(12)
    from paper_2210_03192_gb300 import _lib
    assert _lib.load().lx3c_dfj_info(plan.handle, info.ctypes.data, 12) == 0
    return info[11], plan


def test_bound_is_per_atom():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03192_gb300 as lx
    small, plan = bound(lx, 4)
    large, _ = bound(lx, 64)
    # six pairs and three kets an atom; every ket sees the pairs of all atoms
    # (Coulomb tail), one primitive each: at most 6 * 64 tiles with 32 lanes
    assert 0 < small < large <= 3 * 6 * 64 * 32 + 6 * 2
    # every ket's contributions are counted: no fewer than one per ket and class
    assert small >= 3
