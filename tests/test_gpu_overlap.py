"""Steps of one call are placed while the step before still runs: their results
are those of the same steps made one call at a time, bit for bit."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 9


def _pair(make):
    a, b = make(), make()
    a.step(STEPS)
    for _ in range(STEPS):
        b.step(1)
    return a, b


@pytest.mark.parametrize("storage", [lbm.FP64, lbm.FP32_DEV, lbm.FP16_DEV])
@pytest.mark.parametrize("shape", [(70, 1, 1), (5, 33, 1), (191, 129, 1), (640, 515, 1)])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE])
def test_steps_of_one_call_2d(lattice, shape, storage):
    omega = W.d2q9_omega(0.7) if lattice == lbm.D2Q9 else W.d2q5_omega(0.7)

    def make():
        L = lbm.Lattice(lattice, shape, omega, wall=(0, 1 if lattice == lbm.D2Q9 else 0, 0), storage=storage)
        rng = np.random.default_rng(3)
        u = 0.02 * rng.standard_normal((2, L.N))
        L.init_equilibrium(1.0, u)
        if lattice == lbm.D2Q9:  # a force that may vary in time: a launch per step at every size
            L.set_envelope(lambda t: 1.0, STEPS)
        return L

    a, b = _pair(make)
    assert np.array_equal(a.get_populations(), b.get_populations())


# both sides of the D3Q27 FP64 line (2^20 nodes), part of a block per SM to several waves
@pytest.mark.parametrize("shape,storage", [((3, 5, 7), lbm.FP64), ((40, 40, 40), lbm.FP64), ((64, 64, 64), lbm.FP64),
                                           ((128, 128, 64), lbm.FP64), ((129, 128, 64), lbm.FP64),
                                           ((40, 40, 40), lbm.FP32_DEV), ((41, 40, 40), lbm.FP16_DEV)])
def test_steps_of_one_call_d3q27(shape, storage):
    def make():
        L = lbm.Lattice(lbm.D3Q27, shape, W.d3q27_omega(0.6), storage=storage)
        L.init_equilibrium(1.0, 0.02 * np.random.default_rng(4).standard_normal((3, L.N)))
        return L

    a, b = _pair(make)
    assert np.array_equal(a.get_populations(), b.get_populations())


@pytest.mark.parametrize("every", [2, 4])
def test_steps_of_one_call_at_a_local_reference(every):
    """Rebuilds lie between the steps: none is overlapped with the step after it."""
    def make():
        L = lbm.Lattice(lbm.D2Q9, (192, 130, 1), W.d2q9_omega(0.7), wall=(0, 1, 0), storage=lbm.FP16_DEV)
        L.set_local_reference(every)
        L.init_equilibrium(1.0, 0.02 * np.random.default_rng(5).standard_normal((2, L.N)))
        return L

    a, b = _pair(make)
    assert np.array_equal(a.get_populations(), b.get_populations())


@pytest.mark.parametrize("graph", [0, 4])
def test_steps_of_one_call_of_a_batch(graph):
    def make():
        Ls = []
        for k, s in enumerate([(33, 17, 1), (64, 64, 1), (200, 100, 1)]):
            L = lbm.Lattice(lbm.D2Q9, s, W.d2q9_omega(0.6 + 0.1 * k), wall=(0, 1, 0))
            L.init_equilibrium(1.0, 0.02 * np.random.default_rng(k).standard_normal((2, L.N)))
            Ls.append(L)
        return Ls, lbm.Batch(Ls)

    (la, a), (lb, b) = make(), make()
    if graph:
        a.set_graph(graph)
    a.step(STEPS)
    for _ in range(STEPS):
        b.step(1)
    for p, q in zip(la, lb):
        assert np.array_equal(p.get_populations(), q.get_populations())
