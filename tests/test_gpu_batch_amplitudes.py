"""Batched FP64 members under an envelope that varies in time, in the collisions that
take the amplitudes of both half steps: the same lattice stepped alone, bit for bit on
D3Q27 and D2Q5, on D2Q9 and D3Q15 up to the compiler's multiply-add contraction."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ONE = np.array([1.0])
GENERAL = {lbm.D2Q9: W.d2q9_omega(0.7, 1.1, 1.2, 1.3, 1.4), lbm.D2Q5_CDE: W.d2q5_omega(0.7, 1.1, 0.9),
           lbm.D3Q27: W.d3q27_omega(0.7, 1.1, (1.2, 1.3, 1.4, 1.5)), lbm.D3Q15: W.d3q15_omega(0.7, 1.1, 1.2, 1.3)}


def _envelope(t):
    return 2.0 ** -40 / 3.0 if t % 2 else 1.0 + 0.1 * np.sin(t)  # every other amplitude much smaller


# 2 members: amplitudes in the launch arguments; 40: in a table; graph replays: in the graph's table
@pytest.mark.parametrize("members,graph", [(2, 0), (40, 0), (2, 4)])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE, lbm.D3Q27, lbm.D3Q15])
def test_general_collisions_are_the_single_lattice_ones(lattice, members, graph):
    """Contraction moves single roundings of 2^-53 of values of order 1: a few per
    population and step."""
    shape = {2: (9, 7, 1), 3: (5, 4, 3)}[2 if lattice in (lbm.D2Q9, lbm.D2Q5_CDE) else 3]

    def make(k):
        rng = np.random.default_rng(k)
        L = lbm.Lattice(lattice, shape, GENERAL[lattice], wall=(0, 0 if lattice == lbm.D2Q5_CDE else 1, 0))
        L.init_equilibrium(1.0, 0.02 * rng.standard_normal((L.dim, L.N)))
        if lattice == lbm.D2Q5_CDE:
            L.set_velocity(full=0.05 * rng.standard_normal((2, L.N)))
            L.set_source([(1e-3 * rng.standard_normal(shape[0]), ONE, ONE)])
        else:
            L.set_force([(1e-3 * rng.standard_normal(shape[0]), ONE, ONE) for _ in range(L.dim)])
        L.set_envelope(_envelope, 16)
        return L

    batched, alone = [make(k) for k in range(members)], [make(k) for k in range(members)]
    B = lbm.Batch(batched)
    if graph:
        B.set_graph(graph)
    B.step(8)
    for a, b in zip(alone, batched):
        for _ in range(8):
            a.step(1)
        fa, fb = a.get_populations(), b.get_populations()
        if lattice in (lbm.D3Q27, lbm.D2Q5_CDE):
            assert np.array_equal(fa, fb)
        else:
            assert np.abs(fa - fb).max() <= 8 * 8 * 2.0 ** -53
