"""FP32 D2Q9 and D2Q5: two steps in one pass against the same steps made one call
at a time, bit for bit."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# a few more nodes than the line (136 MB of FP32 buffers), in strips of one column, of
# less, just and more than a block's, and a handful of very long rows
@pytest.mark.parametrize("wall,force", [((0, 0, 0), "separable"), ((0, 1, 0), "constant"), ((1, 0, 0), "none"),
                                        ((1, 1, 0), "separable")])
@pytest.mark.parametrize("nx", [1, 127, 128, 129, 2049, 700001])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE])
def test_two_steps_in_one_pass(lattice, nx, wall, force):
    omega = W.d2q9_omega(0.7) if lattice == lbm.D2Q9 else W.d2q5_omega(0.7)
    ny = (136 << 20) // (8 * lbm.Q[lattice]) // nx + 2
    rng = np.random.default_rng(3)
    state = (1.0, 0.02 * rng.standard_normal((2, nx * ny)))
    one = np.array([1.0])
    comps = 2 if lattice == lbm.D2Q9 else 1
    tables = {"constant": [(np.array([1e-4 * (k + 1)]), one, one) for k in range(comps)],
              "separable": [(1e-4 * rng.standard_normal(nx), rng.standard_normal(ny), one) for _ in range(comps)]}

    def make():
        L = lbm.Lattice(lattice, (nx, ny, 1), omega, wall=wall, storage=lbm.FP32_DEV)
        L.init_equilibrium(*state)
        if force != "none":
            (L.set_force if lattice == lbm.D2Q9 else L.set_source)(tables[force])
        L.set_envelope(lambda t: 1.0 + 0.1 * t, 8)  # another amplitude each half step
        return L

    a, b = make(), make()
    n0 = a.launch_count()
    a.step(5)
    assert a.launch_count() == n0 + 3
    for _ in range(5):
        b.step(1)
    assert a.t == b.t
    assert np.array_equal(a.get_populations(), b.get_populations())
