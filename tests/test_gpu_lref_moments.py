"""The fields of a lattice stored at a local reference, read without the FP32 copy,
against sums over its populations (which are read through the copy)."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [lbm.FP16_DEV, lbm.BF16_DEV])
@pytest.mark.parametrize("shape,wall", [((1, 3, 1), (0, 0, 0)), ((33, 9, 1), (0, 1, 0)), ((64, 40, 1), (0, 0, 0)),
                                        ((257, 31, 1), (1, 1, 0))])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE])
def test_fields_are_the_populations_sums(lattice, shape, wall, storage):
    """FP64 sums of values of order 1: a few 2^-53 each way."""
    omega = W.d2q9_omega(0.7) if lattice == lbm.D2Q9 else W.d2q5_omega(0.7)
    L = lbm.Lattice(lattice, shape, omega, wall=wall, storage=storage)
    L.set_local_reference(4)
    L.init_equilibrium(1.0, 0.02 * np.random.default_rng(6).standard_normal((2, L.N)))
    L.step(6)
    got = L.moments(half_forced=False)
    f = L.get_populations()
    if lattice == lbm.D2Q5_CDE:
        assert np.abs(got - f.sum(axis=0)).max() <= 2e-15
        return
    rho, u = got
    ex, ey = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    assert np.abs(rho - f.sum(axis=0)).max() <= 2e-15
    for e, v in zip((ex, ey), u):
        assert np.abs(v * rho - e @ f).max() <= 2e-15
