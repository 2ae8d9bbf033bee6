"""lbm_reduce at densities whose reciprocal is not an FP64 number."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from test_gpu_fixed_point import OMEGA, SHAPE, _velocity, _weight

pytestmark = pytest.mark.gpu


def _state(lattice, scale, s):
    q, n = lbm.Q[lattice], int(np.prod(SHAPE[lattice]))
    w = np.array([_weight(lattice, a) for a in range(q)])
    ex = np.array([_velocity(lattice, a)[0] for a in range(q)], dtype=np.float64)
    return np.repeat((scale * (w * (1.0 + 3.0 * s * ex)))[:, None], n, axis=1)


@pytest.mark.parametrize("scale", [2.0 ** -1030, 2.0 ** -1020, 1.0, 2.0 ** 1018])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D3Q27, lbm.D3Q15])
def test_any_density_is_reduced(lattice, scale):
    """The velocities of such a state are ordinary numbers: it is no instability, and it does
    not change between two calls."""
    L = lbm.Lattice(lattice, SHAPE[lattice], OMEGA[lattice])
    L.set_populations(_state(lattice, scale, 0.1))
    L.reduce()
    assert L.reduce()[4] == 0.0


@pytest.mark.parametrize("value", [0.0, -1.0, np.nan, np.inf])
def test_no_density_is_an_instability(value):
    L = lbm.Lattice(lbm.D2Q9, SHAPE[lbm.D2Q9], OMEGA[lbm.D2Q9])
    f = _state(lbm.D2Q9, 1.0, 0.1)
    f[:, 5] = value
    L.set_populations(f)
    with pytest.raises(lbm.LBMError):
        L.reduce()
