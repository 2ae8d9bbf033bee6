"""Every readback's velocity is j times the correctly rounded 1 / rho, j and rho the exact
sums rounded once, bit for bit."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from test_gpu_fixed_point import OMEGA

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,shape,right", [(lbm.D2Q9, (2048, 1024, 1), 1), (lbm.D3Q27, (128, 128, 64), 14),
                                                 (lbm.D3Q15, (128, 128, 64), 1)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300])
def test_velocity_bits(lattice, shape, right, scale):
    """Two populations a node, at rest (of any value) and along x (1/2): u = RN(1 / rho) / 2,
    a product without rounding."""
    rng = np.random.default_rng(8)
    q, n = lbm.Q[lattice], int(np.prod(shape))
    f = np.zeros((q, n))
    f[13 if lattice == lbm.D3Q27 else 0] = scale * rng.uniform(0.25, 1.0, n)
    f[right] = scale * 0.5
    rho_ref = f.sum(axis=0)  # one addition, rounded once
    L = lbm.Lattice(lattice, shape, OMEGA[lattice])
    L.set_populations(f)
    rho, u = L.moments(half_forced=False)
    assert np.array_equal(rho, rho_ref)
    assert np.array_equal(u[0], scale * 0.5 * (1.0 / rho))
    assert not u[1:].any()
