"""Stochastic rounding to FP16 over its magnitude ranges: each stored value is one
of the two neighbours of the FP32 deviation, the one further from zero as often
as the distance says."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# four, two and one node per thread; FP16-subnormal, normal and large deviations
@pytest.mark.parametrize("nx", [512, 514, 513])
@pytest.mark.parametrize("scale", [2e-7, 3e-5, 2.0 ** -14, 0.02, 3000.0])
def test_fp16_share_of_each_neighbour(nx, scale):
    """2^18 nodes of one value: the share of the upper neighbour within 5 standard
    deviations of a fair draw (5 * 0.5 / 512) and what FP32 rounding of the value
    in the collision moves it (a few 2^-24 of the value, 2^-11 of a step each: 0.003)."""
    shape = (nx, 512, 1)
    omega = W.d2q5_omega(0.7)
    w = np.array([1 / 3, 1 / 6, 1 / 6, 1 / 6, 1 / 6])
    d = scale * np.array([0.37, -0.21, 0.45, 0.13, -0.3])
    A = lbm.Lattice(lbm.D2Q5_CDE, shape, omega, storage=lbm.FP16_DEV)
    B = lbm.Lattice(lbm.D2Q5_CDE, shape, omega, storage=lbm.FP32_DEV)
    A.init_equilibrium(1.0)
    B.init_equilibrium(1.0)
    A.set_populations(np.repeat((w + d)[:, None], A.N, axis=1))
    B.set_populations(A.get_populations())
    A.set_stochastic_rounding(True, seed=5)
    A.step(1)
    B.step(1)
    fa, fb = A.get_populations(), B.get_populations()
    for a in range(5):
        v = fb[a, 0] - w[a]
        assert np.all(fb[a] == fb[a, 0])
        lo = np.float16(v)
        if abs(float(lo)) > abs(v):
            lo = np.nextafter(lo, np.float16(0))
        step = abs(float(np.nextafter(lo, np.float16(np.copysign(np.inf, v)))) - float(lo))
        k = np.round((np.abs(fa[a] - w[a]) - abs(float(lo))) / step)
        assert np.all((k == 0) | (k == 1)), (a, v, np.unique(k))
        share = (abs(v) - abs(float(lo))) / step
        assert abs(np.mean(k) - share) <= 5 * 0.5 / 512 + 0.003, (a, v, np.mean(k), share)
