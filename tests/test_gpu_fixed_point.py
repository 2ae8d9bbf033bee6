"""Fixed-point arithmetic of the FP64 kernels (csrc/lbm_fixed.cuh): the sums of
the readbacks over every scale and sign a state can have, against exact sums."""
import math

import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# S of csrc/lbm_fixed.cuh FxGrid: a population is rounded at 2^-S of the power of
# two at or below the node's largest one (D2Q5 is summed in FP64)
GRID = {lbm.D3Q27: 55, lbm.D3Q15: 56, lbm.D2Q9: 57, lbm.D2Q5_CDE: 53}
SHAPE = {lbm.D3Q27: (7, 5, 3), lbm.D3Q15: (5, 4, 9), lbm.D2Q9: (33, 5, 1), lbm.D2Q5_CDE: (31, 6, 1)}
OMEGA = {lbm.D3Q27: W.d3q27_omega(0.7), lbm.D3Q15: W.d3q15_omega(0.7), lbm.D2Q9: W.d2q9_omega(0.7),
         lbm.D2Q5_CDE: W.d2q5_omega(0.7)}


def _state(lattice, kind, rng):
    q = lbm.Q[lattice]
    n = int(np.prod(SHAPE[lattice]))
    f = rng.uniform(0.01, 1.0, (q, n))
    if kind == "signed":
        f *= rng.choice([-1.0, 1.0], (q, n))
        f[0] = 1.0 + q
    elif kind == "spread":  # 200 binary orders of magnitude inside a node
        f *= 2.0 ** rng.integers(-200, 1, (q, n))
    elif kind == "tiny":  # below the fixed-point range
        f *= 2.0 ** -600
    elif kind == "huge":  # above it
        f *= 2.0 ** 60
    elif kind == "edge":  # both sides of the range's upper end, node by node
        f *= 2.0 ** rng.integers(48, 53, (1, n))
    elif kind == "zeros":
        f[1:] = 0.0
    return np.ascontiguousarray(f)


@pytest.mark.parametrize("kind", ["plain", "signed", "spread", "tiny", "huge", "edge", "zeros"])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE, lbm.D3Q27, lbm.D3Q15])
def test_readback_sums(lattice, kind):
    """rho and j of lbm_moments against exact sums: each population rounded at
    2^-S (Q / 2 units in all), the sum rounded once; outside the range, and on
    D2Q5, Q - 1 FP64 additions.  u = j (1/rho): two more roundings of 2^-53."""
    rng = np.random.default_rng(7)
    f = _state(lattice, kind, rng)
    L = lbm.Lattice(lattice, SHAPE[lattice], OMEGA[lattice])
    L.set_populations(f)
    got = L.moments(half_forced=False)
    rho, u = (got, None) if lattice == lbm.D2Q5_CDE else got
    q = lbm.Q[lattice]
    e = np.array([_velocity(lattice, a) for a in range(q)])
    top = np.abs(f).max(axis=0)
    if kind in ("tiny", "huge", "edge") or lattice == lbm.D2Q5_CDE:
        err = q * 2.0 ** -53 * np.abs(f).sum(axis=0)
    else:
        err = 0.5 * q * 2.0 ** -GRID[lattice] * top + 2.0 ** -53 * np.abs(f.sum(axis=0))
    exact = np.array([math.fsum(f[:, k]) for k in range(L.N)])
    assert (np.abs(rho - exact) <= err).all()
    if u is None:
        return
    for d in range(L.dim):
        j = np.array([math.fsum(f[:, k] * e[:, d]) for k in range(L.N)])
        bound = (err + 2.0 ** -53 * np.abs(j)) / np.abs(exact) + np.abs(j / exact) * (err / np.abs(exact) + 2.0 ** -51)
        assert (np.abs(u[d] - j / exact) <= bound).all()


def _velocity(lattice, a):
    if lattice == lbm.D3Q27:
        return (a % 3 - 1, (a // 3) % 3 - 1, a // 9 - 1)
    if lattice == lbm.D3Q15:
        axes = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        return axes[a] if a < 7 else (1 if a % 2 else -1, -1 if ((a - 7) // 2) % 2 else 1, 1 if a <= 10 else -1)
    nine = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    return nine[a]


@pytest.mark.parametrize("storage", [lbm.FP32_DEV, lbm.FP16_DEV, lbm.BF16_DEV])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE, lbm.D3Q27])
@pytest.mark.parametrize("amp", [0.0, 1e-3, 1e-30])
def test_readback_sums_of_deviations(lattice, storage, amp):
    """The deviations' sums (24-bit integers, 32 bits below the node's largest
    one's last) plus the reference, against the populations read back in FP64:
    those are rounded once each (Q 2^-53 in all), u to three more roundings."""
    rng = np.random.default_rng(3)
    q, shape = lbm.Q[lattice], SHAPE[lattice]
    n = int(np.prod(shape))
    L = lbm.Lattice(lattice, shape, OMEGA[lattice], storage=storage)
    L.init_equilibrium(1.0)
    f = L.get_populations()
    f = f + amp * rng.standard_normal((q, n)) * 10.0 ** rng.integers(-6, 1, (q, n))
    L.set_populations(f)
    f = L.get_populations()
    got = L.moments(half_forced=False)
    rho, u = (got, None) if lattice == lbm.D2Q5_CDE else got
    assert np.abs(rho - f.sum(axis=0)).max() <= 2 * q * 2.0 ** -53
    if u is not None:
        e = np.array([_velocity(lattice, a) for a in range(q)])
        for d in range(L.dim):
            assert np.abs(u[d] - (f * e[:, d, None]).sum(axis=0) / rho).max() <= 2 * q * 2.0 ** -53
