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
    off = np.array([math.fsum([*f[:, k], -rho[k]]) for k in range(L.N)])  # the exact difference
    assert (np.abs(off) <= err).all()
    exact = np.array([math.fsum(f[:, k]) for k in range(L.N)])
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


def _oracle(lattice, shape, wall, omega, f, tables=None, uadv=None):
    from oracle import oracle as O
    R = O.OracleContext(lattice, shape, omega=omega, wall=wall)
    assert R.set_populations(f, 0) == 0
    if tables is not None:
        P = O.expand_separable(tables, shape)
        assert (R.set_source(P[0]) if lattice == lbm.D2Q5_CDE else R.set_force(P)) == 0
    if uadv is not None:
        n = int(np.prod(shape))
        assert R.set_velocity(np.repeat(np.asarray(uadv)[:, None], n, axis=1)) == 0
    return R


@pytest.mark.parametrize("kind", ["plain", "mixed", "negative", "fast", "tiny", "huge", "forced"])
@pytest.mark.parametrize("lattice", [lbm.D2Q9, lbm.D2Q5_CDE, lbm.D3Q27, lbm.D3Q15])
def test_step_in_and_out_of_range(lattice, kind):
    """One step of every single-lattice and batched launch from states on both
    sides of what the fixed-point form takes (scale, sign, speed, size of the
    force), walls on one axis, against the oracle to the parity bar: 1e-12 of the
    largest population."""
    rng = np.random.default_rng(11)
    q, shape = lbm.Q[lattice], SHAPE[lattice]
    n = int(np.prod(shape))
    e = np.array([_velocity(lattice, a) for a in range(q)], dtype=np.float64)
    w = np.array([_weight(lattice, a) for a in range(q)])
    speed = 0.35 if kind == "fast" else 0.02
    u = speed * rng.standard_normal((e.shape[1], n))
    f = w[:, None] * (1.0 + 3.0 * (e @ u)) * (1.0 + 0.01 * rng.standard_normal((q, n)))
    if kind == "mixed":  # one node in three far outside the others' scale
        f[:, ::3] *= 2.0 ** rng.integers(-700, 1, (1, len(range(0, n, 3))))
    elif kind == "negative":
        f[1, ::4] *= -0.3
    elif kind == "tiny":
        f *= 2.0 ** -600
    elif kind == "huge":
        f *= 2.0 ** 55
    f = np.ascontiguousarray(f)
    scale = np.abs(f).max()
    x = np.arange(shape[0])
    # (no force where a node's density may be 2^-700: the method itself overflows there)
    amp = {"forced": 0.4, "mixed": 0.0}.get(kind, 1e-4) * scale
    one = np.array([1.0])
    comp = [(amp * np.sin(1.0 + x), one, one), (amp * np.cos(x), one, one), (amp * np.sin(2.0 * x), one, one)]
    scalar = lattice == lbm.D2Q5_CDE
    wall = (0, 0, 0) if scalar else (0, 1, 0)
    for ncomp in (1,) if scalar else (1, 3 if q > 9 else 2):
        dims = 1 if scalar else (2 if q == 9 else 3)
        tables = [comp[d] if d < ncomp else (np.zeros(shape[0]), one, one) for d in range(dims)]
        R = _oracle(lattice, shape, wall, OMEGA[lattice], f, tables, (0.05, -0.02) if scalar else None)
        assert R.step(1) == 0
        ref = R.populations()[1]
        for members in (0, 2):
            lats = []
            for _ in range(max(1, members)):
                L = lbm.Lattice(lattice, shape, OMEGA[lattice], wall=wall)
                if scalar:
                    L.set_velocity(tables=[(np.array([0.05]), one, one), (np.array([-0.02]), one, one)])
                    L.set_source(tables=tables)
                else:
                    L.set_force(tables=tables)
                L.set_populations(f)
                lats.append(L)
            if members:
                B = lbm.Batch(lats)
                B.step(1)
            else:
                lats[0].step(1)
            for L in lats:
                assert np.abs(L.get_populations() - ref).max() <= 1e-12 * scale


def _weight(lattice, a):
    e = np.abs(_velocity(lattice, a)).sum()
    if lattice == lbm.D3Q27:
        return (2 / 3) ** (3 - e) * (1 / 6) ** e
    if lattice == lbm.D3Q15:
        return (2 / 9, 1 / 9, 0, 1 / 72)[e]
    if lattice == lbm.D2Q5_CDE:
        return (1 / 3, 1 / 6)[e]
    return (4 / 9, 1 / 9, 1 / 36)[e]


def test_step_passes_nan_on():
    """A NaN population is passed on by the step (and reported by lbm_reduce)."""
    for lattice in (lbm.D2Q9, lbm.D2Q5_CDE, lbm.D3Q27, lbm.D3Q15):
        L = lbm.Lattice(lattice, SHAPE[lattice], OMEGA[lattice])
        L.init_equilibrium(1.0)
        f = L.get_populations()
        f[2, 3] = np.nan
        L.set_populations(f)
        L.step(1)
        assert np.isnan(L.get_populations()).any()
        with pytest.raises(lbm.LBMError):
            L.reduce()
