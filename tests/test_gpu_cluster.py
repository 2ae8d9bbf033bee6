"""Small D2Q9 lattices step in one launch: the result does not depend on how the steps
are cut into calls, is that of single-step launches, and nodes that leave the
fixed-point form take the FP64 one."""
import numpy as np
import pytest

from paper_1806_10247_gb300 import lbm
from paper_1806_10247_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ONE = np.array([1.0])
STEPS = 24


def _lattice(shape, kind, omega):
    rng = np.random.default_rng(9)
    L = lbm.Lattice(lbm.D2Q9, shape, omega, wall=(0, 1, 0))
    rho = np.ones(L.N)
    force = 1e-5
    if kind == "force":  # as large as a channel of a few rows allows (a centre line at 0.1)
        force = 2e-3
    elif kind == "large force":  # F / 4 above 2^-6 of the largest population: the FP64 form at every node
        force = 0.03
    elif kind == "spread":  # neighbours far apart in scale
        rho[:: 3] = 2.0 ** -6
    L.init_equilibrium(rho, 0.01 * rng.standard_normal((2, L.N)) * rho)
    if kind == "zeros":  # no density at some nodes: the method divides by it
        f = L.get_populations()
        f[:, ::5] = 0.0
        L.set_populations(f)
    if kind != "none":
        L.set_force([(np.array([force]), ONE, ONE), (np.array([-0.3 * force]), ONE, ONE)])
    return L


# one block, several, the largest cluster; unit and general rates
@pytest.mark.parametrize("shape", [(3, 9, 1), (31, 17, 1), (70, 69, 1)])
@pytest.mark.parametrize("kind", ["none", "weak", "force", "large force", "spread", "zeros"])
@pytest.mark.parametrize("omega", [W.d2q9_omega(0.8), W.d2q9_omega(0.8, 1.1, 1.2, 1.3, 1.4)])
def test_cuts_and_single_steps(shape, kind, omega):
    steps = 2 if kind == "large force" else STEPS
    whole, cut, single = (_lattice(shape, kind, omega) for _ in range(3))
    n0 = whole.launch_count()
    whole.step(steps)
    assert whole.launch_count() == n0 + 1
    if steps > 2:
        for n in (2, 3, steps - 5):
            cut.step(n)
        assert np.array_equal(whole.get_populations(), cut.get_populations(), equal_nan=True)
    for _ in range(steps):
        single.step(1)
    f, g = whole.get_populations(), single.get_populations()
    fixed = omega[6] == 1.0 and kind in ("none", "weak", "force")
    if kind == "zeros":
        assert np.array_equal(np.isnan(f), np.isnan(g)) and np.isnan(g).any()
    elif fixed:  # every node in fixed point at every step: no contraction in it
        assert np.array_equal(f, g)
    else:  # the FP64 form's contraction: a few roundings per population and step
        assert np.abs(f - g).max() <= steps * 8 * 2.0 ** -53 * np.abs(g).max()


def test_restart_from_a_checkpoint(tmp_path):
    """Steps, a saved state, the rest of the steps in another lattice: the same bits."""
    a, b, c = (_lattice((31, 17, 1), "weak", W.d2q9_omega(0.8)) for _ in range(3))
    a.step(20)
    b.step(9)
    b.save_checkpoint(str(tmp_path / "c.npz"))
    c.load_checkpoint(str(tmp_path / "c.npz"))
    c.step(11)
    assert np.array_equal(a.get_populations(), c.get_populations())
