"""The fixed-point scalar collision over every uniform velocity that it takes, and
beyond: accurate where it applies, reported where it does not."""
import numpy as np
import pytest

from test_fixed_point_cpu import call, d2q5, host  # noqa: F401


@pytest.mark.parametrize("u", [(0.75, 0.75), (0.8, 0.8), (0.89, -0.89), (-0.89, 0.89), (0.89, 0.0), (0.0, -0.89),
                               (-0.6, -0.6), (0.95, 0.0), (1.5, -2.0)])
@pytest.mark.parametrize("w12", [0.05, 1.4, 1.9, 1.99])
@pytest.mark.parametrize("w34", [0.05, 0.2, 1.0, 1.99])
def test_scalar_collision_at_large_velocities(host, u, w12, w34):  # noqa: F811
    rng = np.random.default_rng(3)
    g = np.array([1 / 3] + [1 / 6] * 4) + 0.3 * rng.standard_normal((500, 5))
    g[::5] = rng.choice([-1.0, 1.0], (100, 5)) * (2.0 - 2.0 ** -40)  # all as large as the scale has room for
    P = 1e-3 * rng.standard_normal(500)
    om = np.array([0.0, w12, w12, w34, w34])
    got, ok = call(host.fixed5, g, P, 0.7, 0.2, om, *u)
    S, Sq = np.longdouble(0.7) * P, np.longdouble(0.2) * P
    ref, dbl = [d2q5(g, S, Sq, om, *u, T)[ok] for T in (np.longdouble, np.float64)]
    c1, c3 = w12 / 2, w34 / 4
    r2 = u[0] ** 2 + u[1] ** 2
    taken = max(abs(u[0]), abs(u[1])) < 0.9 and abs(c3 * (2 / 3 - r2) + c1 * r2) < 0.99
    assert ok.mean() > 0.9 if taken else not ok.any()
    if taken:
        assert np.abs(got[ok] - ref).max() <= np.abs(dbl - ref).max()
