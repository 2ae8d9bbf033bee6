"""The fixed-point collisions of csrc/lbm_fixed.cuh, compiled for the host, against
the collision of the method in extended precision: they must apply to every
ordinary state and be at least as accurate as the same collision in FP64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_10247_gb300", "csrc")
V9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
V27 = [(a % 3 - 1, (a // 3) % 3 - 1, a // 9 - 1) for a in range(27)]
V15 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
    [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
M15 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2),
       (1, 2, 0), (2, 1, 0), (2, 0, 1), (1, 1, 1), (2, 2, 0)]


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fx") / "fixed.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC,
                           os.path.join(HERE, "fixed_point_host.cpp"), "-o", so])
    return ctypes.CDLL(so)


def call(fn, f, P, *args):
    f, P = np.array(f, order="C"), np.ascontiguousarray(P)  # the results replace the copy
    ok = np.zeros(len(f), dtype=np.int32)
    dp = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    conv = [ctypes.c_double(a) if isinstance(a, float) else (dp(a) if isinstance(a, np.ndarray) else ctypes.c_int(a))
            for a in args]
    fn(ctypes.c_long(len(f)), dp(f), dp(P), *conv, dp(ok))
    return f, ok.astype(bool)


def product(f, F, Fq, vel, wb, wd, ws, T):
    """D2Q9 / D3Q27 with unit higher rates, in the number type T."""
    dim = len(vel[0])
    m = {tuple(c + 1 for c in e): f[:, a].astype(T) for a, e in enumerate(vel)}
    keys = sorted(m)

    def lines(d):
        return [[k[:d] + (i,) + k[d + 1:] for i in range(3)] for k in keys if k[d] == 0]

    for d in range(dim):
        for p, q, r in lines(d):
            m[p], m[q], m[r] = m[p] + m[q] + m[r], m[r] - m[p], m[r] + m[p]
    ax = [tuple(1 if i == d else 0 for i in range(dim)) for d in range(dim)]
    zero = (0,) * dim
    for d in range(dim):
        m[ax[d]] = m[ax[d]] + F[:, d].astype(T) / 2
    rho = m[zero]
    u = [m[a] / rho for a in ax]
    for d in range(dim):
        for p, q, r in lines(d):
            m[r] = m[r] - 2 * u[d] * m[q] + u[d] * u[d] * m[p]
            m[q] = m[q] - u[d] * m[p]
    two = [tuple(2 * c for c in a) for a in ax]
    tr = sum(m[a] for a in two)
    tr1 = tr + T(wb) * (T(dim) / 3 * rho - tr)
    c = {k: np.zeros_like(rho) for k in keys}
    for k in keys:
        if all(i in (0, 2) for i in k) and sum(k) != 2:
            c[k] = rho / T(3) ** (sum(k) // 2)
    for d in range(dim):
        c[two[d]] = tr1 / dim + (1 - T(wd)) * (m[two[d]] - tr / dim)
        for e in range(d + 1, dim):
            k = tuple(i + j for i, j in zip(ax[d], ax[e]))
            c[k] = (1 - T(ws)) * m[k]
    for d in range(dim):
        for p, q, r in lines(d):
            c[r] = c[r] + 2 * u[d] * c[q] + u[d] * u[d] * c[p]
            c[q] = c[q] + u[d] * c[p]
    for d in range(dim):
        g = (F[:, d].astype(T) + Fq[:, d].astype(T)) / (12 if dim == 2 else 36)
        for k in keys:
            if k[d] == 1 and all(i in (0, 2) for j, i in enumerate(k) if j != d):
                n = sum(1 for i in k if i == 2)
                if n == 0:
                    c[k] = c[k] + Fq[:, d].astype(T) / 2
                else:
                    c[k] = c[k] + g * (4 if dim == 2 else (12, 8)[n - 1])
    for d in range(dim):
        for p, q, r in lines(d):
            c[p], c[q], c[r] = (c[r] - c[q]) / 2, c[p] - c[r], (c[r] + c[q]) / 2
    return np.stack([c[tuple(i + 1 for i in e)] for e in vel], axis=1)


def d3q15(f, F, Fq, wb, ws, T):
    from math import comb
    M = np.array([[x ** a * y ** b * z ** c for x, y, z in V15] for a, b, c in M15], dtype=np.float64)
    # the inverse has entries in eighths and halves: exact
    Minv = np.round(np.linalg.inv(M) * 8) / 8
    assert np.array_equal(Minv @ M, np.eye(15))
    m = [sum(T(M[k, a]) * f[:, a].astype(T) for a in range(15) if M[k, a]) for k in range(15)]
    j = m[1:4]
    for d in range(3):
        m[1 + d] = m[1 + d] + F[:, d].astype(T) / 2
    rho = m[0]
    u = [m[1 + d] / rho for d in range(3)]
    at = {e: i for i, e in enumerate(M15)}

    def shift(v, s):
        return [sum(comb(e[0], i) * comb(e[1], k) * comb(e[2], l) * (s * u[0]) ** (e[0] - i) * (s * u[1]) ** (e[1] - k) *
                    (s * u[2]) ** (e[2] - l) * v[at[(i, k, l)]] for i in range(e[0] + 1) for k in range(e[1] + 1)
                    for l in range(e[2] + 1)) for e in M15]

    k = shift(m, -1)
    tr = k[7] + k[8] + k[9]
    tr1 = tr + T(wb) * (rho - tr)
    c = [np.zeros_like(rho) for _ in range(15)]
    c[0] = rho
    for i in (7, 8, 9):
        c[i] = tr1 / 3 + (1 - T(ws)) * (k[i] - tr / 3)
    for i in (4, 5, 6):
        c[i] = (1 - T(ws)) * k[i]
    c[14] = c[7] * c[8] / rho
    c = shift(c, 1)
    for d in range(3):
        s = F[:, d].astype(T) + Fq[:, d].astype(T)
        c[1 + d] = j[d] + s / 2
        c[10 + d] = c[10 + d] + s * 2 / 5
    return np.stack([sum(T(Minv[a, i]) * c[i] for i in range(15) if Minv[a, i]) for a in range(15)], axis=1)


def d2q5(g, S, Sq, om, ux, uy, T):
    g = [g[:, a].astype(T) for a in range(5)]
    ux, uy, om = T(ux), T(uy), [T(v) for v in om]
    kx, ky, xx, yy = g[1] - g[3], g[2] - g[4], g[1] + g[3], g[2] + g[4]
    S, Sq = S.astype(T), Sq.astype(T)
    phi = g[0] + xx + yy + S / 2
    h1, h2 = om[1] / 2 * (phi * ux - kx), om[2] / 2 * (phi * uy - ky)
    h3 = om[3] / 4 * (T(2) / 3 * phi - (xx + yy) + 2 * (ux * kx + uy * ky) - (ux * ux + uy * uy) * phi) + ux * h1 + uy * h2
    h4 = om[4] / 4 * (-(xx - yy) + 2 * (ux * kx - uy * ky) - (ux * ux - uy * uy) * phi) + ux * h1 - uy * h2
    H = (S + Sq) / 10
    return np.stack([g[0] + H - 4 * h3, g[1] + H + h3 + h1 + h4, g[2] + H + h3 + h2 - h4, g[3] + H + h3 - h1 + h4,
                     g[4] + H + h3 - h2 - h4], axis=1)


def flow_state(vel, amp, scale, rng, n=4000):
    dim = len(vel[0])
    u = amp * rng.standard_normal((n, dim))
    f = np.empty((n, len(vel)))
    for a, e in enumerate(vel):
        v = np.ones(n)
        for d in range(dim):
            s = 1.0 / 3.0 + u[:, d] ** 2
            v *= 1 - s if e[d] == 0 else 0.5 * (s + e[d] * u[:, d])
        f[:, a] = v
    if len(vel) == 15:
        w = np.array([2 / 9] + [1 / 9] * 6 + [1 / 72] * 8)
        f = w * (1 + 3 * (u @ np.array(vel, dtype=np.float64).T))
    f *= scale * (1 + 0.5 * amp * rng.uniform(-1, 1, f.shape))
    return f, scale * 1e-5 * rng.standard_normal((n, dim))


@pytest.mark.parametrize("lattice", ["d2q9", "d3q27", "d3q15"])
@pytest.mark.parametrize("amp", [0.0, 1e-5, 0.02, 0.09])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -500, 3e14])
@pytest.mark.parametrize("envelope", [(1.0, 1.0), (0.3, -0.7)])
def test_flow_collision(host, lattice, amp, scale, envelope):
    rng = np.random.default_rng(1)
    vel = {"d2q9": V9, "d3q27": V27, "d3q15": V15}[lattice]
    f, P = flow_state(vel, amp, scale, rng)
    ap, aq = envelope
    for xo in (0, 1):
        if xo:
            P[:, 1:] = 0.0
        for wb, wd, ws in ((1.0, 1.9, 1.9), (0.4, 0.7, 1.2)):
            if lattice == "d2q9":
                got, ok = call(host.fixed9, f, P, ap, aq, wb, wd, ws, xo)
            else:
                ws = wd
                got, ok = call(host.fixed27 if lattice == "d3q27" else host.fixed15, f, P, ap, aq, wb, ws, xo)
            F, Fq = ap * P.astype(np.longdouble), aq * P.astype(np.longdouble)
            ref, dbl = [d3q15(f, F, Fq, wb, ws, T) if lattice == "d3q15" else product(f, F, Fq, vel, wb, wd, ws, T)
                        for T in (np.longdouble, np.float64)]
            # every node whose results are positive and not tiny is taken
            assert ok[ref.min(axis=1) > 2.0 ** -24 * f.max(axis=1)].all() and ok.mean() > 0.95
            got, ref, dbl, f1 = got[ok], ref[ok], dbl[ok], f[ok]
            assert np.abs(got - ref).max() <= np.abs(dbl - ref).max()
            # mass: the sum of the rounded results, each half a unit of its own last place at most
            assert np.abs((got - f1).astype(np.longdouble).sum(axis=1)).max() <= len(vel) * 2.0 ** -53 * np.abs(f1).max()


@pytest.mark.parametrize("base", [1.0, 0.0])
@pytest.mark.parametrize("amp", [1e-6, 0.3])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -500, 3e14])
def test_scalar_collision(host, base, amp, scale):
    """Populations of either sign (a scalar about zero), any uniform velocity below 0.9."""
    rng = np.random.default_rng(2)
    g = scale * (base * np.array([1 / 3] + [1 / 6] * 4) + amp * rng.standard_normal((4000, 5)))
    P = scale * amp * 1e-3 * rng.standard_normal(4000)
    for ux, uy in ((0.01, 0.01), (0.0, 0.0), (-0.4, 0.2)):
        for om in ((0, 1.9, 0.6, 1.0, 1.0), (0, 0.3, 1.7, 0.5, 1.9)):
            om = np.array(om, dtype=np.float64)
            got, ok = call(host.fixed5, g, P, 0.7, 0.2, om, ux, uy)
            assert ok.mean() > 0.99  # a value 2^25 below the node's largest takes the FP64 form
            S, Sq = np.longdouble(0.7) * P, np.longdouble(0.2) * P
            ref, dbl = [d2q5(g, S, Sq, om, ux, uy, T)[ok] for T in (np.longdouble, np.float64)]
            assert np.abs(got[ok] - ref).max() <= np.abs(dbl - ref).max()


def test_states_left_to_fp64(host):
    """What the fixed-point form does not take is reported, not computed."""
    f, P = flow_state(V27, 0.01, 1.0, np.random.default_rng(3), n=16)
    f[0, 3] = np.nan
    f[1, 5] = np.inf
    f[2] *= 2.0 ** -600
    f[3] *= 2.0 ** 60
    f[4] = 0.0
    f[5, 2::3] *= 50.0   # |u_x| above 1/2
    f[6] *= -1.0
    f[7, 0] = 1e-12      # a result below 2^-25 of the largest: not reached by a relaxed state
    P[8] = 1.0           # a force as large as the populations
    _, ok = call(host.fixed27, f, P, 1.0, 1.0, 1.0, 1.9, 0)
    assert not ok[:7].any() and not ok[8] and ok[9:].all()
