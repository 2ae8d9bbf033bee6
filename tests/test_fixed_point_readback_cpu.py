"""The readbacks' integer arithmetic (csrc/lbm_fixed.cuh), compiled for the host."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_10247_gb300", "csrc")
EX = np.array([a % 3 - 1 for a in range(27)], dtype=np.float64)


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fx") / "readback.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC,
                           os.path.join(HERE, "fixed_point_readback_host.cpp"), "-o", so])
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("top", [-126, -100, -87, -86, -80, -72, -71, -70, -40, 0, 60])
@pytest.mark.parametrize("kind", ["one", "few", "all", "subnormal", "spread"])
def test_sums_of_deviations(host, top, kind):
    """Largest deviations of about 2^top among exact zeros and values of any size: each
    is rounded at 2^-55 of the largest one's power of two, the sums once more."""
    rng = np.random.default_rng(5)
    n = 200
    d = 2.0 ** top * rng.uniform(-1, 1, (n, 27))
    if kind in ("one", "few"):
        d[rng.uniform(size=d.shape) < (0.97 if kind == "one" else 0.7)] = 0.0
        d[np.arange(n), rng.integers(0, 27, n)] = 2.0 ** top
    elif kind == "subnormal":
        d[:, ::2] = 2.0 ** -149 * rng.integers(-2 ** 22, 2 ** 22, d[:, ::2].shape)
    elif kind == "spread":
        d *= 2.0 ** rng.integers(-120, 1, d.shape)
    d[::3, ::4] = -0.0
    d = d.astype(np.float32)
    m0, jx, taken = np.zeros(n), np.zeros(n), np.zeros(n, np.int32)
    host.deviation_sums(ctypes.c_long(n), _p(d), _p(m0), _p(jx), _p(taken))
    d = d.astype(np.float64)
    big = np.abs(d).max(axis=1)
    assert taken[big >= 2.0 ** -71].all() and not taken[big < 2.0 ** -71].any()
    for k in np.flatnonzero(taken):
        unit = 2.0 ** (np.floor(np.log2(big[k])) - 55)
        for got, vals in ((m0[k], d[k]), (jx[k], EX * d[k])):
            off = abs(math.fsum([*vals, -got]))
            assert off <= 27 * unit + 2.0 ** -53 * abs(got)


def test_non_finite_deviations_are_left_to_fp64(host):
    d = np.full((2, 27), 1e-3, np.float32)
    d[0, 3], d[1, 7] = np.nan, np.inf
    m0, jx, taken = np.zeros(2), np.zeros(2), np.zeros(2, np.int32)
    host.deviation_sums(ctypes.c_long(2), _p(d), _p(m0), _p(jx), _p(taken))
    assert not taken.any()


def test_reciprocals_are_correctly_rounded(host):
    rng = np.random.default_rng(6)
    x = np.concatenate([1.0 + rng.uniform(size=1000000), 1.0 + 2.0 ** -52 * np.arange(1000), 2.0 - 2.0 ** -52 * np.arange(1, 1000),
                        1.0 / (1.0 - 2.0 ** -53 * np.arange(1, 100000)), 2.0 ** np.arange(-1019, 1020.0),
                        rng.uniform(1, 2, 10000) * 2.0 ** rng.integers(-1019, 1019, 10000)])
    r = np.empty_like(x)
    host.reciprocals(ctypes.c_long(len(x)), _p(x), _p(r))
    assert np.array_equal(r, 1.0 / x)
