"""Index arithmetic of the network's kernels (csrc/k_nn_index.cuh), compiled for the host,
against Python's integers, up to the largest shapes that the kernels are given."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_10247_gb300", "csrc")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("nn") / "index.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC,
                           os.path.join(HERE, "nn_index_host.cpp"), "-o", so])
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _taps(rng, k, count):
    return np.stack([rng.integers(0, k[d], count) for d in range(3)], axis=1).astype(np.int32)


def _source(p, dhw, k, dil, tap, sgn):
    z = [p // (dhw[1] * dhw[2]), p // dhw[2] % dhw[1], p % dhw[2]]
    z = [z[d] + sgn * dil[d] * (int(tap[d]) - (k[d] - 1) // 2) for d in range(3)]
    if any(not 0 <= z[d] < dhw[d] for d in range(3)):
        return -1
    return (z[0] * dhw[1] + z[1]) * dhw[2] + z[2]


@pytest.mark.parametrize("n,dhw,k,dil", [
    (3, (1, 20, 17), (1, 3, 3), (1, 1, 1)), (2, (4, 9, 6), (3, 3, 1), (1, 2, 1)),
    (1, (1, 30000, 30000), (1, 3, 3), (1, 1, 1)),          # 9e8 values a channel: 7 channels are above 2^32
    (1, (2, 15000, 30000), (1, 3, 3), (1, 2000, 7000)), (2, (1, 32767, 32700), (1, 3, 3), (1, 1, 1)),
    (1, (1, 46400, 46400), (1, 3, 3), (1, 3, 3)),          # 64-bit positions
    (5, (7, 100000, 9000), (3, 3, 3), (1, 50000, 4000))])
def test_gathered_values(host, n, dhw, k, dil):
    rng = np.random.default_rng(1)
    sp, count, ch = int(np.prod(dhw)), 3000, 56
    q = rng.integers(0, n * sp, count)
    q[:3], q[-3:] = np.arange(3), n * sp - 1 - np.arange(3)
    c = rng.integers(0, ch, count).astype(np.int32)
    c[-3:] = ch - 1
    tap = _taps(rng, k, count)
    v = np.array([n, ch, ch, *dhw, *k, *dil], np.int32)
    for sgn in (1, -1):
        sample, off = np.empty(count, np.int64), np.empty(count, np.int64)
        host.gather_offsets(_p(v), ctypes.c_long(count), _p(q), _p(c), _p(tap), ctypes.c_int(sgn), _p(sample), _p(off))
        for i in range(count):
            at = _source(int(q[i]) % sp, dhw, k, dil, tap[i], sgn)
            assert sample[i] == int(q[i]) // sp and off[i] == (int(c[i]) * sp + at if at >= 0 else -1)


@pytest.mark.parametrize("n,dhw,k,dil,narrow", [
    (3, (2, 20, 17), (1, 3, 3), (1, 1, 4), 1), (2, (1, 5, 9), (1, 3, 5), (1, 1, 5), 1), (2, (1, 5, 9), (1, 3, 3), (1, 1, 9), 1),
    (1, (1, 32700, 32700), (1, 3, 3), (1, 1, 32699), 1), (1, (1, 32700, 32700), (1, 3, 3), (1, 1, 32700), 1),
    (2, (1, 32700, 32700), (1, 3, 3), (1, 1, 1), 1), (2, (1, 32767, 32767), (1, 3, 3), (1, 1, 1), 0),
    (1, (1, 46400, 46400), (1, 3, 3), (1, 3, 3), 0), (5, (7, 100000, 9000), (3, 3, 3), (1, 50000, 4000), 0),
    (1, (1, 1, 2 ** 30 - 1), (1, 1, 3), (1, 1, 2 ** 29), 0), (1, (1, 1, 2 ** 30 - 1), (1, 1, 3), (1, 1, 2 ** 30 - 2), 0)])
def test_line_of_positions(host, n, dhw, k, dil, narrow):
    """Every position's place, to the last one and past it, and that position + shift is the
    shifted pixel of the same row or none."""
    rng = np.random.default_rng(2)
    w = dhw[2]
    shifts = [dil[2] * (e - (k[2] - 1) // 2) for e in range(k[2])]
    reach = max(s for s in shifts if s < w)
    wp, rows = w + reach, n * dhw[0] * dhw[1]
    total = rows * wp
    q = rng.integers(0, total, 2000)
    q[:6] = [0, w - 1, wp - 1, total - 1, total, total + reach]
    v = np.array([n, 1, 1, *dhw, *k, *dil], np.int32)

    def places(q):
        pos, t, r = np.empty((len(q), 4), np.int32), np.zeros(1, np.int64), np.zeros(1, np.int64)
        assert host.positions(_p(v), ctypes.c_long(len(q)), _p(q), _p(pos), _p(t), _p(r)) == narrow
        assert t[0] == total and r[0] == reach
        return pos

    for s in [s for s in shifts if abs(s) <= reach]:
        for p, m in zip(places(np.ascontiguousarray(q + s)), q.tolist()):
            row, col = m // wp, m % wp + s
            if m % wp >= w or row >= rows:
                continue  # the shifts of an empty position are not used
            if not 0 <= col < w:
                assert p[3] == -1
            else:
                assert tuple(p) == (row // dhw[1] // dhw[0], row // dhw[1] % dhw[0], row % dhw[1], col)
    for p, m in zip(places(q), q.tolist()):
        assert (p[3] >= 0) == (m < total and m % wp < w)
