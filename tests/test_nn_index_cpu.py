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
    (1, (2, 15000, 30000), (1, 3, 3), (1, 2000, 7000)), (2, (1, 32767, 32767), (1, 3, 3), (1, 1, 1))])
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
