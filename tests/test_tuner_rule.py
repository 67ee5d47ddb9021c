"""The rule by which the GEMM tuner picks a launch shape from timings (csrc/tuner_rule.h): noise of
a few per cent does not decide between shapes that take the same time, because the shape
also decides the order of the sums."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1774_gb300", "csrc")


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text('#include "tuner_rule.h"\n'
                                'extern "C" int pick(const float* t, int n) { return (int)tvcs::tuned_shape(t, n); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "rule.so"),
                           str(d / "rule.cpp")])
    lib = ctypes.CDLL(str(d / "rule.so"))

    def f(t):
        t = np.ascontiguousarray(t, np.float32)
        return lib.pick(t.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), len(t))
    return f


def test_the_pick_is_the_same_under_noise(pick):
    # us per launch at n = 128, m = 4915: single blocks on 152, 133, 114, 76 SMs, then pairs
    six = [72.3, 77.1, 83.3, 111.6, 63.4, 63.9, 70.8, 96.2]
    many = [96.7, 103.5, 113.6, 154.9, 81.9, 87.6, 96.0, 130.6]
    rng = np.random.default_rng(3)
    for t in (six, many):
        for _ in range(500):   # (2 % either way: what the medians of five launches showed)
            assert pick(np.array(t) * rng.uniform(0.98, 1.02, len(t))) == 4


def test_the_pick_is_within_the_margin_of_the_fastest(pick):
    rng = np.random.default_rng(4)
    for _ in range(500):
        t = np.float32(20.0) * np.exp(rng.normal(0, 0.1, 8)).astype(np.float32)
        assert t[pick(t)] <= 1.0527 * t.min()   # 1 / 0.95
    assert pick([20.0]) == 0 and pick([20.0, 19.1]) == 0 and pick([20.0, 18.9]) == 1


def test_small_products_are_timed_in_groups(tmp_path):
    # us per launch at n = 128, m = 1638, one image (both products) and n = 64, m = 200, 40 images: medians of
    # groups of four launches differ by 1 % either way, of single launches by 5 % at this length
    (tmp_path / "launches.cpp").write_text('#include "tuner_rule.h"\n'
                                           'extern "C" int launches(long long r, long long c) { return tvcs::tuner_launches(r, c); }\n'
                                           'extern "C" int pick(const float* t, int n) { return (int)tvcs::tuned_shape(t, n); }\n')
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(tmp_path / "launches.so"),
                           str(tmp_path / "launches.cpp")])
    lib = ctypes.CDLL(str(tmp_path / "launches.so"))
    lib.launches.argtypes = [ctypes.c_longlong] * 2
    rng = np.random.default_rng(5)
    for rows, cols, t in ((1638, 16384, [31.7, 33.5, 36.8, 44.3, 30.9, 31.6, 34.0, 41.2]),
                          (16384, 1638, [28.9, 30.9, 33.0, 42.8, 26.9, 28.9, 31.0, 39.1]),
                          (200, 4096, [28.9, 28.9, 28.3, 20.8, 29.6, 29.4, 28.9, 22.8])):
        noise = 0.01 if lib.launches(rows, cols) >= 4 else 0.05
        picks = set()
        for _ in range(500):
            v = np.ascontiguousarray(np.array(t) * rng.uniform(1 - noise, 1 + noise, len(t)), np.float32)
            picks.add(lib.pick(v.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), len(t)))
        assert len(picks) == 1
    # long launches one by one, whatever the number of rows
    assert lib.launches(4915, 16384) == 1 and lib.launches(1 << 24, 65536) == 1
