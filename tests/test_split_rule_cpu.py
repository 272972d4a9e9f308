"""How many CTAs share a tile's candidates in the backward (csrc/split.h, plain
C++): the rule itself, compiled for the host."""
import ctypes
import os
import subprocess

import pytest

from paper_2405_20067_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "split.h"
static ndg::SplitCost cost(int N, int tc) {
  return !tc ? ndg::split_fp32(N) : N <= 6 ? ndg::kSplitPsi : ndg::kSplitBeta;
}
extern "C" int launch(int N, int tc, long long T, long long E_cap, int sms) {
  return ndg::launch_parts(T, E_cap, sms, cost(N, tc), tc);
}
extern "C" int tile(int N, int tc, unsigned T, unsigned steps, unsigned most, unsigned sms) {
  return ndg::split_parts(T, steps, most, sms, cost(N, tc), false);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "split.cpp").write_text(SRC)
    so = str(d / "split.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2405_20067_gb300", "csrc"), str(d / "split.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.launch.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    return L


# (N, tensor cores, tiles, candidates a tile) -> parts that measured best or equal to it
MEASURED = [
    (6, 1, 256, 600, {1}), (6, 1, 400, 300, {1}), (6, 1, 1400, 300, {1}), (8, 1, 256, 300, {1}), (10, 1, 1400, 300, {1}),
    (6, 1, 40, 4000, {3}), (10, 1, 64, 4000, {2}), (8, 1, 8, 4000, {8}),
    (3, 0, 304, 64, {1}), (3, 0, 300, 300, {1, 2}), (6, 0, 100, 64, {1}), (8, 0, 152, 64, {1}), (3, 0, 400, 4000, {3, 4, 6, 8}),
    (6, 0, 1024, 6000, {4}), (12, 0, 152, 64, {1}), (12, 0, 152, 4000, {1}), (12, 0, 64, 1200, {2}), (11, 0, 152, 1200, {1}),
]


@pytest.mark.parametrize("N,tc,T,n,best", MEASURED)
def test_measured_sizes(rule, N, tc, T, n, best):
    step = 128 if tc else 256
    S = rule.launch(N, tc, T, T * n, 152)
    if tc:  # on the tensor cores the tile's own list decides, also under a large capacity
        assert rule.tile(N, tc, T, -(-n // step), S, 152) in best
        S = rule.tile(N, tc, T, -(-n // step), rule.launch(N, tc, T, 5 * T * n, 152), 152)
    assert S in best


def test_lists_of_one_step_and_large_launches_stay_whole(rule):
    for N in (1, 6, 12):
        for tc in (0, 1):
            step = 128 if tc else 256
            for T in (1, 16, 152, 153, 5000):
                assert rule.launch(N, tc, T, T * step, 152) == 1
                assert rule.tile(N, tc, T, 1, 8, 152) == 1
            assert rule.launch(N, tc, (1 << 20) + 1, 1 << 30, 152) == 1
            assert rule.launch(N, tc, 10, 0, 152) == 1


def test_parts_never_cost_more_than_one_and_fit_the_launch(rule):
    r = synth.rng(5)
    for _ in range(3000):
        N, tc, sms = int(r.integers(1, 13)), int(r.integers(0, 2)), int(r.choice([1, 132, 152]))
        T, steps, most = int(2 ** r.uniform(0, 20)), int(2 ** r.uniform(0, 14)), int(r.integers(1, 9))
        S = rule.tile(N, tc, T, steps, most, sms)
        assert 1 <= S <= min(most, steps)
        setup, lone = (3.0 if N <= 6 else 1.25, 1.0) if tc else (0.1, 1.3 if N <= 10 else 1.0 if N == 11 else 0.7)


        def cost(s):
            waves = -(-T * s // sms)
            part = steps / s if waves >= 8 and not tc else -(-steps // s)
            return waves * (setup + part) * (lone if waves == 1 else 1.0)

        assert cost(S) <= min(cost(s) for s in range(1, min(most, steps) + 1)) * (1 + 1e-12)
