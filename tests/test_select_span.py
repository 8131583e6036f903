"""The span arithmetic of the Gamma builder's select (csrc/bsp_span.cuh), compiled by the host compiler and driven as the kernels drive it:
whatever the keys are, the rounds end and the threshold is that of a sort."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_09453_b200", "csrc")
HARNESS = r"""
#include <algorithm>
#include <vector>
#include "bsp_span.cuh"
typedef unsigned long long u64;
// Rounds taken, or -1: a round found no bin, or the bound on the rounds came first.
extern "C" int select_by_spans(const u64 *key, int n, long long need, int width, int few, u64 *T, long long *ties, int *same)
{
    u64 lo = *std::min_element(key, key + n), hi = *std::max_element(key, key + n);
    int left = n;
    std::vector<int> hist(1u << width);
    for (int round = 0;; ++round) {
        if (lo == hi) { *T = lo; *ties = need; *same = left; return round; }
        if (round == bsp::span_rounds(width)) return -1;
        if (left <= few) {
            std::vector<u64> c;
            for (int i = 0; i < n; ++i) if (key[i] >= lo && key[i] <= hi) c.push_back(key[i]);
            if ((int)c.size() != left || need < 1 || need > left) return -1;
            std::sort(c.begin(), c.end());
            *T = c[need - 1];
            *ties = need - (std::lower_bound(c.begin(), c.end(), *T) - c.begin());
            *same = (int)(std::upper_bound(c.begin(), c.end(), *T) - std::lower_bound(c.begin(), c.end(), *T));
            return round;
        }
        const int shift = bsp::span_shift(lo, hi, width);
        if ((hi - lo) >> shift >= 1ull << width) return -1;
        std::fill(hist.begin(), hist.end(), 0);
        for (int i = 0; i < n; ++i) if (key[i] >= lo && key[i] <= hi) ++hist[(key[i] - lo) >> shift];
        long long cum = 0;
        unsigned bin = 0;
        while (bin < hist.size() && cum + hist[bin] < need) cum += hist[bin++];
        if (bin == hist.size()) return -1;
        need -= cum;
        left = hist[bin];
        bsp::span_to_bin(lo, hi, bin, shift);
    }
}
"""


@pytest.fixture(scope="module")
def select(tmp_path_factory):
    d = tmp_path_factory.mktemp("span")
    (d / "span.cpp").write_text(HARNESS)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "span.cpp"), "-o", str(d / "span.so")])
    f = C.CDLL(str(d / "span.so")).select_by_spans

    def run(keys, need, width, few=32):
        T, ties, same = C.c_uint64(0), C.c_longlong(0), C.c_int(0)
        rounds = f(keys.ctypes.data_as(C.c_void_p), len(keys), C.c_longlong(need), width, few, C.byref(T), C.byref(ties), C.byref(same))
        return rounds, T.value, ties.value, same.value
    return run


def scores(seed, n):
    return np.abs(np.random.default_rng(seed).normal(size=n)) ** 2


NEGATIVE_NAN, NAN = 0xFFF8000000000000, 0x7FF8000000000000
ODD = {
    "a negative NaN": [NEGATIVE_NAN],
    "negative NaNs": [NEGATIVE_NAN + k for k in range(40)],
    "equal negative NaNs": [NEGATIVE_NAN] * 300,
    "the last key": [2 ** 64 - 1],
    "the last keys": [2 ** 64 - 1 - k for k in range(50)],
    "NaNs of both signs": [NAN, NEGATIVE_NAN] * 30,
    "infinities and NaNs": [0x7FF0000000000000] * 40 + [NAN] * 40,
    "zeros and the sign bit": [0] * 60 + [2 ** 63] * 60,
    "both ends": [0, 2 ** 64 - 1],
}


@pytest.mark.parametrize("width", [11, 12])
@pytest.mark.parametrize("what", sorted(ODD))
def test_threshold_equals_a_sort(select, what, width):
    for seed, n in ((1, 100), (2, 700), (3, 4000)):
        odd = np.array(ODD[what], dtype=np.uint64)
        keys = np.concatenate([scores(seed, n).view(np.uint64), odd])
        np.random.default_rng(seed + 10).shuffle(keys)
        order = np.sort(keys)
        for need in sorted({1, n // 2, n, n + 1, n + (len(odd) + 1) // 2, n + len(odd)}):
            rounds, T, ties, same = select(keys, need, width)
            assert rounds >= 0, (n, need)
            assert T == int(order[need - 1])
            assert ties == need - int((keys < order[need - 1]).sum()) and same == int((keys == order[need - 1]).sum())


@pytest.mark.parametrize("width", [11, 12])
def test_keys_anywhere_in_64_bits(select, width):
    rng = np.random.default_rng(7)
    for _ in range(300):
        n = int(rng.integers(2, 600))
        keys = rng.integers(0, 2 ** 64, n, dtype=np.uint64) >> np.uint64(rng.integers(0, 64))
        if rng.integers(0, 2):
            keys = ~keys
        order = np.sort(keys)
        for need in (1, int(rng.integers(1, n + 1)), n):
            for few in (1, 32):
                rounds, T, ties, same = select(keys, need, width, few)
                assert rounds >= 0 and T == int(order[need - 1]) and same == int((keys == order[need - 1]).sum())
