"""CPU check of the host rules that split a sweep into CTAs (mfc_launch.cuh), compiled
from the header."""
import ctypes
import os
import re
import subprocess
import time

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LAUNCH = os.path.join(HERE, os.pardir, "paper_2305_09163_gb300", "csrc", "mfc_launch.cuh")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    with open(LAUNCH) as f:
        src = f.read()
    d = tmp_path_factory.mktemp("split")
    cpp, so = str(d / "split.cpp"), str(d / "split.so")
    with open(cpp, "w") as f:
        f.write(re.search(r"inline int stream_segment\(.*?\n}\n", src, re.S).group(0))
        f.write('extern "C" int segment(long long c, int n, int f) { return stream_segment(c, n, f != 0); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", cpp, "-o", so], check=True)
    return ctypes.CDLL(so)


def _segment(lib, plane, n, fp64):
    return lib.segment(ctypes.c_longlong(plane * n), n, int(fp64))


def _least(plane, n, fp64):
    """The rule without a bound on the search."""
    L = np.arange(2, n + 4, 4)
    L = L[:np.searchsorted(L, n) + 1]
    whole, rest = n // L, n % L
    walk = (L + 2) // 4 + 0.25
    chunks = whole * walk + np.where(rest > 0, (rest + 5) // 4 + 0.25, 0.0)
    t = chunks * float((plane + 31) // 32) / 152.0 + (1.0 if fp64 else 2.5) * walk
    return int(L[np.argmin(t)])


def test_segment_has_the_least_estimate(lib):
    rng = np.random.default_rng(0)
    cases = [(3, 3), (9, 5), (31, 131), (32, 127), (65536, 256), (9, 3000), (147456, 384), (262144, 512)]
    cases += [(int(np.exp(rng.uniform(1.1, 13))), int(np.exp(rng.uniform(1.1, 9)))) for _ in range(2000)]
    for plane, n in cases:
        for fp64 in (True, False):
            assert _segment(lib, plane, n, fp64) == _least(plane, n, fp64), (plane, n, fp64)


def test_segment_search_is_bounded(lib):
    # a search through every length takes ~10 ns each: 0.25 s for these 10^8 rows
    t = time.perf_counter()
    _segment(lib, 3, 100_000_000, True)
    assert time.perf_counter() - t < 0.02
