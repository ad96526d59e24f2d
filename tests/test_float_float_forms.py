"""The float-float operations of the FP64 sweeps (csrc/mfc_df.cuh), compiled for
the host (df_host.cpp), against exact rational arithmetic.

Bounds, with u = 2^-24 and operands |lo| <= k u |hi| (k = 1: normalised), all to
first order in u^2: a rounded FP32 term costs u of itself, a neglected product
lo lo costs k^2 u^2, and the approximate reciprocal (off by up to 4 u, and by k u
from the operand's hi part alone) scales a correction of (2 k + 1) u."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
U = Fraction(1, 1 << 24)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("df_host") / "df_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I", "/usr/local/cuda/include", os.path.join(HERE, "df_host.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _n(a):
    return ctypes.c_longlong(len(a))


def _exact(d):
    return [Fraction(float(h)) + Fraction(float(l)) for h, l in d]


def _pairs(rng, n, k, positive=False):
    hi = np.exp2(rng.uniform(-20, 20, n)) * (1 if positive else rng.choice([-1, 1], n))
    hi = hi.astype(np.float32)
    lo = (hi * k * 2.0 ** -24 * rng.uniform(-1, 1, n)).astype(np.float32)
    return np.ascontiguousarray(np.stack([hi, lo], 1))


def _neighbours(rng, n, gap):
    """Pairs of doubles whose difference is about gap of them."""
    x = np.exp2(rng.uniform(-60, 60, n)) * rng.choice([-1, 1], n)
    return x, x * (1 + gap * rng.uniform(-1, 1, n))


def test_three_parts_hold_the_value(lib):
    rng = np.random.default_rng(0)
    x = np.concatenate([np.exp2(rng.uniform(-73, 100, 20000)) * rng.choice([-1, 1], 20000),
                        [0.0, 1.0, -1.0, 1 - 2.0 ** -53, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 1 + 2.0 ** -24, 1 + 2.0 ** -25]])
    t = np.empty((len(x), 3), np.float32)
    lib.df_host_tf(_n(x), _p(x), _p(t))
    assert np.array_equal(t.astype(np.float64).sum(1), x)
    d = np.empty((len(x), 2), np.float32)
    lib.df_host_split(_n(x), _p(x), 1, _p(d))
    assert np.array_equal(d[:, 0], t[:, 0]) and np.array_equal(d[:, 1], t[:, 1] + t[:, 2])


@pytest.mark.parametrize("gap", [2.0 ** -6, 1e-3, 1e-6, 1e-8, 1e-11, 1e-15])
def test_difference_of_near_values_is_exact(lib, gap):
    x, y = _neighbours(np.random.default_rng(1), 20000, gap)
    d = np.empty((len(x), 2), np.float32)
    lib.df_host_tf_diff(_n(x), _p(x), _p(y), _p(d))
    assert _exact(d) == [Fraction(a) - Fraction(b) for a, b in zip(x, y)]


@pytest.mark.parametrize("gap", [0.1, 1.0, 3.0, 1e3, 1e9])
def test_difference_of_far_values(lib, gap):
    # rounded terms: the mid parts' difference (2^-25 of the larger value, which is at
    # most 2 + 1/gap differences), the last two sums (u of the result's lo part each)
    # and the result itself
    x, y = _neighbours(np.random.default_rng(2), 20000, gap)
    d = np.empty((len(x), 2), np.float32)
    lib.df_host_tf_diff(_n(x), _p(x), _p(y), _p(d))
    for got, a, b in zip(_exact(d), x, y):
        want = Fraction(a) - Fraction(b)
        assert abs(got - want) <= U * U * (4 * abs(want) + max(abs(Fraction(a)), abs(Fraction(b))) / 2)


@pytest.mark.parametrize("nearest,bound", [(0, Fraction(1, 1 << 47)), (1, Fraction(1, 1 << 49))])
def test_splits(lib, nearest, bound):
    rng = np.random.default_rng(3)
    x = np.exp2(rng.uniform(-70, 100, 20000)) * rng.choice([-1, 1], 20000)
    d = np.empty((len(x), 2), np.float32)
    lib.df_host_split(_n(x), _p(x), nearest, _p(d))
    assert all(abs(g - Fraction(v)) <= bound * abs(Fraction(v)) for g, v in zip(_exact(d), x))


def _call(lib, name, a, b):
    r = np.empty_like(a)
    assert lib.df_host_op(name.encode(), _n(a), _p(a), _p(b), _p(r)) == 0
    return _exact(r)


@pytest.mark.parametrize("k", [1, 4])
def test_products_and_sums(lib, k):
    rng = np.random.default_rng(4)
    a, b = _pairs(rng, 8000, k), _pairs(rng, 8000, k)
    X, Y = _exact(a), _exact(b)
    UU = U * U
    for g, x, y in zip(_call(lib, "prod", a, b), X, Y):
        assert abs(g - x * y) <= UU * (k * k + (k + 1) + (2 * k + 1) + 1) * abs(x * y)
    for g, x in zip(_call(lib, "square", a, b), X):
        assert abs(g - x * x) <= UU * (k * k + (2 * k + 1) + 1) * x * x
    for g, x, y in zip(_call(lib, "scale", a, b), X, b):
        f = Fraction(float(y[0]))
        assert abs(g - x * f) <= UU * (k + 2) * abs(x * f)
    for g, x, y in zip(_call(lib, "sum", a, b), X, Y):
        assert abs(g - x - y) <= UU * (2 * k + 2) * (abs(x) + abs(y))
    for g, x in zip(_call(lib, "norm", a, b), X):
        assert abs(g - x) == 0 or k > 1 and abs(g - x) <= UU * k * abs(x)


@pytest.mark.parametrize("k", [1, 4])
def test_quotients_and_roots(lib, k):
    rng = np.random.default_rng(5)
    a, b = _pairs(rng, 8000, k), _pairs(rng, 8000, k)
    X, Y = _exact(a), _exact(b)
    # residual 1, a.lo - q b.lo 2 k, their sum 2 k + 1, the correction's factor 5 + k
    bound = U * U * (1 + 2 * k + (2 * k + 1) * (1 + 5 + k) + 1)
    for g, x, y in zip(_call(lib, "quot", a, b), X, Y):
        assert abs(g * y - x) <= bound * abs(x)
    for g, x, y in zip(_call(lib, "quot_f", a, b), a, Y):
        x = Fraction(float(x[0]))
        assert abs(g * y - x) <= bound * abs(x)
    # (s (1 + d))^2 = x with |d| = (1 + k/2) u corrected to first order
    a = _pairs(rng, 8000, k, positive=True)
    bound = U * U * ((2 + k) + (2 + k) * 6 + (2 + k) ** 2 / Fraction(2) + 1)
    for g, x in zip(_call(lib, "root", a, b), _exact(a)):
        assert abs(g * g - x) <= bound * x
