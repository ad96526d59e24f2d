"""The six-equation model's volume-fraction edges next to a trace phase: the edge is
the cell value plus a float-float increment rounded to FP64, the differences are a few
units in the last place of 1, and an increment of exactly half a unit must round as the
exact one does.  The increments' functions are taken from mfc_weno.cuh and compiled for
the host (df_host.cpp).

Exact increments: the indicators (~1e-32) vanish against eps, so the weights are
the ideal ones: (-2 D0 + 11 D1 + 24 D2 - 3 D3)/60 for WENO5, (A + 2 B)/6 for WENO3 at the
right edge, the mirrored stencil at the left.  Halves are the only ties, and off them
the nearest rounding boundary is 1/60 of a unit away, far beyond the arithmetic's error."""
import ctypes
import os
import re
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
WENO = os.path.join(HERE, os.pardir, "paper_2305_09163_gb300", "csrc", "mfc_weno.cuh")
ENTRY = """
extern "C" void edges(int order, long long n, const double* D, double eps, double vc, double* out) {
    const df e = df_from_double(eps);
    for (long long i = 0; i < n; ++i) {
        df d[4];
        for (int k = 0; k < 4; ++k) d[k] = df_from_double(D[4 * i + k]);
        const df2 I = order == 5 ? weno5_increments_pair<true>(d, e) : weno3_increments_pair<true>(d[1], d[2], e);
        out[2 * i] = vc + df_to_double(df2_x(I));
        out[2 * i + 1] = vc + df_to_double(df2_y(I));
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    with open(WENO) as f:
        src = f.read()
    fns = [re.search(r"template <[^>]*>\n[^\n]* %s\(.*?\n}\n" % name, src, re.S).group(0)
           for name in ("weno5_increments_pair", "weno3_increments_pair")]
    d = tmp_path_factory.mktemp("edges")
    cpp, so = str(d / "edges.cpp"), str(d / "edges.so")
    with open(cpp, "w") as f:
        f.write('#include "%s"\n' % os.path.join(HERE, "df_host.cpp") + "\n".join(fns) + ENTRY)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I", "/usr/local/cuda/include", cpp, "-o", so], check=True)
    return ctypes.CDLL(so)


def _right(order, d):
    return Fraction(-2 * d[0] + 11 * d[1] + 24 * d[2] - 3 * d[3], 60) if order == 5 else Fraction(d[1] + 2 * d[2], 6)


@pytest.mark.parametrize("order,eps", [(5, 0.75e-6), (3, 1e-6)])
@pytest.mark.parametrize("vc", [1 - 1e-6, 1 - 3e-9, 0.75])
def test_half_units_round_as_the_exact_increment(lib, order, eps, vc):
    unit = 2.0 ** -53   # of [1/2, 1)
    K = np.random.default_rng(order).integers(-6, 7, (20000, 4))
    D = np.ascontiguousarray(K * unit)
    out = np.empty((len(K), 2))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.edges(order, ctypes.c_longlong(len(K)), p(D), ctypes.c_double(eps), ctypes.c_double(vc), p(out))
    base, ties = int(vc / unit), 0
    for k, got in zip(K.tolist(), out):
        for inc, g in zip((_right(order, k), _right(order, [-x for x in reversed(k)])), got):
            ties += inc.denominator == 2
            assert int(g / unit) == round(base + inc)   # round(): ties to even
    assert ties > 300
