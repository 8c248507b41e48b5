"""The index arithmetic of the Gabor map (csrc/gabor_window.h), compiled for the host: for
any contents of the array of times and any window, the bins of a time and the pairs of a
block stay within the bins, the two halves of a block's range meet, and every bin of the
window belongs to exactly one pair."""
import ctypes as C
import itertools
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_17164_gb300", "csrc")
WRAP = """#include "gabor_window.h"
extern "C" void window(double tj, double t0, double dt, double sigma, long long n, long long* w, double* delta) {
    const sfhk::GaborWindow v = sfhk::gabor_window(tj, t0, dt, sigma, n);
    w[0] = v.lo; w[1] = v.hi; w[2] = v.c; w[3] = sfhk::gabor_reach(v.lo, v.hi, v.c);
    w[4] = sfhk::gabor_middle(w[3]); *delta = v.delta;
}
"""
INF, NAN = math.inf, math.nan
TIMES = [NAN, INF, -INF, 0.0, -0.0, 3.3, -35.0, -35.04, 34.9, 34.96, 40.0, -60.0, 500.0, -1e6, 1e6, 1e18, -1e19, 1e30,
         1e300, -1e308, 5e-324]
SIGMAS = [1e-300, 1e-9, 0.004, 0.03, 0.9, 2.85, 40.0, 1e3, 1e6, 1e18, 1e30, 1e200, 1.7e308]


@pytest.fixture(scope="module")
def window(tmp_path_factory):
    d = tmp_path_factory.mktemp("gw")
    (d / "w.cpp").write_text(WRAP)
    cxx = shutil.which("g++") or shutil.which("c++")
    assert cxx, "a C++ compiler is required"
    subprocess.run([cxx, "-O1", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", str(d / "w.so"),
                    str(d / "w.cpp")], check=True)
    fn = C.CDLL(str(d / "w.so")).window
    fn.argtypes = [C.c_double] * 4 + [C.c_longlong, C.POINTER(C.c_longlong), C.POINTER(C.c_double)]

    def call(tj, t0, dt, sigma, n):
        w, delta = (C.c_longlong * 5)(), C.c_double()
        fn(tj, t0, dt, sigma, n, w, C.byref(delta))
        return (*w, delta.value)
    return call


@pytest.mark.parametrize("n", [0, 1, 2, 700, 88257])
@pytest.mark.parametrize("t0,dt", [(-35.0, 0.1), (0.0, 1e-300), (-1e300, 1e300)])
def test_windows_stay_within_the_bins(window, n, t0, dt):
    for tj, sigma in itertools.product(TIMES, SIGMAS):
        lo, hi, c, reach, mid, delta = window(tj, t0, dt, sigma, n)
        if lo > hi:
            assert reach == -1 and mid == 0
            assert math.isnan(delta) == (math.isnan(tj) and n > 0)
            continue
        assert not math.isnan(tj) and 0 <= lo <= c <= hi < n, (tj, sigma)
        assert max(c - lo, hi - c) == reach < n and 0 <= mid <= reach + 1


@pytest.mark.parametrize("sigma", SIGMAS[:10])
def test_a_window_is_the_bins_within_nine_sigma(window, sigma):
    n, t0, dt = 700, -35.0, 0.1
    for tj in TIMES[3:14]:
        lo, hi, c, reach, mid, delta = window(tj, t0, dt, sigma, n)
        # bins next to the cut may fall on either side by the rounding of the cut's own place
        sure = [k for k in range(n) if abs(t0 + k * dt - tj) < 9 * sigma - 1e-9 * (1 + abs(tj))]
        if sure:
            assert lo <= sure[0] and hi >= sure[-1]
            assert all(abs(t0 + k * dt - tj) <= 9 * sigma + 1e-9 * (1 + abs(tj)) for k in (lo, hi))
            assert abs(delta - (t0 + c * dt - tj)) <= 1e-12 * (1 + abs(tj))
            pairs = [k for m in range(reach + 1) for k in {c - m, c + m} if lo <= k <= hi]
            assert sorted(pairs) == list(range(lo, hi + 1))
