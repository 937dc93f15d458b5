"""The loss gradient's difference, phi_out - target - mean, against exact arithmetic (CPU only).

The device code forms it from FP32 sums; it has to be as near as the FP64 difference rounded once,
also where the terms cancel. The header is compiled for the host and compared with fractions.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "lbnop_diff.cuh"
extern "C" void diffs(const float* a, const float* b, const double* m, long n, float* out) {
  for (long k = 0; k < n; ++k) {
    float r[4];
    lbnop_diff::diff4({a[k], a[k], 0.0f, 0.0f}, {b[k], b[k], 0.0f, 0.0f}, lbnop_diff::split(m[k]), r);
    out[k] = r[0];
  }
}
"""


@pytest.fixture(scope="module")
def diffs(tmp_path_factory):
    d = tmp_path_factory.mktemp("diff")
    (d / "diff.cpp").write_text(SRC)
    lib = str(d / "libdiff.so")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2501_03759_gb300", "csrc"), str(d / "diff.cpp"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).diffs

    def call(a, b, m):
        a, b, m = (np.ascontiguousarray(v, t) for v, t in ((a, np.float32), (b, np.float32), (m, np.float64)))
        out = np.empty(a.size, np.float32)
        fn(*(v.ctypes.data_as(ctypes.c_void_p) for v in (a, b, m)), ctypes.c_long(a.size), out.ctypes.data_as(ctypes.c_void_p))
        return a, b, m, out

    return call


def samples(kind, n, rng):
    a = rng.uniform(-1.1, 1.1, n).astype(np.float32)
    if kind == "fields":  # a target a little away, a mean far below the differences
        return a, (a + 0.01 * rng.standard_normal(n)).astype(np.float32), rng.uniform(-1e-5, 1e-5, n)
    if kind == "scales":  # terms of very different sizes
        return (a * 2.0 ** rng.integers(-30, 30, n), rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-30, 30, n),
                rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-30, 30, n))
    b = (rng.uniform(-1.1, 1.1, n) * 2.0 ** rng.integers(-20, 1, n)).astype(np.float32)
    d = a.astype(np.float64) - b.astype(np.float64)
    # the mean cancels the difference down to a few of the last bits of FP64, or to some bits more
    return a, b, d + np.spacing(d) * rng.integers(-3, 4, n) * 2.0 ** rng.integers(0, 34, n)


@pytest.mark.parametrize("kind", ["fields", "scales", "cancelling"])
def test_difference_is_as_near_as_fp64(diffs, kind):
    a, b, m, got = diffs(*samples(kind, 6000, np.random.default_rng(11)))
    f64 = (a.astype(np.float64) - b.astype(np.float64) - m).astype(np.float32)
    for x, y, z, g, r in zip(a, b, m, got, f64):
        exact = Fraction(float(x)) - Fraction(float(y)) - Fraction(float(z))
        # half an ulp of the result, and the tail: three roundings 2^-23 below what one rounding drops
        bound = abs(exact) * Fraction(1, 2 ** 24) * (1 + Fraction(1, 2 ** 18)) + Fraction(1, 2 ** 149)
        assert abs(Fraction(float(g)) - exact) <= bound, (x, y, z)
        assert abs(Fraction(float(g)) - exact) <= abs(Fraction(float(r)) - exact) + abs(exact) / 2 ** 42, (x, y, z)


def test_difference_beyond_fp32(diffs):
    big, inf, nan = 3e38, np.inf, np.nan
    a = [big, big, inf, -inf, inf, nan, 1.0, 1.0, big]
    b = [-big, -big, 1.0, 1.0, inf, 1.0, nan, 1.0, 0.0]
    m = [0.0, 5e38, 0.0, 0.0, 0.0, 0.0, 0.0, np.inf, 1e300]
    a, b, m, got = diffs(a, b, m)
    with np.errstate(all="ignore"):
        want = (a.astype(np.float64) - b.astype(np.float64) - m).astype(np.float32)
    assert np.array_equal(got, want, equal_nan=True)
