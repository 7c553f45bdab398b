"""The stop test's comparison (r12_below: by the words of the doubles outside
a band around tol) against the formula sqrt(num) / sqrt(den) < tol, on the
host: ratios from far below to far above tol and within rounding of it, zero,
denormal, infinite and NaN sums, and tolerances of either sign."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2202_13449_gb300", "csrc")
SRC = r"""
#include "rtlbfs_dev.cuh"
extern "C" void below(const double* num, const double* den, const double* tol, int n, int* out)
{
    for (int i = 0; i < n; ++i) out[i] = rtlbfs::r12_below(num[i], den[i], tol[i]);
}
"""


@pytest.fixture(scope="module")
def below(tmp_path_factory):
    d = tmp_path_factory.mktemp("stop")
    (d / "t.cu").write_text(SRC)
    so = d / "libstop.so"
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-O1", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-diag-suppress", "20011,20014", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, str(d / "t.cu"), "-o", str(so)],
                   check=True)
    f = C.CDLL(str(so)).below

    def call(num, den, tol):
        a = [np.ascontiguousarray(x, dtype=np.float64) for x in np.broadcast_arrays(num, den, tol)]
        out = np.zeros(a[0].size, dtype=np.int32)
        f(*[x.ctypes.data_as(C.POINTER(C.c_double)) for x in a], C.c_int(out.size),
          out.ctypes.data_as(C.POINTER(C.c_int)))
        return out.astype(bool)

    return call


def formula(num, den, tol):
    with np.errstate(all="ignore"):
        r = np.where(den > 0, np.sqrt(num) / np.sqrt(den), np.inf)
        return (r < tol) & (den > 0) & (tol > 0)


def test_random_ratios(below):
    g = np.random.default_rng(1)
    n = 200000
    den = 10.0 ** g.uniform(-40, 12, n)
    tol = 10.0 ** g.uniform(-14, 1, n)
    # log2 of num / (tol^2 den): wide, near the band's edges, and near 0
    k = np.concatenate([g.uniform(-60, 60, n // 2), g.uniform(-0.4, 0.4, n // 4),
                        g.uniform(-1e-12, 1e-12, n - n // 2 - n // 4)])
    num = tol * tol * den * 2.0 ** k
    np.testing.assert_array_equal(below(num, den, tol), formula(num, den, tol))


def test_special_values(below):
    v = np.array([0.0, 5e-324, 1e-310, 1e-300, 1e-20, 1.0, 1e300, np.inf, np.nan])
    num, den, tol = (a.ravel() for a in np.meshgrid(v, v, np.concatenate([v, [-1.0, -0.0, -np.inf]])))
    np.testing.assert_array_equal(below(num, den, tol), formula(num, den, tol))
