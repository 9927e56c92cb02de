"""The binary64 tanh of k_tanh64.cuh, compiled for the host, against 120-bit
values: its error is the final rounding (0.5 ulp) plus the table's and the
truncation's parts, derived in the header as below 0.2 ulp from 2^-9 on; the
series below 2^-9 rounds its factor and its product, below 1.1 ulp."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_math64_host import KDIR, _max_ulp

mpmath = pytest.importorskip("mpmath")

SHIM = r"""
#include <cmath>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __align__(n) alignas(n)
struct double2 { double x, y; };
static inline double2 __ldg(const double2* p) { return *p; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline long long __double_as_longlong(double x) { long long v; std::memcpy(&v, &x, 8); return v; }
static inline double __longlong_as_double(long long v) { double x; std::memcpy(&x, &v, 8); return x; }
#include "k_tanh64.cuh"
extern "C" void t64(long n, const double* x, double* y) {
  for (long i = 0; i < n; ++i) y[i] = dcp_tanh64(x[i]);
}
"""


@pytest.fixture(scope="module")
def t64(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("t64")
    src = d / "t64.cpp"
    src.write_text(SHIM)
    lib = d / "libt64.so"
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC",
                    "-I", KDIR, "-o", str(lib), str(src)], check=True)
    so = ctypes.CDLL(str(lib))

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        so.t64(ctypes.c_long(x.size), x.ctypes.data_as(ctypes.c_void_p),
               y.ctypes.data_as(ctypes.c_void_p))
        return y
    return run


def _edges():
    """Both sides of every interval boundary of the table."""
    lo = [2.0 ** e * (1 + k / n) for e0, e1, n in ((-9, -3, 16), (-3, 0, 64), (0, 5, 128))
          for e in range(e0, e1) for k in range(n)]
    lo = np.array([v for v in lo if v <= 20.0] + [20.0])
    return np.concatenate([lo, np.nextafter(lo, 0.0)])


@pytest.mark.parametrize("lo,hi,bound", [(2.0 ** -9, 20.0, 0.7), (1e-300, 2.0 ** -9, 1.1)])
def test_tanh64_ulp(t64, lo, hi, bound):
    rng = np.random.default_rng(5)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 6000))
    if hi > 1:
        x = np.concatenate([x, rng.uniform(0.3, 3.0, 3000), _edges()])
    x = x[(x >= lo) & (x < hi)] * np.where(rng.random(np.count_nonzero((x >= lo) & (x < hi))) < 0.5, -1, 1)
    assert _max_ulp(mpmath.tanh, x, t64(x)) <= bound


def test_tanh64_special(t64):
    y = t64(np.array([0.0, -0.0, 5e-324, -5e-324, 20.0, -700.0, np.inf, -np.inf]))
    assert y.tolist() == [0.0, 0.0, 5e-324, -5e-324, 1.0, -1.0, 1.0, -1.0]
    assert np.signbit(y[:2]).tolist() == [False, True]
    assert np.isnan(t64(np.array([np.nan]))).all()
