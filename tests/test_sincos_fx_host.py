"""The FP64 HMF stages' fixed-point sine and cosine (csrc/sincos_fx.cuh), compiled for the host
and checked against long-double libm: within 2^-57 (its omitted term r^5/5! is 2^-58.4 at
most, the rest below 2^-60, long-double libm 2^-63) for angles over the table's range, at
the table points, half way between them and next to those; the conversion of the integer
force to a double rounded to nearest."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_0262_gb300", "csrc")

SRC = r"""
#include "sincos_fx.cuh"
using namespace scfx;
static Entry tab[4096];
extern "C" {
void init() {
  const long double pi = 3.141592653589793238462643383279502884L;
  for (int k = 0; k < 4096; k++) {
    const long double x = (long double)k * pi / 2048.0L;
    const Limbs s = split(llrintl(sinl(x) * 0x1p62L)), c = split(llrintl(cosl(x) * 0x1p62L));
    tab[k] = Entry{s.h, s.l, c.h, c.l};
  }
}
// the largest error of n angles in units of 2^-62; -1 where an angle was refused
double worst(const double *th, long n) {
  long double w = 0;
  for (long i = 0; i < n; i++) {
    i64 s, c;
    if (!sincos_fx(th[i], tab, s, c)) return -1;
    w = fmaxl(w, fmaxl(fabsl((long double)s - sinl(th[i]) * 0x1p62L), fabsl((long double)c - cosl(th[i]) * 0x1p62L)));
  }
  return (double)w;
}
int refused(double th) { i64 s, c; return !sincos_fx(th, tab, s, c); }
double conv(i64 v) { return to_double60(v); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    d = tmp_path_factory.mktemp("sc")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-I", inc, "-o",
                    str(d / "t.so"), str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    so.worst.restype = so.conv.restype = ctypes.c_double
    so.worst.argtypes = [ctypes.c_void_p, ctypes.c_long]
    so.refused.argtypes = [ctypes.c_double]
    so.conv.argtypes = [ctypes.c_int64]
    so.init()
    return so


def _worst(lib, th):
    th = np.ascontiguousarray(th, dtype=np.float64)
    w = lib.worst(th.ctypes.data, th.size)
    assert w >= 0
    return w


@pytest.mark.parametrize("span", [1e-9, 1e-3, 1.0, 7.0, 1e3, 1e6, 2.0**20 * 0.9999999])
def test_within_2_to_minus_57(lib, span):
    g = np.random.default_rng(1)
    assert _worst(lib, (2 * g.random(200_000) - 1) * span) < 2.0**5


def test_at_and_between_the_table_points(lib):
    k = np.concatenate([np.arange(-6000, 6000), 667_000_000 + np.arange(-3000, 3000), -667_000_000 + np.arange(-3000, 3000)])
    for off in (0.0, 0.5):
        th = (k + off) * (np.pi / 2048)
        for x in (th, np.nextafter(th, 1e30), np.nextafter(th, -1e30)):
            assert _worst(lib, x) < 2.0**5


def test_small_angles_and_the_ends_of_the_range(lib):
    e = 2.0 ** np.arange(-1074, 20)
    assert _worst(lib, np.concatenate([e, -e, [0.0, -0.0], np.nextafter(e[1:], 0)])) < 2.0**5
    for th in (2.0**20, -(2.0**20), 1e300, np.inf, -np.inf, np.nan):
        assert lib.refused(th)


def test_conversion(lib):
    g = np.random.default_rng(2)
    v = (g.standard_normal(20_000) * np.exp2(g.uniform(0, 59, 20_000))).astype(np.int64)
    v = np.concatenate([v, [0, 1, -1, 2**32, -(2**32), 2**32 - 1, 2**60, -(2**60), 2**61]])
    for x in v:
        exact = int(x)
        got = lib.conv(int(x)) * 2.0**60
        assert abs(got - exact) <= abs(exact) * 2.0**-53
    assert lib.conv(0) == 0.0
