"""The column sums' limbs (csrc/fx64.cuh), compiled for the host: 32 lanes' 96-bit sums, added
limb by limb as the warp reductions do, are each within half of 2^5 units of the exact sum,
and the rounding has no sign but for its ties, which go up: over 400 warps of 32 lanes the
mean error of a lane is within 5 standard errors (2^5 / sqrt(12 x 400 x 32) units) of the half
unit that 1 tie of 16 units in 32 numbers makes."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_0262_gb300", "csrc")

SRC = r"""
#include "fx64.cuh"
using namespace fx64;
// limbs of 32 lanes added with the width of the device's reductions
extern "C" void warp(const u32 *w, u32 *o0, u32 *o1, int *o2) {
  u32 t0 = 0, t1 = 0, t2 = 0;
  for (int i = 0; i < 32; i++) {
    u32 l0, l1; int l2;
    Acc96 a = column_start();
    add96(a, w[3 * i + 2], w[3 * i + 1], w[3 * i]);
    column_limbs(a, l0, l1, l2);
    t0 += l0; t1 += l1; t2 += (u32)l2;
  }
  *o0 = t0; *o1 = t1; *o2 = (int)t2;
}
extern "C" double total(u64 a, u64 b, int64_t c) { return limbs_total(a, b, c); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("columns")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    so.warp.argtypes = [ctypes.c_void_p] * 4
    so.total.argtypes, so.total.restype = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int64], ctypes.c_double
    return so


def _warp(lib, lanes):
    w = np.array([[v >> s & 0xFFFFFFFF for s in (0, 32, 64)] for v in lanes], np.uint32)
    o = np.zeros(3, np.uint32)
    lib.warp(w.ctypes.data, o.ctypes.data, o[1:].ctypes.data, o[2:].ctypes.data)
    a, b, c = int(o[0]), int(o[1]), int(o[2:].view(np.int32)[0])
    t = ((c << 54) + (b << 27) + a) * 32
    assert abs(lib.total(a, b, c) * 32 - t) <= abs(t) * 2.0**-52
    return t - sum(lanes)


@pytest.mark.parametrize("bits", [3, 20, 33, 60, 84])
def test_sums_are_rounded_to_nearest(lib, bits):
    g = np.random.default_rng(bits)
    rnd = lambda: int.from_bytes(g.bytes(12), "little") % (1 << bits)  # noqa: E731
    errs = []
    for k in range(400):
        lanes = [rnd() if k % 3 == 0 else -rnd() if k % 3 == 1 else rnd() - rnd() for _ in range(32)]
        errs.append(_warp(lib, lanes))
        assert abs(errs[-1]) <= 32 * 16
    if bits > 5:
        assert abs(sum(errs) - 0.5 * 400 * 32) <= 5 * 32 * np.sqrt(400 * 32 / 12)


def test_the_largest_and_the_zero_sums(lib):
    top = int(0.77 * 2**85)
    for v in (0, 1, -1, 15, 16, -16, -17, top, -top):
        assert abs(_warp(lib, [v] * 32)) <= 32 * 16
    assert _warp(lib, [0] * 32) == 0
