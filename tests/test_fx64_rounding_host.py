"""Terms shifted to the unit of their sum and rounded to nearest (csrc/fx64.cuh), compiled for
the host: a term and its carry add +-round(w 2^-k), ties up in magnitude, for both signs and
every shift; a term that vanishes adds exactly zero."""
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
extern "C" void term(const u32 *w, int k, int neg, int small, u32 *acc) {
  u32 w2 = w[2], w1 = w[1], w0 = w[0];
  Acc96 a{acc[0], acc[1], acc[2]};
  const u32 c = small ? signed_shift96<true>(w2, w1, w0, k, neg ? ~0u : 0u) : signed_shift96<false>(w2, w1, w0, k, neg ? ~0u : 0u);
  add96_carry(a, w2, w1, w0, c);
  acc[0] = a.w0; acc[1] = a.w1; acc[2] = a.w2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("rounding")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    so.term.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    return so


@pytest.mark.parametrize("small", [1, 0])
def test_rounded_terms(lib, small):
    g = np.random.default_rng(3)
    words = lambda v: np.array([v >> s & 0xFFFFFFFF for s in (0, 32, 64)], np.uint32)  # noqa: E731
    for k in list(range(1, 32)) + ([] if small else [32, 33, 63, 64, 65, 92, 95, 96, 97, 300]):
        for n in range(60):
            w = int.from_bytes(g.bytes(12), "little") >> int(g.integers(4, 96))
            if n % 5 == 0:
                w = (2 * (w >> k) + 1) << max(0, k - 1)  # a tie
            w &= (1 << 92) - 1
            start = int.from_bytes(g.bytes(12), "little")
            for neg in (0, 1):
                acc, ww = words(start), words(w)
                lib.term(ww.ctypes.data, k, neg, small, acc.ctypes.data)
                got = sum(int(x) << s for x, s in zip(acc, (0, 32, 64)))
                r = (w + (1 << (k - 1))) >> k
                assert got == (start + (-r if neg else r)) % (1 << 96)
