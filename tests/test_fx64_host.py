"""The integer reciprocals and products of the FP64 pair kernels (csrc/fx64.cuh), compiled
for the host and checked against exact rational arithmetic.

Each result is at least as exact as a correctly rounded double (2^-53): the squared
distance within 2^-55, a product with its reciprocal within 2^-54 (the squared distance's
error and the reciprocal's 2^-58), for any seed of the reciprocal within 2^-22 of the true
value, as the device's approximate reciprocal is."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_0262_gb300", "csrc")

SRC = r"""
#include "fx64.cuh"
using namespace fx64;
template <int D> static void quotient(const double *x, double eps, float bias, u32 *out) {
  u32 yh[D], yl[D]; int ex[D], es; u32 Mh, Ml;
  for (int d = 0; d < D; d++) { ex[d] = (int)((hi_word(x[d]) >> 20) & 0x7ffu); mantissa62(hi_word(x[d]), lo_word(x[d]), yh[d], yl[d]); }
  square_sum<D>(yh, yl, ex, soft_of(eps), Mh, Ml, es);
  const u64 R = rcp_mantissa(Mh, Ml, bias);
  out[0] = Mh; out[1] = Ml; out[2] = (u32)es;
  mul_mantissa(yh[0], yl[0], R, out[3], out[4], out[5]);
}
extern "C" {
void quotient2(const double *x, double eps, float bias, u32 *out) { quotient<2>(x, eps, bias, out); }
void quotient3(const double *x, double eps, float bias, u32 *out) { quotient<3>(x, eps, bias, out); }
void ring_term(double si, double ci, double sj, double cj, double he, float bias, i64 *S, u32 *out) {
  const i64 s = dot2(limbs_of(si), limbs_of(ci), limbs_of(cj), limbs_of(-sj));
  u32 Mh, Ml; int z;
  square_plus(s, fix92_of(he), Mh, Ml, z);
  const u64 W = rsqrt3_mantissa(Mh, Ml, bias), V = rsqrt_mantissa(Mh, Ml, bias);
  *S = s; out[0] = Mh; out[1] = Ml; out[2] = (u32)z;
  mul_fixed(s, W, out[3], out[4], out[5], out[6]);
  out[7] = (u32)(W >> 32); out[8] = (u32)W; out[9] = (u32)(V >> 32); out[10] = (u32)V;
}
u64 product(u64 a, u64 b, int *e) { return mul_renorm63(a, b, *e); }
double total(const u32 *w, int n, int lsb) { Acc96 a{0, 0, 0}; for (int i = 0; i < n; i++) add96(a, w[3 * i], w[3 * i + 1], w[3 * i + 2]); return total96(a, lsb); }
void shift(u32 *w, int k) { shift96_any(w[0], w[1], w[2], k); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx64")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    for f in (so.quotient2, so.quotient3):
        f.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_float, ctypes.c_void_p]
    so.total.restype = ctypes.c_double
    so.total.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    so.ring_term.argtypes = [ctypes.c_double] * 5 + [ctypes.c_float, ctypes.c_void_p, ctypes.c_void_p]
    so.product.restype = ctypes.c_uint64
    so.product.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_void_p]
    return so


def _pow2(e):
    return Fraction(2) ** e


@pytest.mark.parametrize("dim", [2, 3])
def test_quotients_are_exact_to_better_than_a_double(lib, dim):
    g = np.random.default_rng(5)
    fn = lib.quotient2 if dim == 2 else lib.quotient3
    out = np.zeros(6, np.uint32)
    for i in range(4000):
        eps = float(np.ldexp(1 + g.random(), -int(g.integers(0, 28))))
        x = np.ldexp(2 * g.random(dim) - 1, g.integers(-30, 10, dim))
        if i % 7 == 0:
            x[g.integers(dim)] = 0.0
        if i % 11 == 0:
            x[:] = np.ldexp(1.0, int(g.integers(-8, 8)))  # equal powers of two
        bias = np.float32(1 + (2 * g.random() - 1) * 2.0**-22)
        fn(x.ctypes.data, eps, bias, out.ctypes.data)
        Mh, Ml, es, w2, w1, w0 = (int(v) for v in out)
        s = Fraction(eps) + sum(Fraction(float(v)) ** 2 for v in x)
        assert Mh >> 31 == 1
        m = Fraction((Mh << 32) | Ml) * _pow2(-63 + es - 1023)
        assert abs(m / s - 1) < _pow2(-55)
        if x[0] != 0.0:
            ex = (int(x[:1].view(np.uint64)[0]) >> 52) & 0x7FF
            t = Fraction((w2 << 64) | (w1 << 32) | w0) * _pow2(-91 + ex - es)
            assert w2 < 1 << 28 and abs(t * s / abs(Fraction(float(x[0]))) - 1) < _pow2(-54)


def test_ring_terms(lib):
    """S and sin(d/2) within 2^-59, sin^2 + eps/2 within the rounding of its argument (one
    unit of 2^-60) and 2^-60, the powers -1/2 and -3/2 within 2^-56."""
    g = np.random.default_rng(7)
    S = ctypes.c_int64()
    out = np.zeros(11, np.uint32)
    for i in range(4000):
        he = float(np.ldexp(1 + g.random(), -int(g.integers(0, 18))))
        a = (2 * g.random() - 1) * np.pi
        b = a if i % 50 == 0 else a + (2 * g.random() - 1) * 2.0 ** -int(g.integers(0, 24))
        v = [float(x) for x in (np.sin(a), np.cos(a), np.sin(b), np.cos(b))]
        bias = np.float32(1 + (2 * g.random() - 1) * 2.0**-22)
        lib.ring_term(*v, he, bias, ctypes.byref(S), out.ctypes.data)
        Mh, Ml, z, sg, w2, w1, w0, Wh, Wl, Vh, Vl = (int(x) for x in out)
        f = [Fraction(x) for x in v]
        s = Fraction(S.value) * _pow2(-60)
        assert abs(s - (f[0] * f[3] - f[1] * f[2])) < _pow2(-59)
        if a == b:
            assert S.value == 0
        d = s * s + Fraction(he)
        ms = Fraction((Mh << 32) | Ml) * _pow2(-63)
        assert z % 2 == 1 and Fraction(1, 4) <= ms < 1
        assert abs(ms * _pow2(3 - z) - d) < 2 * abs(s) * _pow2(-60) + _pow2(-60) * d
        W, V = Fraction((Wh << 32) | Wl) * _pow2(-58), Fraction((Vh << 32) | Vl) * _pow2(-60)
        assert abs(W * W * ms**3 - 1) < 2 * _pow2(-56) and abs(V * V * ms - 1) < 2 * _pow2(-56)
        t = Fraction((w2 << 64) | (w1 << 32) | w0) * _pow2(-86)
        assert abs((-t if sg else t) - s * W) < 8 * _pow2(-60) + 2 * _pow2(-64)


def test_products_keep_their_exponent(lib):
    g = np.random.default_rng(8)
    for i in range(3000):
        a, b = (int(g.integers(2**62, 2**63, dtype=np.uint64)) for _ in range(2))
        if i % 10 == 0:
            a = 2**62
        e = ctypes.c_int(2)
        m = lib.product(a, b, ctypes.byref(e))
        assert 2**62 <= m < 2**63
        exact = Fraction(a * b) * _pow2(-124)
        # the caller adds the factor's own exponent + 2
        assert abs(Fraction(m) * _pow2(-62) * _pow2(e.value) / exact - 1) < _pow2(-59)


def test_shifts_and_sums(lib):
    g = np.random.default_rng(6)
    for k in list(range(0, 100)) + [1000]:
        w = g.integers(0, 2**32, 3, dtype=np.uint32)
        v = (int(w[0]) << 64) | (int(w[1]) << 32) | int(w[2])
        lib.shift(w.ctypes.data_as(ctypes.c_void_p), k)
        assert ((int(w[0]) << 64) | (int(w[1]) << 32) | int(w[2])) == v >> k
    w = g.integers(0, 2**32, (50, 3), dtype=np.uint32)
    w[:, 0] = (g.integers(-2**20, 2**20, 50)).astype(np.int32).view(np.uint32)
    tot = sum((int(np.int32(a)) << 64) + (int(b) << 32) + int(c) for a, b, c in w)
    got = lib.total(w.ctypes.data, 50, -80)
    assert abs(Fraction(got) / (Fraction(tot) * _pow2(-80)) - 1) < _pow2(-51)
