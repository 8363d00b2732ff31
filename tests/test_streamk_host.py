"""The finish phases' chunks (csrc/streamk.cuh), compiled for the host: the grid holds every
chunk of every tile, and every segment and column-partial row lies in one of its chunks.  The
largest count need not be at the first or last tile: 2D mixed tiles (m = 4, columns of the
diagonal too) at 32 tiles and 510 ranges have it at tile 16."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_0262_gb300", "csrc")

SRC = r"""
#include "streamk.cuh"
extern "C" {
int most(int64_t U, int P, int64_t ubeg, int64_t n_it, int m, int diag, int ch, int direct) { return most_chunks(U, P, ubeg, n_it, m, diag, ch, direct); }
int64_t units(int64_t n_it, int m) { return sym_rowstart(n_it, m * n_it, m); }
void row(int64_t U, int P, int64_t ubeg, int64_t n_it, int m, int64_t T, int64_t rows, int ch, int direct, int64_t *o) {
  const RowChunks r = row_chunks(U, P, ubeg, m * n_it, m, T, rows, ch, direct);
  o[0] = r.cf; o[1] = r.cl; o[2] = r.cols; o[3] = r.segs; o[4] = r.ubeg; o[5] = unit_begin(U, P, r.cf); o[6] = unit_begin(U, P, r.cl + 1);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("streamk")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    so = ctypes.CDLL(str(d / "t.so"))
    i64, i32 = ctypes.c_int64, ctypes.c_int
    so.most.argtypes = [i64, i32, i64, i64, i32, i32, i32, i32]
    so.units.argtypes, so.units.restype = [i64, i32], i64
    so.row.argtypes = [i64, i32, i64, i64, i32, i64, i64, i32, i32, ctypes.c_void_p]
    return so


def _check(lib, U, P, ubeg, n_it, m, diag, ch, direct=0):
    nc, at = lib.most(U, P, ubeg, n_it, m, diag, ch, direct), []
    o = (ctypes.c_int64 * 7)()
    first = ubeg
    for T in range(n_it):
        rows = T + diag
        lib.row(U, P, ubeg, n_it, m, T, rows, ch, direct, o)
        cf, cl, cols, segs, u0, lo, hi = o
        assert u0 == first and lo <= first  # the row's units are those of the ranges cf .. cl
        first += m * (n_it - T)
        assert hi >= first and (cols - 1) * ch < rows <= cols * ch
        assert segs == 0 if cl - cf < direct else (segs - 1) * ch < cl - cf + 1 <= segs * ch
        at.append(cols + segs)
    assert max(1, *at) == nc
    return at


def test_every_chunk_is_launched(lib):
    for m, diag, ch in ((4, 1, 16), (1, 1, 16), (1, 1, 64), (2, 0, 16), (4, 0, 16), (8, 1, 16)):
        for n_it in (1, 2, 15, 16, 17, 31, 32, 33, 48, 64, 79, 130):
            U = lib.units(n_it, m)
            for P in sorted({min(U, p) for p in (1, 152, 510, 608, 1135, 1216, 2432, 4864)}):
                _check(lib, U, P, 0, n_it, m, diag, ch)


@pytest.mark.parametrize("n_it,P", [(32, 510), (48, 1135), (48, 1136), (48, 1144), (48, 1145), (48, 1146)])
def test_a_tile_in_the_middle_has_the_most_chunks(lib, n_it, P):
    at = _check(lib, lib.units(n_it, 4), P, 0, n_it, 4, 1, 16)
    assert max(at) > max(at[0], at[-1])


def test_systems_of_an_ensemble(lib):
    tiles = [16, 256, 31, 77, 130, 255]
    U = sum(lib.units(n, 1) for n in tiles)
    for P in (608, 1216, 3648, U):
        ubeg = 0
        for n in tiles:
            _check(lib, U, P, ubeg, n, 1, 1, 128, 4)
            ubeg += lib.units(n, 1)
