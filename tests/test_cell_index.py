"""The column arithmetic of the tiles (csrc/cell_index.h), compiled for the host, up to the largest mesh:
no mesh of 2^30 cells or more in a row is run."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_19169_gb300", "csrc")
SHIM = """
#include "cell_index.h"
using namespace dgk;
extern "C" int column(long long x, int n, int periodic) { return cell_column(column_of(x), n, periodic != 0); }
extern "C" int wrap(int x, int n) { return wrap_column(x, n); }
extern "C" int inside(long long x, int n) { return column_inside(column_of(x), n); }
extern "C" long long tiles(long long n, long long out) { return tiles_of(n, out); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("cell_index")
    (d / "t.cpp").write_text(SHIM)
    # -ftrapv ends the process on a signed overflow
    subprocess.check_call([gxx, "-O1", "-ftrapv", "-shared", "-fPIC", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t.so")])
    L = C.CDLL(str(d / "t.so"))
    L.column.argtypes = [C.c_longlong, C.c_int, C.c_int]
    L.inside.argtypes = [C.c_longlong, C.c_int]
    L.tiles.argtypes, L.tiles.restype = [C.c_longlong, C.c_longlong], C.c_longlong
    return L


# tiles up to 256 columns wide with 6 of halo: columns from -6 to n + 255
@pytest.mark.parametrize("n", [1, 2, 5, 6, 7, 40, 255, 256, 1 << 30, (1 << 30) + 1, (1 << 31) - 29, (1 << 31) - 1])
def test_columns_stay_in_the_row(lib, n):
    for x in {x for c in (0, n // 2, n - 1, n) for x in range(c - 6, c + 256) if -6 <= x <= n + 255}:
        assert lib.column(x, n, 1) == x % n
        assert lib.column(x, n, 0) == min(max(x, 0), n - 1)
        assert lib.inside(x, n) == (0 <= x < n)


# 2D strips: 32 columns from 2 before a multiple of 28 inside the row
@pytest.mark.parametrize("n", [1, 2, 27, 28, 29, 90, (1 << 30) - 1, (1 << 30) + 1, (1 << 31) - 28])
def test_strip_columns_wrap(lib, n):
    last = (lib.tiles(n, 28) - 1) * 28
    for x in {x for s in (0, last) for x in range(s - 2, s + 30)}:
        assert x < 1 << 31 and lib.wrap(x, n) == x % n


@pytest.mark.parametrize("n", [1, 19, 20, 21, (1 << 30) + 3, (1 << 31) - 1])
@pytest.mark.parametrize("out", [20, 28, 116, 244])
def test_tiles_cover_the_row(lib, n, out):
    t = lib.tiles(n, out)
    assert (t - 1) * out < n <= t * out


@pytest.mark.parametrize("nx,ny,status", [(1, (1 << 31) - 5, 0), (1, (1 << 31) - 4, -8),
                                          ((1 << 31) - 28, 1, 0), ((1 << 31) - 27, 1, -8)])
def test_limits_of_2d_meshes(nx, ny, status):
    # the row march counts two rows past the last, and the columns of the last strip, in 32 bits
    from paper_2407_19169_gb300 import _native as N
    L = N.load()
    p = N.Params()
    assert L.dg_params_default(C.byref(p)) == 0
    m = N.Mesh(2, nx, ny, 0.0, 1.0, 0.0, 1.0, (C.c_int * 4)(0, 0, 0, 0))
    assert L.dg_workspace_size(C.byref(m), 1, N.EQ_ADVECTION, C.byref(p), C.byref(C.c_size_t())) == status
