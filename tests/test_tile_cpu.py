"""The planned queue's walk over an image visits every pixel once, up to the
widest rows that a buffer of 2^31 - 1 rays can hold.

The walk is plain C++ (csrc/tile.h); it is compiled for the host here, as the
states of such a row would take 200 GB of device memory."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

PROGRAM = r"""
#include "tile.h"
extern "C" void walk(const unsigned *p, long n, unsigned nx, unsigned ny, int by_row, unsigned *row, unsigned *col)
{
    for (long i = 0; i < n; ++i) {
        const gray::Pixel x = gray::tile_pixel(p[i], nx, ny, by_row != 0);
        row[i] = x.row;
        col[i] = x.col;
    }
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile")
    src, lib = str(d / "walk.cpp"), str(d / "walk.so")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1303_5057_gb300", "csrc"),
                    "-o", lib, src], check=True)
    L = C.CDLL(lib)
    u = np.ctypeslib.ndpointer(np.uint32, flags="C_CONTIGUOUS")
    L.walk.argtypes = [u, C.c_long, C.c_uint, C.c_uint, C.c_int, u, u]
    L.walk.restype = None

    def call(p, nx, ny, by_row):
        p = np.ascontiguousarray(p, dtype=np.uint32)
        row, col = np.empty_like(p), np.empty_like(p)
        L.walk(p, p.size, nx, ny, int(by_row), row, col)
        return row.astype(np.int64), col.astype(np.int64)
    return call


def expected(p, nx, ny, by_row):
    """The same walk in 64-bit arithmetic."""
    high = 1 if by_row else 4
    strip = p // (high * nx)
    q = p - strip * high * nx
    rows = np.minimum(high, ny - high * strip)
    col = q // rows
    return high * strip + q - col * rows, col


@pytest.mark.parametrize("by_row", [False, True])
@pytest.mark.parametrize("nx, ny", [(1, 1), (70, 1), (1, 70), (33, 4), (33, 5), (7, 6), (50, 7), (8, 9)])
def test_every_pixel_once(walk, nx, ny, by_row):
    p = np.arange(nx * ny)
    row, col = walk(p, nx, ny, by_row)
    assert np.array_equal(np.sort(row * nx + col), p)
    want = expected(p, nx, ny, by_row)
    assert np.array_equal(row, want[0]) and np.array_equal(col, want[1])


@pytest.mark.parametrize("by_row", [False, True])
@pytest.mark.parametrize("nx, ny", [
    (2 ** 30 - 1, 1), (2 ** 30 + 1, 1), (2 ** 30, 1), (3 * 2 ** 29 + 5, 1), (2 ** 31 - 1, 1),  # 4 nx passes 2^32
    (2 ** 30 - 1, 2), (2 ** 29 + 3, 3), (2 ** 29 - 1, 4), (2 ** 28 + 1, 5), (1, 2 ** 31 - 1), (46341, 46340)])
def test_widest_images(walk, nx, ny, by_row):
    n = nx * ny
    assert n < 2 ** 31
    rng = np.random.default_rng(1)
    p = np.unique(np.concatenate([np.arange(100), n - 1 - np.arange(100), rng.integers(0, n, 20000),
                                  np.clip(n // 2 + np.arange(-50, 50), 0, n - 1)]))
    row, col = walk(p, nx, ny, by_row)
    assert row.min() >= 0 and row.max() < ny and col.min() >= 0 and col.max() < nx
    want = expected(p, nx, ny, by_row)
    assert np.array_equal(row, want[0]) and np.array_equal(col, want[1])
