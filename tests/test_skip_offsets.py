"""Offsets into the skip boxes' rectangle tables, over flat, narrow and ordinary
grids: computed in the type that the build chooses, they are the exact ones."""

import ctypes as C
import subprocess

import pytest

from paper_2507_18713_gb300.build import CSRC

SRC = r"""
#include "skip_shape.h"
extern "C" long long offset(long long table, int px, int i, int j, int dy, int dx) {
  return skip_wide_offsets(table) ? skip_rect_offset<long long>(i, j, table, px, dy, dx)
                                  : skip_rect_offset<int>(i, j, (int)table, px, dy, dx);
}
extern "C" int wide(long long table) { return skip_wide_offsets(table); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("skip")
    (tmp / "offset.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-fwrapv", "-shared", "-fPIC", "-I", CSRC,
                    str(tmp / "offset.cpp"), "-o", str(tmp / "offset.so")], check=True)
    f = C.CDLL(str(tmp / "offset.so"))
    f.offset.restype = C.c_longlong
    f.offset.argtypes = [C.c_longlong] + [C.c_int] * 5
    f.wide.argtypes = [C.c_longlong]
    return f


def _bricks(dims):
    """Bricks per axis of voxels that span the grid: 4x4x1 cells, larger ones (first in z)
    while a grid has more than 2^28 of them."""
    p, q = 2, 0
    while True:
        n = [-(-dims[0] // (1 << p)), -(-dims[1] // (1 << p)), -(-dims[2] // (1 << q))]
        if n[0] * n[1] * n[2] <= 1 << 28:
            return n
        p, q = (p, q + 1) if q < 2 else (p + 1, q + 1)


@pytest.mark.parametrize("dims,wide", [
    ((708, 708, 41), False), ((1, 1, 1), False), ((37000, 37000, 1), False),
    ((38000, 38000, 1), True), ((40000, 40000, 2), True), ((40000, 40000, 4), True),
    ((100000, 16000, 4), True), ((65536, 65536, 1), True), ((1 << 21, 1 << 11, 1), True),
    ((4, 512, 1 << 21), False), ((4, 1 << 21, 512), False), ((1 << 21, 4, 65), False),
    ((20000, 20000, 65), False)])
def test_offsets_are_exact(lib, dims, wide):
    n = _bricks(dims)
    px, py, words = n[0] + 15, n[1] + 15, -(-n[2] // 64)
    table = px * py * words
    assert bool(lib.wide(table)) == wide
    for i in range(5):
        for j in range(5):
            for dy in (0, 1 - 31, 31 - (1 << j), 1 - (1 << j)):
                for dx in (0, 1 - 31, 31 - (1 << i), 1 - (1 << i)):
                    want = (i * 5 + j) * table + dy * px + dx
                    assert lib.offset(table, px, i, j, dy, dx) == want
