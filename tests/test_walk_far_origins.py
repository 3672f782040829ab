"""Explicit rays from any origin a float can hold: the walk reads nothing outside
its buffers and ends, and a finite origin has a finite cell and fraction whose
sum is the origin's.  The traversal header itself runs here, compiled for the
host with bounds-checked reads (host/walk.cpp), on a grid whose skip boxes reach
its faces."""

import ctypes as C
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2507_18713_gb300.build import CSRC, INCLUDE, _nvcc

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("walk")
    src = open(os.path.join(CSRC, "traverse.cuh")).read()
    src = "\n".join(l for l in src.split("\n") if "prefetch.global" not in l)
    (tmp / "traverse_host.cuh").write_text(re.sub(r"\(int\)([fk])\b", r"to_int(\1)", src))
    lib = str(tmp / "walk.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fwrapv", "-ffp-contract=off",
                    "-w", "-I", str(tmp), "-I", INCLUDE, "-I", CSRC, "-I", cuda,
                    os.path.join(HERE, "host", "walk.cpp"), "-o", lib], check=True)
    f = C.CDLL(lib).walk_ray
    f.restype = C.c_long
    return f


def _grid(nb, voxels):
    """Occupancy words and skip boxes of nb[a] blocks of 4x4x4 cells holding some
    level-0 voxels: an empty brick's box is the run of empty columns towards the
    octant's x, whole in y and z only one brick wide."""
    cells = np.zeros((4 * nb[2], 4 * nb[1], 4 * nb[0]), bool)
    for x, y, z in voxels:
        cells[z, y, x] = True
    words = np.zeros((nb[2], nb[1], nb[0], 4), np.uint32)
    for z, y, x in np.argwhere(cells):
        b = (x & 1) | (y & 1) << 1 | (z & 1) << 2 | (x & 2) << 2 | (y & 2) << 3 | (z & 2) << 4
        words[z // 4, y // 4, x // 4, b // 32] |= np.uint32(1 << (b % 32))
    words[..., 3] = 0  # any block's first voxel will do
    n = (nb[0], nb[1], 4 * nb[2])
    full = cells.reshape(n[2], n[1], 4, n[0], 4).any(axis=(2, 4))
    skip = np.zeros((8, n[2], n[1], n[0]), np.uint16)
    for o in range(8):
        f = full[::-1 if o & 4 else 1, ::-1 if o & 2 else 1, ::-1 if o & 1 else 1]
        run = np.zeros(f.shape[:2], int)
        for x in reversed(range(n[0])):
            run = np.where(f[:, :, x], 0, np.minimum(run + 1, 31))
            skip[o, :, :, x] = np.where(f[:, :, x], 0, run | 1 << 5 | 1 << 10)
    return words, skip, n


FAR = [0.0, 1.0, 3e5, 2.0 ** 29, 2.2e9, 4.3e9, 1e12, 1e30, 3.4e38]


@pytest.mark.parametrize("ahead", [0, 1])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("cell", [0.2, 1.0, 8.0])
@pytest.mark.parametrize("blocks", [25, 40])
def test_reads_stay_inside(walk, blocks, cell, axis, ahead):
    nb = (blocks, blocks, blocks)
    e = 4 * blocks - 1
    words, skip, n = _grid(nb, [(0, 0, 0), (e, e, e), (e // 2, e // 2, e // 2)])
    box = np.array([0, 0, 0, e + 1, e + 1, e + 1], np.int32)
    origin = np.array([-3.0, 0.5, 0.25])
    for far in FAR:
        for side in (-1.0, 1.0):
            for way in (-1.0, 1.0):
                for slope in (0.0, 0.01):
                    _check(walk, words, skip, n, nb, box, origin, cell, axis, ahead, side * far,
                           way, slope)
    for odd in (np.inf, -np.inf, np.nan):
        _check(walk, words, skip, n, nb, box, origin, cell, axis, ahead, odd, 1.0, 0.01)


def _check(walk, words, skip, n, nb, box, origin, cell, axis, ahead, far, way, slope):
    ray = np.zeros(8, np.float32)
    ray[:3] = origin + cell * np.array([41.3, 61.7, 21.9])
    ray[axis] = far
    ray[3:6] = slope
    ray[3 + axis] = way
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    st, hits = C.c_int(), C.c_int()
    Oi, Of = np.zeros(3, np.int32), np.zeros(3, np.float32)
    mdim, nn = np.array(nb, np.int32), np.array(n, np.int32)
    what = (cell, axis, ahead, far, way, slope)
    assert walk(p(ray), p(origin), C.c_double(cell), p(mdim), p(nn), p(box), p(words), p(skip),
                ahead, 4000, C.byref(st), C.byref(hits), p(Oi), p(Of)) == 0, what
    if not np.isfinite(far):
        return
    assert np.isfinite(Of).all(), what
    exact = (ray[:3].astype(np.float64) - origin) / cell
    near = np.abs(exact) < 2.0 ** 31 - 2.0 ** 23
    # 48 bits of the origin, and the fraction's own rounding
    err = np.abs(Oi.astype(np.float64) + Of - exact)[near]
    assert (err <= 2.0 ** -46 * np.abs(exact[near]) + 2.0 ** -24).all(), what
    assert ((Of >= 0) & (Of <= 1))[near].all(), what
    # beyond that the cell stays so far out that no plane's distance from it wraps
    assert (np.abs(Oi.astype(np.int64)) <= 2 ** 31 - 2 ** 23).all(), what
