"""Skip boxes of empty space (one 2-byte box per empty brick and direction
octant): visit lists against the oracle on voxel sets where the boxes reach
their limits -- single voxels at the corners of the tight box, grids of 64, 65
and 130 brick layers (boxes end at words of 64 layers), empty stretches longer
than the largest box, offsets that are not whole bricks, and grids so large
that bricks hold more than a layer of a block."""

import numpy as np
import pytest

import synth
from tests.parity_util import check_visits, gpu_render, visit_cap

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def salf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    return P


def _set(rng, dims, lo, size, n, K):
    """n distinct voxels (half of them level K children) in a box of level-0
    cells at lo, and one voxel at each of two opposite corners of the box."""
    cells = np.unique(rng.integers(0, size, size=(n, 3)), axis=0)
    cells = np.unique(np.concatenate([cells, [[0, 0, 0], np.array(size) - 1]]), axis=0)
    level = np.zeros(len(cells), np.uint8)
    ijk = cells + np.array(lo)
    if K:
        split = rng.random(len(cells)) < 0.5
        level[split] = K
        ijk[split] = (ijk[split] << K) + rng.integers(0, 1 << K, size=(split.sum(), 3))
    params = synth.draw_params(rng, len(cells), "exp")
    return synth.SceneData((-1.0, 0.5, 0.25), 0.2, dims, K, level, ijk.astype(np.int32), params,
                           "exp", "sparse")


def _rays(rng, sc, lo, size, R):
    """Rays in all octants, some parallel to an axis or an axis plane, through
    points of the voxels' box, from inside and outside it."""
    a = np.array(sc.origin) + np.array(lo) * sc.s0
    e = np.array(size) * sc.s0
    to = a + rng.random((R, 3)) * e
    o = a + rng.uniform(-0.3, 1.3, size=(R, 3)) * e
    half = rng.random(R) < 0.5
    v = np.argmax(rng.random((R, sc.n)), axis=1) if sc.n < 500 else rng.integers(0, sc.n, R)
    edge = sc.s0 / (1 << sc.level[v].astype(int))
    to[half] = (np.array(sc.origin) + (sc.ijk[v] + rng.random((R, 3))) * edge[:, None])[half]
    d = to - o
    d[:R // 20, 0] = 0.0
    d[R // 20:R // 10, 2] = 0.0
    d[R // 10:R // 8, :2] = 0.0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return np.concatenate([o, d, np.zeros((R, 2))], axis=1).astype(np.float32)


@pytest.mark.parametrize("dims,lo,size,n,K", [
    ((64, 64, 64), (0, 0, 0), (64, 64, 64), 60, 0),
    ((200, 180, 65), (3, 5, 0), (190, 170, 65), 40, 1),
    ((300, 40, 130), (1, 2, 3), (290, 37, 126), 90, 2),
    ((33, 400, 200), (0, 1, 6), (33, 395, 190), 30, 1),
    ((64, 64, 4), (9, 10, 1), (50, 40, 1), 25, 0),
    ((4096, 4096, 272), (1501, 2003, 65), (90, 70, 60), 150, 1),     # bricks of 4x4x2 cells
    ((16384, 16384, 68), (9001, 13, 2), (150, 60, 60), 150, 1),     # bricks of 8x8x8 cells
])
def test_visits_of_sparse_sets(salf, oracle_lib, dims, lo, size, n, K):
    rng = np.random.default_rng(n + dims[2])
    sc = _set(rng, dims, lo, size, n, K)
    rays = _rays(rng, sc, lo, size, 4000)
    sen = synth.explicit_rays(rays)
    cap = 200
    ref = oracle_lib.render(oracle_lib.OracleScene(sc), sen, t_min=0.0, visits_cap=cap,
                            brute_force=True)
    dev = salf.VoxelSet(sc.origin, sc.s0, sc.dims, K, torch.from_numpy(sc.level).cuda(),
                        torch.from_numpy(sc.ijk).cuda(), torch.from_numpy(sc.params).cuda(), "exp")
    host_too = np.prod(np.array(dims, np.int64)) < 10 ** 8
    for voxels in (sc, dev) if host_too else (dev,):  # host and device builds
        g = salf.Scene(voxels)
        out = gpu_render(g, sen, t_min=0.0, visits_cap=cap)
        g.check()
        m, bad = check_visits(oracle_lib, oracle_lib.OracleScene(sc), sen, sc, out["visits"],
                              out["visit_count"], ref["visits"], ref["n_visits"], None)
        assert bad <= visit_cap(m)
        assert out["visit_count"].sum() > m // 4
        g.close()
    torch.cuda.empty_cache()
