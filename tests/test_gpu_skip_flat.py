"""Skip boxes of flat grids with more columns of bricks than 32-bit table offsets
reach (test_skip_offsets.py): visit lists against the oracle at the grid's far
corner, where the offsets are largest, and rays across the whole grid."""

import numpy as np
import pytest

import synth
from tests.parity_util import check_visits, gpu_render, visit_cap
from tests.test_gpu_skip import _rays, _set

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def salf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    return P


@pytest.mark.parametrize("dims,size", [
    ((37000, 37000, 1), (70, 60, 1)),   # the last with 32-bit offsets
    ((40000, 40000, 4), (70, 60, 4)),   # bricks of 4x4x2 cells
])
def test_visits_of_a_flat_grid(salf, oracle_lib, dims, size):
    rng = np.random.default_rng(dims[2])
    lo = tuple(np.array(dims) - np.array(size))
    sc = _set(rng, dims, lo, size, 120, 0)
    rays = _rays(rng, sc, lo, size, 4000)
    # the grid's other corners; rays along its two long sides, from outside, to each of them
    x1, y1 = dims[0] - 1, dims[1] - 1
    sc.ijk = np.concatenate([sc.ijk, [[0, 0, 0], [x1, 0, 0], [0, y1, 0]]]).astype(np.int32)
    sc.level = np.zeros(len(sc.ijk), np.uint8)
    sc.params = np.concatenate([sc.params, synth.draw_params(rng, 3, "exp")])
    a, e = np.array(sc.origin), sc.s0
    mid = lambda c: a + (np.array(c) + 0.5) * e
    long = [(mid([x1, 0, 0]) + [5.0, 0, 0], [-1, 0, 0]), (mid([0, 0, 0]) - [5.0, 0, 0], [1, 0, 0]),
            (mid([0, y1, 0]) + [0, 5.0, 0], [0, -1, 0]), (mid([0, 0, 0]) - [0, 5.0, 0], [0, 1, 0])]
    rays[:4] = [np.concatenate([o, d, [0, 0]]) for o, d in long]
    sen = synth.explicit_rays(rays)
    cap = 200
    ref = oracle_lib.render(oracle_lib.OracleScene(sc), sen, t_min=0.0, visits_cap=cap,
                            brute_force=True)
    dev = salf.VoxelSet(sc.origin, sc.s0, sc.dims, 0, torch.from_numpy(sc.level).cuda(),
                        torch.from_numpy(sc.ijk).cuda(), torch.from_numpy(sc.params).cuda(), "exp")
    g = salf.Scene(dev)
    out = gpu_render(g, sen, t_min=0.0, visits_cap=cap)
    g.check()
    m, bad = check_visits(oracle_lib, oracle_lib.OracleScene(sc), sen, sc, out["visits"],
                          out["visit_count"], ref["visits"], ref["n_visits"], None)
    assert bad <= visit_cap(m)
    assert out["visit_count"].sum() > m // 4
    np.testing.assert_array_equal(out["visits"][:4], ref["visits"][:4])
    assert (out["visit_count"][:4] >= 2).all()
    g.close()
    torch.cuda.empty_cache()
