"""Spans per ray when the caller leaves the choice to the library: LiDAR sweeps on
both sides of both lines (128 and 320 rays per level-0 cell of the voxels' longest
side) have the bits of the explicit count, alone and in a batch."""

import numpy as np
import pytest

import synth
from tests.parity_util import to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def scene():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    sc = synth.random_multilevel_scene(seed=8, max_level=2, dims=(42, 30, 6), p_occ=0.15)
    lo = (sc.ijk >> sc.level[:, None]).min(axis=0)
    side = int(((sc.ijk >> sc.level[:, None]).max(axis=0) + 1 - lo).max())
    return P.Scene(sc), side


def _lidar(beams, azimuths):
    return synth.lidar(beams, azimuths, synth.lidar_pose((0.35, 0.55, 1.05), 0.2),
                       synth.lidar_pose((0.95, 0.7, 1.05), 0.45), t0=0.0, t1=0.1)


@pytest.mark.parametrize("per_side,above,spans", [(128, 0, 8), (128, 1, 4), (320, 0, 4),
                                                  (320, 1, 1)])
def test_both_sides_of_the_lines(scene, per_side, above, spans):
    g, side = scene
    sen = _lidar(8, per_side * side // 8 + above)  # `above`: 8 rays past the line
    outputs = ("rgb", "depth", "opacity", "intensity")
    kw = dict(t_min=1e-3, outputs=outputs, want_intensity=True)
    free = g.render(sen, **kw)
    fixed = {n: g.render(sen, ray_segments=n, **kw) for n in (1, 4, 8)}
    batch = g.render_batch([_lidar(16, 700), sen, _lidar(4, 100)], **kw)[1]
    torch.cuda.synchronize()
    g.check()
    differ = {n: any((to_np(fixed[n][k]) != to_np(free[k])).any() for k in outputs) for n in fixed}
    assert differ == {n: n != spans for n in fixed}
    for k in outputs:
        np.testing.assert_array_equal(to_np(batch[k]), to_np(free[k]))
