"""Launches of few rays read each next step's box ahead, launches of many (for the scene's
side) read it when the step needs it: a frame alone, below the line, and the same frame in
batches beyond it give the same bits.  Sides of 9 to 42 level-0 cells put the line at 648 to
3024 tiles of 32 rays."""

import numpy as np
import pytest

import synth
from tests.parity_util import to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def salf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    return P


def _sensor(kind):
    pose = synth.camera_pose_looking((-1.9, 0.27, 0.83), 0.1)
    if kind == "pinhole":
        return synth.pinhole(150, 117, 70.0, pose)  # 19 x 30 tiles
    if kind == "fisheye":
        return synth.fisheye(150, 117, 170.0, pose)
    if kind == "lidar":
        return synth.lidar(32, 500, synth.lidar_pose((0.35, 0.55, 1.05), 0.2),
                           synth.lidar_pose((0.95, 0.7, 1.05), 0.45), t0=0.0, t1=0.1)
    rng = np.random.default_rng(2)
    rays = np.zeros((17000, 8), np.float32)  # 532 tiles
    rays[:, :3] = rng.uniform(-2, 6, (17000, 3))
    d = rng.uniform(0, 2, (17000, 3)) - rays[:, :3]
    rays[:, 3:6] = d / np.linalg.norm(d, axis=1, keepdims=True)
    return synth.explicit_rays(rays)


@pytest.mark.parametrize("mode", ["exp", "sdf"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["pinhole", "fisheye", "lidar", "explicit"])
@pytest.mark.parametrize("dims", [(9, 5, 4), (42, 30, 6)])
def test_same_bits_on_both_sides_of_the_line(salf, kind, dtype, mode, dims):
    sc = synth.random_multilevel_scene(seed=8, max_level=2, dims=dims, p_occ=0.15, mode=mode)
    g = salf.Scene(sc, dtype=dtype)
    sen = _sensor(kind)
    lidar = kind == "lidar"
    outputs = ("rgb", "depth", "opacity") + (("intensity",) if lidar else ())
    kw = dict(t_min=1e-3, outputs=outputs, want_intensity=lidar)
    if lidar:
        kw["ray_segments"] = 1
    lone = g.render(sen, **kw)
    batch = g.render_batch([sen] * 7, **kw)
    torch.cuda.synchronize()
    g.check()
    assert to_np(lone["opacity"]).max() > 0
    for k in outputs:
        a = to_np(lone[k])
        for b in batch:
            np.testing.assert_array_equal(a, to_np(b[k]))
