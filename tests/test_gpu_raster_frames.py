"""The tile kernel's variants for small and large frames: the pixels that a frame
just below the line shares with frames above it are equal bit for bit, and equal
the ray kernel's, on lists longer than a chunk of either variant."""

import numpy as np
import pytest

import synth
from tests.parity_util import to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

OUTS = ("rgb", "depth", "opacity", "intensity")


@pytest.fixture(scope="module")
def salf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    return P


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode", ["exp", "sdf"])
def test_same_pixels_on_both_sides_of_the_line(salf, mode, dtype):
    sc = synth.driving_scene(300_000, seed=4, ground_extent=77, n_actors=40, mode=mode)
    g = salf.Scene(sc, dtype=dtype)
    pose = synth.camera_pose_looking((0.13, 0.07, 1.71), 0.1)
    frames = {}
    for w, h in ((1600, 1600), (1601, 1600), (1613, 1607)):  # 10000, 10100, 10201 tiles
        cam = dict(synth.pinhole(1600, 1600, 70.0, pose), width=w, height=h)
        stats = {}
        kw = dict(outputs=OUTS, want_intensity=True, t_min=1e-3)
        out = g.render_raster(cam, stats=stats, **kw)
        assert stats["tiles"] == -(-w // 16) * -(-h // 16)
        frames[w] = {k: to_np(out[k]).reshape(h, w, -1)[:1600, :1600] for k in OUTS}
    ray = g.render(cam, **kw)
    torch.cuda.synchronize()
    g.check()
    assert frames[1600]["opacity"].max() > 0.5
    same = np.ones((1600, 1600), bool)
    for k in OUTS:
        for w in (1601, 1613):
            np.testing.assert_array_equal(frames[1600][k], frames[w][k])
        same &= (to_np(ray[k]).reshape(h, w, -1)[:1600, :1600] == frames[1600][k]).all(axis=2)
    assert same.mean() > 0.9999
