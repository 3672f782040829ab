"""Tile classification of actor frames of a pinhole camera (blocks of 32 tiles,
one lane per tile): the same rays given explicitly take the general
classification, ray by ray, and the same merge of hits.  Ragged tile counts, one-pixel
frames, wide and narrow views, more actors than a mask word holds, a camera
inside an actor's sphere, clipped ray ranges."""

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


def _grid_of_actors(salf, n, rng):
    """n small cars on a jittered grid, clear of one another and of the origin."""
    shells = [salf.Scene(synth.actor_shell(0.9, 0.5, 0.5, seed=60 + k)) for k in range(3)]
    spots = [(x, y) for x in np.arange(-9.0, 9.1, 1.8) for y in np.arange(-9.0, 9.1, 1.8)
             if x * x + y * y > 0.7]
    out = []
    for k in rng.permutation(len(spots))[:n]:
        x, y = np.array(spots[k]) + rng.uniform(-0.2, 0.2, 2)
        c, s = np.cos(a := rng.uniform(0, 6.28)), np.sin(a)
        p = np.array([[c, -s, 0, x], [s, c, 0, y], [0, 0, 1, rng.uniform(-0.3, 0.4)]])
        out.append((shells[k % 3], p, p, 0))
    return out


@pytest.mark.parametrize("w,h,hfov,n,clip", [
    (1, 1, 40.0, 40, None), (8, 4, 60.0, 1, None), (61, 47, 90.0, 40, None),
    (257, 4, 120.0, 70, None), (40, 300, 20.0, 33, None), (96, 64, 170.0, 40, None),
    (640, 360, 60.0, 64, None), (96, 64, 75.0, 40, (1.5, 4.0)),
])
def test_pinhole_frame_equals_its_explicit_rays(salf, w, h, hfov, n, clip):
    rng = np.random.default_rng(w + h)
    sc = synth.random_multilevel_scene(seed=3, max_level=1, dims=(8, 8, 4), p_occ=0.2,
                                       origin=(-2.0, -2.0, -0.6))
    g = salf.Scene(sc)
    acts = _grid_of_actors(salf, n, rng)
    for yaw in (0.0, 1.9, 4.0):
        cam = synth.pinhole(w, h, hfov, synth.camera_pose_looking((0.05, 0.02, 0.2), yaw))
        if clip:
            cam.update(t_near=clip[0], t_far=clip[1])
        dump = to_np(g.render(cam, ray_dump=True)["ray_dump"]).astype(np.float64)
        rays = np.zeros((w * h, 8), np.float32)
        rays[:, :6] = dump[:, :6]
        rays[:, 6:] = clip or (0.0, 0.0)
        kw = dict(t_min=0.0, outputs=("rgb", "depth", "opacity"), visits_cap=128)
        a = g.render_actors(cam, acts, **kw)
        ex = synth.explicit_rays(rays)
        ex.update(pose0=cam["pose0"], pose1=cam["pose1"])  # actors are placed from this origin
        b = g.render_actors(ex, acts, **kw)
        torch.cuda.synchronize()
        g.check()
        # rays equal to FP32 rounding (directions 1e-7, positions 1e-6 m): hits may differ
        # only where a ray grazes a voxel
        same = (a["visits"] == b["visits"]).all(1)
        assert int((~same).sum()) <= max(2, w * h // 500)
        s = same.cpu()
        assert torch.allclose(a["rgb"].cpu()[s], b["rgb"].cpu()[s], atol=1e-4)
        assert torch.allclose(a["depth"].cpu()[s], b["depth"].cpu()[s], atol=1e-3)
