"""Scenes outlive the context they were built with: every kind of call on a scene
after salf_destroy gives what it gave before, among them L_reg on more voxels
than its blocks add up by themselves (it takes a temporary from the context)."""

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


def _calls(salf, g, params, sen, tmp):
    out = g.render(sen, saved=True, t_min=1e-3)
    dg = g.backward(sen, out["saved"], d_rgb=torch.ones_like(out["rgb"]), t_min=1e-3)
    loss, grads = g.reg_loss(params, 0.7, 1.3, 0.4)
    ras = g.render_raster(sen)
    g.save(str(tmp))
    torch.cuda.synchronize()
    g.check()
    # the gradients' atomics add in any order
    return ([to_np(out[k]) for k in ("rgb", "depth", "opacity")] + [to_np(ras["rgb"])],
            [to_np(dg), to_np(loss), to_np(grads)])


@pytest.mark.parametrize("on_device", [False, True])
def test_scene_after_its_context(salf, tmp_path, on_device):
    from paper_2507_18713_gb300 import _lib as L
    sc = synth.random_multilevel_scene(seed=31, max_level=1, dims=(24, 24, 24), p_occ=0.6, p_sub=0.3)
    assert sc.n > 8192
    params = torch.from_numpy(np.asarray(sc.params, np.float32)).cuda()
    sen = synth.pinhole(150, 117, 70.0, synth.camera_pose_looking((-1.9, 0.27, 0.83), 0.1))
    voxels = sc if not on_device else salf.VoxelSet(
        sc.origin, sc.s0, sc.dims, sc.max_level, torch.from_numpy(sc.level).cuda(),
        torch.from_numpy(sc.ijk).cuda(), params, sc.mode)
    ctx = salf.Context(0)
    a, b = (salf.Scene(voxels, ctx=ctx) for _ in range(2))
    exact, close = _calls(salf, a, params, sen, tmp_path / "before")
    L.load().salf_destroy(ctx._h)
    ctx._h = None
    for g in (a, b):  # b holds the context alone once a is gone
        after, near = _calls(salf, g, params, sen, tmp_path / "after")
        for x, y in zip(exact, after):
            np.testing.assert_array_equal(x, y)
        for x, y in zip(close, near):
            np.testing.assert_allclose(x, y, rtol=1e-4, atol=1e-4 * np.abs(x).max())
        assert (tmp_path / "before").read_bytes() == (tmp_path / "after").read_bytes()
        g.close()
