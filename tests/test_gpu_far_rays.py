"""Explicit rays that start as far from the scene as a float can say (their cells
are clamped: the same rays run on the host in test_walk_far_origins.py): those
that leave the scene behind meet nothing, whatever the kernel variant."""

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


@pytest.mark.parametrize("mode", ["exp", "sdf"])
@pytest.mark.parametrize("dims", [(9, 5, 4), (42, 30, 6)])
def test_rays_leaving_from_afar(salf, mode, dims):
    sc = synth.random_multilevel_scene(seed=8, max_level=2, dims=dims, p_occ=0.15, mode=mode)
    g = salf.Scene(sc)
    mid = np.array(sc.origin) + 0.5 * np.array(dims) * sc.s0
    rows = []
    for axis in range(3):
        for side in (-1.0, 1.0):
            for far in (1e4, 3e8, 2.2e9, 1e12, 1e30, 3.4e38):
                for slope in (0.0, 0.01):
                    r = np.concatenate([mid, np.full(3, slope), [0.0, 0.0]])
                    r[axis], r[3 + axis] = side * far, side
                    rows.append(r)
    rays = np.array(rows, np.float32)
    for many in (rays, np.tile(rays, (300, 1))):  # few and many rays: both ways to read ahead
        out = g.render(salf.rays_sensor(torch.from_numpy(many).cuda()), t_min=0.0,
                       background=(0.25, 0.5, 0.75))
        torch.cuda.synchronize()
        g.check()
        assert not to_np(out["opacity"]).any() and not to_np(out["depth"]).any()
        np.testing.assert_array_equal(to_np(out["rgb"]),
                                      np.tile(np.float32([0.25, 0.5, 0.75]), (len(many), 1)))


def test_spawn_point_of_a_far_primary(salf):
    """The hit point o + (D / O) d of a ray from 2^25 cells away, in the float's own steps of
    4 cells, against 64 bits: the origin's cell takes more than a float's 24 bits."""
    n = 12
    ijk = np.stack(np.meshgrid(np.arange(n), np.arange(3), np.arange(3), indexing="ij"),
                   -1).reshape(-1, 3).astype(np.int32)
    params = synth.draw_params(np.random.default_rng(1), len(ijk), "exp")
    sc = synth.SceneData((1.0, 0.0, 0.0), 1.0, (n, 3, 3), 0, np.zeros(len(ijk), np.uint8), ijk,
                         params, "exp", "block")
    g = salf.Scene(sc)
    far = 2.0 ** 25 + 4.0 * np.arange(1, 9)
    hit = np.array([4.0, 8.0] * 4)
    rays = np.zeros((8, 8), np.float32)
    rays[:, 0], rays[:, 1:3], rays[:, 3] = -far, 1.5, 1.0
    depth = torch.from_numpy((far + hit).astype(np.float32)).cuda()
    assert (depth.cpu().numpy().astype(np.float64) == far + hit).all()
    for kind in ("reflect", "shadow"):
        out = to_np(g.secondary_rays(salf.rays_sensor(torch.from_numpy(rays).cuda()), depth,
                                     torch.ones_like(depth), kind=kind, offset=0.0))
        assert out[:, 3:6].any(axis=1).all()
        np.testing.assert_allclose(out[:, :3], np.stack([hit, 0 * hit + 1.5, 0 * hit + 1.5], 1),
                                   rtol=2.0 ** -23)
