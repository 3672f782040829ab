"""The adjoint's sums over many rays: a voxel's gradient takes one rounding per batch
of 32 rows of its own, so that calls in another order of the atomics differ by no
more than these roundings make.

N_v atomics on voxel v of values of variance s^2 leave partial sums of variance k s^2,
each rounded by at most u = 2^-24 of itself (variance a third of that squared): u^2
s^2 N_v^2 / 6 in all, against a gradient of s^2 N_v.  Over all voxels, and with N_v =
rows of v / 32, the relative noise is at most u sqrt(sum N_v^2 / (6 sum N_v))."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def salf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2507_18713_gb300 as P
    P.load()
    return P


def test_noise_of_large_voxels(salf):
    sc = synth.random_multilevel_scene(seed=1, max_level=2, dims=(6, 5, 4), p_occ=0.6)
    g = salf.Scene(sc)
    cam = synth.pinhole(640, 480, 75.0, synth.camera_pose_looking((-2.2, 0.6, 1.1), 0.15))
    fwd = g.render(cam, saved=True, visits_cap=16)
    torch.cuda.synchronize()
    visits = fwd["visits"].cpu().numpy()
    n = np.bincount(visits[visits >= 0], minlength=sc.n) / 32.0
    bound = 2.0 ** -24 * np.sqrt((n ** 2).sum() / (6.0 * n.sum()))
    grad = torch.randn((640 * 480, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    runs = [g.backward(cam, fwd["saved"], d_rgb=grad).double() for _ in range(24)]
    mean = sum(runs) / len(runs)
    var = sum((r - mean) ** 2 for r in runs) / (len(runs) - 1)
    assert float(var.mean().sqrt() / mean.pow(2).mean().sqrt()) <= bound
