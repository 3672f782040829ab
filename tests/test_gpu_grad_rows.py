"""Gradient rows that many rays of a warp share: frames of one warp tile whose
rays all cross the same voxels (groups of 7, 8, 15, 16, 28 and 32 rows, the
edges of the ways their sums are split), views across voxel faces (two or more
groups in a warp, lanes apart), and ragged frames, against the oracle's
gradient within the adjoint's own bound."""

import numpy as np
import pytest

import synth
from tests.test_gpu_backward import _case, grad_close

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
@pytest.mark.parametrize("w,h", [(7, 1), (4, 2), (5, 3), (8, 2), (7, 4), (8, 4), (19, 9)])
@pytest.mark.parametrize("hfov", [1.0, 25.0])
def test_shared_rows(salf, oracle_lib, w, h, hfov, mode):
    sc = synth.random_multilevel_scene(seed=5, max_level=1, dims=(5, 4, 3), p_occ=0.8, mode=mode)
    sen = synth.pinhole(w, h, hfov, synth.camera_pose_looking((-1.9, 0.27, 0.83), 0.1))
    for want_intensity in (False, True):
        dg, do, bnd, _ = _case(salf, oracle_lib, sc, sen, want_intensity=want_intensity, seed=w)
        assert np.abs(do).max() > 0
        grad_close(dg, do, bnd)
