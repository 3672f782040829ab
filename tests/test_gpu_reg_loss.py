"""L_reg (Eq. 7) where the kernel's gathering of gradients can go wrong: pairs of
unequal size at every level distance, gradient buffers that are not 16-byte
aligned (scalar atomics), voxel counts around a block of threads, and
accumulation into what the buffers already hold."""

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
@pytest.mark.parametrize("n", [None, 1, 255, 256, 257])
def test_gradient_against_oracle(salf, oracle_lib, mode, n):
    sc = synth.random_multilevel_scene(seed=21, max_level=3, dims=(4, 5, 4), p_occ=0.7, p_sub=0.5,
                                       mode=mode)
    if n is not None:
        sc.level, sc.ijk, sc.params = sc.level[:n], sc.ijk[:n], sc.params[:n]
    P = np.asarray(sc.params, dtype=np.float32)
    lam = (0.7, 1.3, 0.4)
    ref_loss, ref = oracle_lib.reg_loss(sc, P.astype(np.float64), *lam)
    g = salf.Scene(sc)
    params = torch.from_numpy(P).cuda()
    start = torch.randn((sc.n, 32), generator=torch.Generator().manual_seed(4))
    for shift in (0, 1):  # floats past a 16-byte boundary
        flat = torch.zeros(sc.n * 32 + 4, device="cuda")
        grads = flat[shift:shift + sc.n * 32].view(sc.n, 32)
        grads.copy_(start)
        loss = torch.full((1,), 2.0, device="cuda")
        g.reg_loss(params, *lam, grads=grads, loss=loss)
        torch.cuda.synchronize()
        # an FP32 sum of a few thousand terms, and of at most 6 x 16 pairs per record
        assert abs(float(loss) - 2.0 - ref_loss) <= 1e-5 * (2.0 + abs(ref_loss))
        got = to_np(grads).astype(np.float64) - start.numpy()
        assert np.abs(got - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("mode", ["exp", "sdf"])
@pytest.mark.parametrize("n", [8192, 8193, 60000])
def test_loss_sum(salf, oracle_lib, mode, n):
    """32 blocks of 256 voxels add their sums to the loss one by one, more go through the sum
    over blocks.  A thread's pairs, a warp, a block: up to 20 roundings; 32 or one in the
    loss; 1e-6 for the pairs' own terms, whose errors have either sign."""
    sc = synth.random_multilevel_scene(seed=31, max_level=1, dims=(40, 40, 40), p_occ=0.6,
                                       p_sub=0.3, mode=mode)
    assert sc.n >= n
    sc.level, sc.ijk, sc.params = sc.level[:n], sc.ijk[:n], sc.params[:n]
    P = np.asarray(sc.params, dtype=np.float32)
    ref, _ = oracle_lib.reg_loss(sc, P.astype(np.float64), 0.7, 1.3, 0.4)
    g = salf.Scene(sc)
    params = torch.from_numpy(P).cuda()
    for _ in range(3):
        loss, _ = g.reg_loss(params, 0.7, 1.3, 0.4)
        rel = abs(float(loss) - ref) / ref
        assert rel <= (20 + (32 if n <= 8192 else 1)) * 2.0 ** -24 + 1e-6
