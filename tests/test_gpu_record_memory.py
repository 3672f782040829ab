"""The memory that callers get pointers to (records, voxel order, gradients) can be
shared with other processes and freed scenes' blocks are taken again: a handle for
cudaIpcOpenMemHandle is to be had, and scenes built and closed in turn, on one
context, of sizes that grow and shrink, leave the device's free memory where it
was but for what a context may keep."""

import ctypes as C

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


def _runtime():
    """The CUDA runtime that torch has loaded."""
    with open("/proc/self/maps") as f:
        return C.CDLL(next(l.split()[-1] for l in f if "libcudart.so" in l))


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("n", [1, 5000])
def test_exported_to_other_processes(salf, on_device, n):
    sc = synth.random_multilevel_scene(seed=3, max_level=1, dims=(24, 24, 24), p_occ=0.6, p_sub=0.3)
    sc.level, sc.ijk, sc.params = sc.level[:n], sc.ijk[:n], sc.params[:n]
    voxels = sc if not on_device else salf.VoxelSet(
        sc.origin, sc.s0, sc.dims, sc.max_level, torch.from_numpy(sc.level).cuda(),
        torch.from_numpy(sc.ijk).cuda(), torch.from_numpy(np.asarray(sc.params, np.float32)).cuda(),
        sc.mode)
    g = salf.Scene(voxels)
    rt = _runtime()
    for p in (g.params_view().data_ptr(), g.info()["dev_order"], g.grads_view().data_ptr()):
        assert rt.cudaIpcGetMemHandle(C.create_string_buffer(64), C.c_void_p(p)) == 0
    g.close()


def test_blocks_are_taken_again(salf):
    ctx = salf.Context(0)
    sc = synth.random_multilevel_scene(seed=3, max_level=0, dims=(90, 90, 90), p_occ=0.9)
    ref = np.asarray(sc.params, np.float32)
    level, ijk = torch.from_numpy(sc.level).cuda(), torch.from_numpy(sc.ijk).cuda()
    params = torch.from_numpy(ref).cuda()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    held = []
    for n in (1000, 600000, 30, 500000, 600000, 2, 400000, 600000, 7000, 1):
        n = min(n, sc.n)
        g = salf.Scene(salf.VoxelSet(sc.origin, sc.s0, sc.dims, 0, level[:n], ijk[:n], params[:n],
                                     "exp"), ctx=ctx)
        order = to_np(salf.device_view(g.info()["dev_order"], (n,), "<i4"))
        np.testing.assert_array_equal(to_np(g.params_view()), ref[order])
        held.append(g)
        if len(held) > 2:
            held.pop(0).close()
        # what is open, and what the context may keep
        open_bytes = sum(h.info()["device_bytes"] for h in held)
        assert free0 - torch.cuda.mem_get_info()[0] <= open_bytes + (1 << 30) + (64 << 20)
    for h in held:
        h.close()
    del ctx, g, held, h
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= 64 << 20


def test_kept_memory_is_given_back(salf):
    """What a context keeps for its next scenes is there for the library's other
    allocations: on a full device, servers' arenas take it all."""
    ctx = salf.Context(0)
    sc = synth.random_multilevel_scene(seed=3, max_level=0, dims=(140, 140, 140), p_occ=0.9)
    level, ijk = torch.from_numpy(sc.level).cuda(), torch.from_numpy(sc.ijk).cuda()
    params = torch.from_numpy(np.asarray(sc.params, np.float32)).cuda()
    part = lambda n: salf.Scene(salf.VoxelSet(sc.origin, sc.s0, sc.dims, 0, level[:n], ijk[:n],
                                              params[:n], "exp"), ctx=ctx)
    small = part(50000)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    part(sc.n).close()  # leaves some 300 MB of records with the context, and pool memory
    free1 = torch.cuda.mem_get_info()[0]
    assert free0 - free1 > 300 << 20
    room, arena = 48 << 20, 32 << 20
    fill = torch.empty(free1 - room, dtype=torch.uint8, device="cuda")
    servers = []
    try:
        for _ in range(64):
            try:
                servers.append(salf.Server(small, arena, n_streams=1))
            except salf.SalfError as e:
                assert e.status == 2  # out of memory
                break
    finally:
        taken = len(servers) * arena
        for s in servers:
            s.close()
        del fill
        torch.cuda.empty_cache()
    assert taken >= free0 - free1 + room - 3 * arena
    small.close()
