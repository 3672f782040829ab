"""L_reg where the device has no room for the block sums: it needs none, the
blocks then add to the loss themselves.  The allocation fails in a fake that a
child process puts in front of the library's own."""

import os
import subprocess
import sys

import pytest

from paper_2507_18713_gb300.build import CSRC, INCLUDE, _nvcc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FAKE = r"""
#include "salf_internal.h"
static bool no_room;
extern "C" void set_no_room(int on) { no_room = on; }
salf_status PoolBuf::get(salf_ctx* ctx, size_t bytes, cudaStream_t stream) {
  if (no_room) return SALF_ERR_OOM;
  st = stream;
  return cudaMallocFromPoolAsync(&p, bytes, ctx->pool, stream) == cudaSuccess ? SALF_OK
                                                                              : SALF_ERR_CUDA;
}
"""

CHILD = r"""
import ctypes as C, sys
import numpy as np, torch
fake = C.CDLL(sys.argv[1], mode=C.RTLD_GLOBAL)
import paper_2507_18713_gb300 as P, synth
sc = synth.random_multilevel_scene(seed=31, max_level=1, dims=(40, 40, 40), p_occ=0.6, p_sub=0.3,
                                   mode="sdf")
g = P.Scene(sc)
params = torch.from_numpy(np.asarray(sc.params, np.float32)).cuda()
loss, grads = g.reg_loss(params, 0.7, 1.3, 0.4)
fake.set_no_room(1)
bare, also = g.reg_loss(params, 0.7, 1.3, 0.4)
torch.cuda.synchronize()
n = sc.n // 256 + 1  # atomics on one float
assert abs(float(bare) - float(loss)) <= n * 2.0 ** -24 * float(loss), (float(bare), float(loss))
assert float((grads - also).abs().max()) <= 1e-4 * float(grads.abs().max())
print("no room, no allocation")
"""


def test_no_room_for_block_sums(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    (tmp_path / "fake.cpp").write_text(FAKE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", INCLUDE, "-I", CSRC,
                    "-I", os.path.join(cuda, "include"), str(tmp_path / "fake.cpp"),
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", "-o", str(tmp_path / "fake.so")],
                   check=True)
    env = dict(os.environ, LD_LIBRARY_PATH=os.path.join(cuda, "lib64") + ":" +
               os.environ.get("LD_LIBRARY_PATH", ""))
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, str(tmp_path / "fake.so")], cwd=root, env=env,
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert "no room" in r.stdout
