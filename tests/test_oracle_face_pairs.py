"""The oracle's face-adjacent pairs and its L_reg at the sizes the GPU tests ask
for: the pairs of a table of cells against all pairs of boxes tried one by one,
the loss and gradient against a sum over pairs, and 60000 voxels in seconds."""

import os
import subprocess
import sys

import numpy as np
import pytest

import synth


def _all_pairs(sc):
    """Every ordered pair of boxes: j touches i's face with positive area and is no smaller
    (of two equal ones the first in input order is i)."""
    e = (1 << (sc.max_level - sc.level.astype(np.int64)))
    lo = sc.ijk.astype(np.int64) * e[:, None]
    hi = lo + e[:, None]
    out = []
    for i in range(sc.n):
        for j in range(sc.n):
            if i == j or e[j] < e[i] or (e[j] == e[i] and j < i):
                continue
            for a in range(3):
                if all(min(hi[i, b], hi[j, b]) > max(lo[i, b], lo[j, b]) for b in range(3) if b != a):
                    if hi[i, a] == lo[j, a]:
                        out.append((i, j, a, +1))
                    elif lo[i, a] == hi[j, a]:
                        out.append((i, j, a, -1))
    return out


@pytest.mark.parametrize("seed,K,dims", [(1, 0, (6, 5, 4)), (2, 1, (4, 4, 3)), (3, 2, (4, 4, 3)),
                                         (4, 3, (5, 5, 4))])
def test_pairs_are_all_pairs(oracle_lib, seed, K, dims):
    sc = synth.random_multilevel_scene(seed=seed, max_level=K, dims=dims, p_occ=0.7, p_sub=0.4)
    order = np.random.default_rng(seed).permutation(sc.n)[:400]
    sc.level, sc.ijk, sc.params = sc.level[order], sc.ijk[order], sc.params[order]
    pairs = oracle_lib.face_pairs(sc)
    assert len(pairs) > 60
    assert [tuple(int(v) for v in p) for p in pairs] == _all_pairs(sc)


@pytest.mark.parametrize("mode", ["exp", "sdf"])
def test_loss_is_the_sum_over_pairs(oracle_lib, mode):
    """One pair at a time: two voxels alone have that pair's loss and gradient."""
    sc = synth.random_multilevel_scene(seed=6, max_level=2, dims=(3, 2, 2), p_occ=0.8, p_sub=0.4,
                                       mode=mode)
    P = np.asarray(sc.params, np.float64)
    P[:3, :3] = 0.0  # no direction: the normal term is 1, without a gradient
    loss, grad = oracle_lib.reg_loss(sc, P, 0.7, 1.3, 0.4)
    total, sums = 0.0, np.zeros_like(P)
    for i, j, _, _ in oracle_lib.face_pairs(sc):
        two = synth.SceneData(sc.origin, sc.s0, sc.dims, sc.max_level, sc.level[[i, j]],
                              sc.ijk[[i, j]], sc.params[[i, j]], mode, "pair")
        l2, g2 = oracle_lib.reg_loss(two, P[[i, j]], 0.7, 1.3, 0.4)
        total += l2
        sums[[i, j]] += g2
    np.testing.assert_allclose(loss, total, rtol=1e-12)
    np.testing.assert_allclose(grad, sums, rtol=1e-10, atol=1e-12)


def test_sixty_thousand_voxels_end():
    code = ("import numpy as np, synth, oracle; oracle.build(); "
            "sc = synth.random_multilevel_scene(seed=31, max_level=1, dims=(40, 40, 40), "
            "p_occ=0.6, p_sub=0.3, mode='sdf'); n = 60000; "
            "sc.level, sc.ijk, sc.params = sc.level[:n], sc.ijk[:n], sc.params[:n]; "
            "loss, grad = oracle.reg_loss(sc, np.asarray(sc.params, np.float64), 0.7, 1.3, 0.4); "
            "assert np.isfinite(loss) and loss > 0 and np.isfinite(grad).all()")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], cwd=root, check=True, timeout=60)
