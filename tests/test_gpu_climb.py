"""Boxes that meet across the blocks of the refit: the tree's box is the box
of the vertices, every triangle lies in the boxes above it (a cast over the
tree blocks the rays that a cast over another tree of the part blocks), and
ten builds and refits of a part give the same bits."""
import numpy as np
import pytest

from common import gpu_cast, gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T", [257, 40_000, 300_001])
def test_rebuilt_trees_agree(T):
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(T)
    A = rng.uniform(0, 10, (T, 1, 3))
    V = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-0.1, 0.1, (T, 2, 3))], 1)).reshape(-1, 3).astype(np.float32)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)[rng.permutation(T)]
    P = rng.uniform(0, 10, (50, 3)).astype(np.float32)
    N = rng.normal(size=(50, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    Vt, Ft = gpu_mesh(V, F)
    p = rc.rc_params_default(n_dirs=128)
    other = rc.Bvh(Vt, Ft, builder=1)
    want = gpu_cast(rc, other.h, P, N, p)
    other.close()
    for k in range(10):
        bvh = rc.Bvh(Vt, Ft)
        if k % 2:
            rc.rc_refit_bvh(bvh.h, Vt)
        info = rc.rc_bvh_get_info(bvh.h)
        assert np.array_equal(np.array(info.scene_lo[:], np.float32), V.min(0))
        assert np.array_equal(np.array(info.scene_hi[:], np.float32), V.max(0))
        assert 0 < info.max_depth < 64
        got = gpu_cast(rc, bvh.h, P, N, p)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and got[2][3] == 0
        bvh.close()
