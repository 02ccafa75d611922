"""Rays left over when the next tile of a point enters the pooled walk move to
other slots of the warp's shared memory.  Parts of many small triangles leave
up to 32 pairs of several tiles behind at almost every entry: the bits of ten
casts are one another's and the binary walk's (a ray per lane, no slots)."""
import numpy as np
import pytest

from common import gpu_cast, gpu_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,size,n,dirs", [(3000, 0.8, 61, 1500), (30000, 0.3, 200, 640)])
def test_leftover_rays_keep_their_directions(T, size, n, dirs):
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(T)
    A = rng.uniform(0, 10, (T, 1, 3))
    V = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-size, size, (T, 2, 3))], 1)).reshape(-1, 3).astype(np.float32)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    P = rng.uniform(0, 10, (n, 3)).astype(np.float32)
    N = rng.normal(size=(n, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    want = gpu_cast(rc, bvh.h, P, N, rc.rc_params_default(n_dirs=dirs, tree_width=2))
    for _ in range(10):
        got = gpu_cast(rc, bvh.h, P, N, rc.rc_params_default(n_dirs=dirs))
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        assert got[2][3] == 0
    bvh.close()
