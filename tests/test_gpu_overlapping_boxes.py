"""Parts whose boxes all overlap: thin diagonal needles, so that a ray meets
nearly every node and leaf and is rarely blocked.  More pairs wait than the
pooled walks' stack holds, and the 32 rays of a warp meet 32 times as many as
one ray can.  Bits, masks and counters are those of the binary walk (a ray per
lane), and no walk ends early (counters[3])."""
import numpy as np
import pytest

import synth
from common import gpu_cast, gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TURN = synth.rotation(12.0, -7.0, 25.0).astype(np.float32).reshape(-1)


def _needles(T, seed=3):
    """T needles along the diagonal of a box of 10 mm, a micrometre thick."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(0, 0.5, (T, 3))
    b = a + 9.0 + rng.uniform(0, 0.5, (T, 3))
    c = b + rng.normal(size=(T, 3)) * 1e-3
    return np.stack([a, b, c], 1).reshape(-1, 3).astype(np.float32), np.arange(3 * T, dtype=np.int32).reshape(T, 3)


def _points(n, seed=5):
    rng = np.random.default_rng(seed)
    N = rng.normal(size=(n, 3))
    return rng.uniform(0, 10, (n, 3)).astype(np.float32), (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("T,n,dirs", [(130, 40, 256), (4000, 40, 97), (20_000, 130, 256), (100_000, 33, 96)])
def test_hemisphere(T, n, dirs):
    import paper_2609_05467_gb300 as rc
    bvh = rc.Bvh(*gpu_mesh(*_needles(T)))
    P, N = _points(n)
    a = gpu_cast(rc, bvh.h, P, N, rc.rc_params_default(n_dirs=dirs))
    b = gpu_cast(rc, bvh.h, P, N, rc.rc_params_default(n_dirs=dirs, tree_width=2))
    assert a[2][3] == 0 and b[2][3] == 0 and a[2][0] == b[2][0] == n * dirs and a[2][1] == b[2][1]
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert 0 < a[1].sum() < n * dirs
    bvh.close()


@pytest.mark.parametrize("T,n", [(130, 100), (20_000, 500), (100_000, 64)])
@pytest.mark.parametrize("frame", [np.eye(3).reshape(-1), TURN], ids=["identity", "turned"])
def test_axes_and_tool(T, n, frame):
    import paper_2609_05467_gb300 as rc
    bvh = rc.Bvh(*gpu_mesh(*_needles(T)))
    P, N = (torch.from_numpy(q).cuda() for q in _points(n))
    out = []
    for width in (0, 2):
        p = rc.rc_params_default(frame=frame, tree_width=width)
        mask, tool = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")
        travel = torch.zeros((n, 6), device="cuda")
        ctr = torch.zeros((2, 4), dtype=torch.int64, device="cuda")
        rc.rc_orthogonal_cast(bvh.h, P, N, p, mask, travel, ctr[0])
        rc.rc_tool_cast(bvh.h, P, N, p, 0.1, 5, tool, ctr[1])
        out.append([q.cpu().numpy() for q in (mask, tool, travel, ctr)])
    a, b = out
    assert (a[3][:, 3] == 0).all() and (b[3][:, 3] == 0).all()
    assert np.array_equal(a[3][:, 0], b[3][:, 0])
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)
    bvh.close()


def test_batch():
    import paper_2609_05467_gb300 as rc
    p = rc.rc_params_default(n_dirs=96)
    b = rc.rc_batch_create(p)
    parts = []
    for k, (V, F) in enumerate((_needles(20_000), synth.pocket_block(1))):
        bvh = rc.Bvh(*gpu_mesh(V, F))
        P, N = (torch.from_numpy(q).cuda() for q in _points(60, k))
        out = [(torch.zeros((60, 3), dtype=torch.int32, device="cuda"), torch.zeros(60, dtype=torch.int32, device="cuda"))
               for _ in range(2)]
        rc.rc_batch_add_part(b, bvh.h, P, N, *out[0])
        rc.rc_hemisphere_cast(bvh.h, P, N, rc.rc_params_default(n_dirs=96, tree_width=2), *out[1])
        parts.append((bvh, P, N, out))
    rc.rc_batch_launch(b)
    torch.cuda.synchronize()
    for bvh, _, _, out in parts:
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        bvh.close()
    rc.rc_batch_destroy(b)
