"""Points on moved faces beside points that only see the edit: the first are
cast tile by tile, the others' rays wait in a queue between.  Every point on
a moved face has the bits of a full cast, whatever its row held before."""
import numpy as np
import pytest

from common import gpu_mesh, unpack

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("width", [2, 4])
@pytest.mark.parametrize("n,dirs,share", [(1, 33, 1.0), (64, 32, 1.0), (300, 321, 1.0), (300, 1024, 0.5), (500, 97, 0.1)])
def test_moved_points_are_cast_anew(n, dirs, share, width):
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(n + dirs)
    T = 500
    A = rng.uniform(0, 10, (T, 1, 3))
    V0 = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-2, 2, (T, 2, 3))], 1)).reshape(-1, 3).astype(np.float32)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    V1 = V0.copy()
    V1.reshape(T, 9)[: max(1, int(share * T))] += rng.uniform(-0.3, 0.3, (max(1, int(share * T)), 9)).astype(np.float32)
    face = rng.integers(0, T, n).astype(np.int32)
    face[0] = 0
    P = rng.uniform(0, 10, (n, 3)).astype(np.float32)
    N = rng.normal(size=(n, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    Vt0, Ft = gpu_mesh(V0, F)
    Vt1, _ = gpu_mesh(V1, F)
    Pt, Nt, ft = (torch.from_numpy(q).cuda() for q in (P, N, face))
    b0, b1 = rc.Bvh(Vt0, Ft), rc.Bvh(Vt1, Ft)
    p = rc.rc_params_default(n_dirs=dirs, tree_width=width)
    W = (dirs + 31) // 32
    bits, cnt = torch.zeros((n, W), dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    full, fcnt = torch.zeros_like(bits), torch.zeros_like(cnt)
    rc.rc_hemisphere_cast(b0.h, Pt, Nt, p, bits, cnt)
    fctr, ctr = (torch.zeros(4, dtype=torch.int64, device="cuda") for _ in range(2))
    rc.rc_hemisphere_cast(b1.h, Pt, Nt, p, full, fcnt, fctr)
    changed = torch.zeros(T, dtype=torch.uint8, device="cuda")
    _, box = rc.rc_changed_faces(Vt0, Vt1, Ft, changed)
    moved = changed[ft.long()] != 0
    bits[moved] = -1                                         # rows of moved points do not count
    cnt[moved] = 12345
    rc.rc_hemisphere_update(b1.h, Pt, Nt, ft, changed, box, p, bits, cnt, ctr)
    got, want = bits.cpu().numpy().view(np.uint32), full.cpu().numpy().view(np.uint32)
    assert int(fctr[1]) == 0 and int(ctr[1]) == 0            # no ray that only an ambiguous pair decides
    assert np.array_equal(got, want) and torch.equal(cnt, fcnt)
    assert np.array_equal(unpack(got, dirs).sum(1), cnt.cpu().numpy())
    assert int(ctr[3]) == 0 and int(moved.sum()) * dirs <= int(ctr[0]) <= n * dirs
    b0.close()
    b1.close()
