"""The update's point list, tile cones and ray queue at their edges: points
inside the edit's box, far from it, on moved faces, with normals that are not
unit; one tile and many, ragged direction counts, both trees and orders, a
warp's share of points and less.  The updated bits equal a full re-cast up to
rays decided by ambiguous pairs, rows that cannot change stay untouched, and
every count is its row's."""
import numpy as np
import pytest

from common import gpu_mesh, unpack

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("width", [2, 4])
@pytest.mark.parametrize("n,dirs,spread,order,unit", [(1, 1, 1, 0, True), (31, 31, 1, 1, True), (33, 33, 3, 0, True), (257, 1000, 1, 0, True),
                                                      (300, 96, 600, 1, True), (200, 2100, 1, 0, True), (90, 256, 3, 0, False)])
def test_update_equals_recast(n, dirs, spread, order, unit, width):
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(dirs + n)
    T = 600
    A = rng.uniform(0, 10, (T, 1, 3))
    V0 = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-2, 2, (T, 2, 3))], 1)).reshape(-1, 3).astype(np.float32)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    V1 = V0.copy()
    near = np.argsort(np.linalg.norm(A[:, 0] - 5.0, axis=1))[:spread]       # moved triangles: one, a few, all
    V1.reshape(T, 9)[near] += rng.uniform(-1, 1, (spread, 9)).astype(np.float32)
    face = rng.integers(0, T, n).astype(np.int32)
    face[0] = near[0] if n > 1 else face[0]
    P = rng.uniform(-10, 20, (n, 3)).astype(np.float32)
    P[n // 2:] = rng.uniform(3, 7, (n - n // 2, 3)).astype(np.float32)      # in the edit's box or near it
    N = rng.normal(size=(n, 3))
    N /= np.linalg.norm(N, axis=1, keepdims=True)
    if not unit:
        N *= rng.uniform(0.5, 2.0, (n, 1))
    Vt0, Ft = gpu_mesh(V0, F)
    Vt1, _ = gpu_mesh(V1, F)
    Pt, Nt, ft = torch.from_numpy(P).cuda(), torch.from_numpy(N.astype(np.float32)).cuda(), torch.from_numpy(face).cuda()
    b0, b1 = rc.Bvh(Vt0, Ft), rc.Bvh(Vt1, Ft)
    p = rc.rc_params_default(n_dirs=dirs, tree_width=width, point_order=order)
    W = (dirs + 31) // 32

    def cast(h):
        bits, cnt = torch.zeros((n, W), dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
        ctr = torch.zeros(4, dtype=torch.int64, device="cuda")
        rc.rc_hemisphere_cast(h, Pt, Nt, p, bits, cnt, ctr)
        return bits, cnt, ctr

    bits, cnt, _ = cast(b0.h)
    old = bits.cpu().numpy().view(np.uint32)
    changed = torch.zeros(T, dtype=torch.uint8, device="cuda")
    nc, box = rc.rc_changed_faces(Vt0, Vt1, Ft, changed)
    assert nc == spread
    ctr = torch.zeros(4, dtype=torch.int64, device="cuda")
    rc.rc_hemisphere_update(b1.h, Pt, Nt, ft, changed, box, p, bits, cnt, ctr)
    full, fcnt, fctr = cast(b1.h)
    got, want = bits.cpu().numpy().view(np.uint32), full.cpu().numpy().view(np.uint32)
    diff = int(np.unpackbits((got ^ want).view(np.uint8)).sum())
    assert diff <= int(ctr[1].item() + fctr[1].item())
    assert np.array_equal(cnt.cpu().numpy(), unpack(got, 32 * W).sum(1))
    if diff == 0:
        assert torch.equal(cnt, fcnt)
    moved = int(changed.cpu().numpy()[face].sum())
    assert ctr[3].item() == 0 and moved * dirs <= ctr[0].item() <= n * dirs
    # a point whose hemisphere lies wholly away from the box keeps its row
    lo, hi = np.array(box[:3], np.float64), np.array(box[3:], np.float64)
    o = P.astype(np.float64) + 1e-4 * N
    top = (np.maximum((lo - o) * N, (hi - o) * N)).sum(1)
    kept = (top < -1e-3) & (changed.cpu().numpy()[face] == 0)
    if unit:
        assert np.array_equal(got[kept], old[kept])
    b0.close()
    b1.close()
