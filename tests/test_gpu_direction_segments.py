"""Direction counts at and beyond the line from which a point is cast in
segments of its tiles: whole points and parts of points, both direction
orders, both kinds of grid, the instrumented cast and its list, the batch.
Bits and counts are those of the binary walk, which has no segments."""
import numpy as np
import pytest

import synth
from common import gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LINE = 1066 * 32


def _part(rc, n):
    bvh = rc.Bvh(*gpu_mesh(*synth.pocket_block(2)))
    P, N = torch.empty((n, 3), device="cuda"), torch.empty((n, 3), device="cuda")
    face = torch.empty(n, dtype=torch.int32, device="cuda")
    rc.rc_sample_points(bvh.h, n, rc.rc_params_default(), P, N, face)
    return bvh, P, N


def _cast(rc, h, P, N, dirs, **kw):
    n, W = len(P), (dirs + 31) // 32
    bits = torch.full((n, W), 5, dtype=torch.int32, device="cuda")
    cnt = torch.full((n,), 5, dtype=torch.int32, device="cuda")
    ctr = torch.zeros(8, dtype=torch.int64, device="cuda")
    rc.rc_hemisphere_cast(h, P, N, rc.rc_params_default(n_dirs=dirs, **kw), bits, cnt, ctr)
    assert ctr[0] == n * dirs and ctr[3] == 0
    return bits, cnt, int(ctr[1])


@pytest.mark.parametrize("dirs", [LINE - 31, LINE, LINE + 1, 50_001, 65_535, 65_536])
@pytest.mark.parametrize("kw", [dict(), dict(tile_mode=1), dict(launch_mode=1), dict(collect_stats=1), dict(origin_offset=0.0)], ids=str)
def test_parts_of_points(dirs, kw):
    import paper_2609_05467_gb300 as rc
    bvh, P, N = _part(rc, 9)
    a, b = _cast(rc, bvh.h, P, N, dirs, **kw), _cast(rc, bvh.h, P, N, dirs, tree_width=2, **kw)
    if "origin_offset" not in kw:
        assert a[2] == b[2]
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    bvh.close()


@pytest.mark.parametrize("dirs", [LINE, LINE + 1, 65_536])
def test_whole_points(dirs):
    """With one block per SM only the last two points per resident warp are cast in parts."""
    import paper_2609_05467_gb300 as rc
    n = 2 * 4 * torch.cuda.get_device_properties(0).multi_processor_count + 77
    bvh, P, N = _part(rc, n)
    a, b = _cast(rc, bvh.h, P, N, dirs, blocks_per_sm=1), _cast(rc, bvh.h, P, N, dirs, tree_width=2)
    assert a[2] == b[2] and torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    bvh.close()


def test_list_of_retested_rays():
    import paper_2609_05467_gb300 as rc
    dirs, n = 65_536, 3
    bvh, P, N = _part(rc, n)
    p = rc.rc_params_default(n_dirs=dirs, origin_offset=0.0)
    bits, cnt = torch.zeros((n, dirs // 32), dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    ctr, lst = torch.zeros(8, dtype=torch.int64, device="cuda"), torch.full((n * dirs,), -1, dtype=torch.int64, device="cuda")
    rc.rc_hemisphere_cast_retests(bvh.h, P, N, p, bits, cnt, ctr, lst)
    k = int(ctr[6])
    got = lst[:k].cpu().numpy()
    assert 0 < k <= int(ctr[2]) and len(np.unique(got)) == k and (lst[k:] == -1).all()
    assert (got // 65536 < n).all() and (got >= 0).all()
    bvh.close()


@pytest.mark.parametrize("dirs", [LINE, LINE + 1, 65_536])
def test_batch(dirs):
    import paper_2609_05467_gb300 as rc
    bvh, P, N = _part(rc, 20)
    b = rc.rc_batch_create(rc.rc_params_default(n_dirs=dirs))
    bits = torch.full((20, (dirs + 31) // 32), 3, dtype=torch.int32, device="cuda")
    cnt = torch.full((20,), 3, dtype=torch.int32, device="cuda")
    ctr = torch.zeros(4, dtype=torch.int64, device="cuda")
    rc.rc_batch_add_part(b, bvh.h, P, N, bits, cnt, ctr)
    want = _cast(rc, bvh.h, P, N, dirs, tree_width=2)
    for _ in range(2):
        rc.rc_batch_launch(b)
        torch.cuda.synchronize()
        assert torch.equal(bits, want[0]) and torch.equal(cnt, want[1])
        assert ctr[0] == 20 * dirs and ctr[3] == 0
    rc.rc_batch_destroy(b)
    bvh.close()
