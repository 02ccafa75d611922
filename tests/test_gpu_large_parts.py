"""Branches for large parts: vertex ranges kept per block of 2,048 instead of
per warp (more than 2^20 vertices) in the frame search, and 64-bit pairs (more
than 2^24 triangles) in the axis casts, the tool cast and the batch."""
import numpy as np
import pytest

from common import gpu_mesh
from oracle import frames as ofr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nV", [2**20 - 1, 2**20, 2**20 + 1, 2**20 + 2048, 2**20 + 333_333])
def test_frame_candidates(nV):
    """6,000 outer vertices, which alone carry faces, scattered among vertices well inside their hull: the boxes are those of
    the outer ones, which the oracle gets alone."""
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(nV)
    k = 6000
    outer = rng.normal(size=(k, 3))
    outer = (10.0 * outer / np.linalg.norm(outer, axis=1, keepdims=True) * [3.0, 2.0, 1.0] + [100.0, -50.0, 7.0]).astype(np.float32)
    F = rng.integers(0, k, (1500, 3)).astype(np.int32)
    F[0] = [0, 1, 2]
    V = (rng.uniform(-4.0, 4.0, (nV, 3)) + [100.0, -50.0, 7.0]).astype(np.float32)
    at = rng.choice(nV, k, replace=False)
    at[:2] = [0, nV - 1]                                     # the first and the last vertex are outer ones
    assert len(set(at)) >= k - 2
    at = np.unique(at)
    at = np.concatenate([at, rng.choice(np.setdiff1d(np.arange(nV), at), k - len(at), replace=False)])
    V[at] = outer
    bvh = rc.Bvh(*gpu_mesh(V, at[F].astype(np.int32)))
    fr = rc.rc_frame_candidates(bvh.h, rc.rc_params_default())
    cands = ofr.frame_candidates(outer, F)
    assert fr.k == len(cands)
    for c, cand in enumerate(cands):
        assert (fr.source[c], fr.box_axis[c], fr.box_step[c]) == (cand["source"], cand["box_axis"], cand["box_step"])
        assert np.array_equal(fr.frame_array(c).view(np.uint32), cand["frame"].view(np.uint32)), c
        assert fr.volume[c] == cand["volume"]
    bvh.close()


@pytest.mark.parametrize("rows", [2048, 2049])
def test_pairs_of_axis_tool_and_batch(rows):
    """2^24 triangles use 32-bit pairs, one row more of the grid 64-bit ones."""
    import paper_2609_05467_gb300 as rc
    cols = 4096
    x = torch.arange(cols + 1, device="cuda", dtype=torch.float32)
    y = torch.arange(rows + 1, device="cuda", dtype=torch.float32)
    z = 3.0 * torch.sin(0.13 * x)[None, :] * torch.cos(0.17 * y)[:, None] + 40.0 * torch.sin(0.003 * y)[:, None]
    V = torch.stack([x[None, :].expand_as(z), y[:, None].expand_as(z), z], 2).reshape(-1, 3).contiguous()
    q = (torch.arange(rows, device="cuda")[:, None] * (cols + 1) + torch.arange(cols, device="cuda")[None, :]).reshape(-1)
    F = torch.cat([torch.stack([q, q + 1, q + cols + 2], 1), torch.stack([q, q + cols + 2, q + cols + 1], 1)]).int()
    assert (F.shape[0] > 1 << 24) == (rows > 2048)
    bvh = rc.Bvh(V, F.contiguous())
    small = rc.Bvh(V[: 3 * (cols + 1)].contiguous(), F[: cols].contiguous())
    n, dirs = 400, 70
    frame = np.array([[0.8, -0.6, 0], [0.6, 0.8, 0], [0, 0, 1]], np.float32).reshape(-1)
    pts = []
    for h in (bvh.h, small.h):
        P, N = torch.empty((n, 3), device="cuda"), torch.empty((n, 3), device="cuda")
        face = torch.empty(n, dtype=torch.int32, device="cuda")
        rc.rc_sample_points(h, n, rc.rc_params_default(), P, N, face)
        pts.append((P, N))
    P, N = pts[0]
    out = []
    for width in (4, 2):
        got = []
        for f in (np.eye(3).reshape(-1), frame):
            p = rc.rc_params_default(frame=f, tree_width=width)
            mask, tool = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")
            travel = torch.zeros((n, 6), device="cuda")
            ctr = torch.zeros((2, 4), dtype=torch.int64, device="cuda")
            rc.rc_orthogonal_cast(bvh.h, P, N, p, mask, travel, ctr[0])
            rc.rc_tool_cast(bvh.h, P, N, p, 1.5, 5, tool, ctr[1])
            assert int(ctr[0, 3]) == 0 and int(ctr[1, 3]) == 0
            got += [mask, tool, travel, ctr[0, :2]]
        p = rc.rc_params_default(n_dirs=dirs, tree_width=width)
        b = rc.rc_batch_create(p)
        for h, (Q, M) in zip((bvh.h, small.h), pts):
            bits = torch.zeros((n, 3), dtype=torch.int32, device="cuda")
            cnt = torch.zeros(n, dtype=torch.int32, device="cuda")
            ctr = torch.zeros(4, dtype=torch.int64, device="cuda")
            rc.rc_batch_add_part(b, h, Q, M, bits, cnt, ctr)
            got += [bits, cnt, ctr]
        rc.rc_batch_launch(b)
        torch.cuda.synchronize()
        rc.rc_batch_destroy(b)
        out.append([g.cpu().numpy() for g in got])
    for k, (a, b) in enumerate(zip(*out)):
        if a.dtype == np.int64 and a.shape == (4,):          # rays, ambiguous, re-tests (differ), errors
            assert a[0] == b[0] == n * dirs and a[1] == b[1] and a[3] == b[3] == 0
        else:
            assert np.array_equal(a, b), k
    assert 0 < out[0][0].sum() and out[0][9].sum() > 0
    bvh.close()
    small.close()
