"""The pooled walk of the axis casts where it can go wrong: groups of fewer
than 32 points, warps with rays in some lanes only, long grazing walks, a
part of many overlapping boxes, and both kinds of grid.  Masks, travel and
the ray and ambiguity counters have to be those of the binary walk (a ray
per lane, world boxes), and the tool's masks likewise."""
import numpy as np
import pytest

import oracle
import synth
from common import gpu_mesh

pytestmark = pytest.mark.gpu

TURN = synth.rotation(12.0, -7.0, 25.0).astype(np.float32).reshape(-1)


def _casts(h, P, N, frame, **kw):
    import torch
    import paper_2609_05467_gb300 as rc
    n = len(P)
    P, N = (torch.from_numpy(np.ascontiguousarray(q, np.float32)).cuda() for q in (P, N))
    out = []
    for width in (0, 2):
        p = rc.rc_params_default(frame=frame, tree_width=width, **kw)
        mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
        tool = torch.zeros_like(mask)
        travel = torch.zeros((n, 6), device="cuda")
        ctr = torch.zeros((2, 4), dtype=torch.int64, device="cuda")
        rc.rc_orthogonal_cast(h, P, N, p, mask, travel, ctr[0])
        rc.rc_tool_cast(h, P, N, p, 2.5, 5, tool, ctr[1])
        out.append([q.cpu().numpy() for q in (mask, tool, travel, ctr)])
    a, b = out
    assert (a[3][:, 3] == 0).all() and (b[3][:, 3] == 0).all()
    assert (a[3][:, 0] == b[3][:, 0]).all()
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)
    return a


@pytest.mark.parametrize("n", [1, 31, 33, 500])
@pytest.mark.parametrize("frame", [np.eye(3).reshape(-1), TURN], ids=["identity", "turned"])
@pytest.mark.parametrize("launch_mode", [0, 1])
def test_masks_equal_binary_walk(n, frame, launch_mode):
    import paper_2609_05467_gb300 as rc
    V, F = synth.prismatic(h=4.0)
    if frame is TURN:
        V = synth.rotate(V, TURN.reshape(3, 3).astype(np.float64))
    bvh = rc.Bvh(*gpu_mesh(V, F))
    P, N, _, _ = oracle.sample_area(V, F, n, seed=n)
    a = _casts(bvh.h, P, N, frame, launch_mode=launch_mode)
    assert n < 500 or 0 < np.unpackbits(a[0]).sum() < a[3][0, 0]
    bvh.close()


def test_soup_with_few_casting_lanes():
    """Every box overlaps most others; two thirds of the points are eligible along no axis of a lane's neighbours."""
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(5)
    T, n = 4000, 97
    A = rng.uniform(0, 10, (T, 1, 3))
    V = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-12, 12, (T, 2, 3))], 1)).reshape(-1, 3).astype(np.float32)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    P = rng.uniform(0, 10, (n, 3)).astype(np.float32)
    N = np.eye(3, dtype=np.float32)[rng.integers(0, 3, n)] * rng.choice([-1, 1], (n, 1)).astype(np.float32)
    _casts(bvh.h, P, N, np.eye(3).reshape(-1), parallel_tol=0.0)
    bvh.close()
