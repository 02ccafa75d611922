"""Axis rays at the ends of fp32's range: parts whose coordinates have squares
beyond it, frames whose columns take the coordinates beyond it or are very
short.  Masks equal the oracle's outside its ambiguous rays, and a walk visits
a small share of the tree, not all of it."""
import numpy as np
import pytest

import oracle
import synth
from common import gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TURN = synth.rotation(12.0, -7.0, 25.0).astype(np.float32)


@pytest.mark.parametrize("part,column", [(1.0, 1e37), (1.0, 1e38), (1.0, 1e-30), (1.0, 1e-37), (1e17, 1.0), (1e23, 1.0), (1e30, 1.0),
                                         (1e30, 1e10), (1e-30, 1.0)])
def test_masks_and_visits(part, column):
    import paper_2609_05467_gb300 as rc
    V, F = synth.prismatic(h=4.0)
    V = (V * np.float32(part)).astype(np.float32)
    frame = TURN.copy()
    frame[:, 1] = (TURN[:, 1].astype(np.float64) * column).astype(np.float32)
    n = 300
    P, N, _, _ = oracle.sample_area(V, F, n, seed=3)
    eps = 1e-4 * max(1.0, part)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    p = rc.rc_params_default(frame=frame.reshape(-1), origin_offset=eps, collect_stats=1)
    mask = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ctr = torch.zeros(8, dtype=torch.int64, device="cuda")
    rc.rc_orthogonal_cast(bvh.h, torch.from_numpy(P).cuda(), torch.from_numpy(N).cuda(), p, mask, torch.zeros((n, 6), device="cuda"), ctr)
    om, oam = oracle.Mesh(V, F).orthogonal(P, N, frame=frame.reshape(-1), eps=eps)
    got, ctr = mask.cpu().numpy(), ctr.cpu().numpy()
    assert np.array_equal(got & ~oam, om & ~oam)
    assert ctr[3] == 0 and ctr[0] > 0
    if part >= 1.0 and column == 1.0:
        # a ray's band is a line but for its drift: nodes of the whole tree, a few times the square root of their number
        assert ctr[4] / ctr[0] < 8 * np.sqrt(len(F))
    bvh.close()
