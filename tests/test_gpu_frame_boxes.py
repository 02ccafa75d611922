"""Vertex boxes in turned frames and the cells of face normals at the edges of
their blocks: fewer vertices than a warp's or a block's share, one more and
one less, far from the origin, with vertices that tie for the extreme, with
unreferenced vertices; normals along axes, on cell edges and spread over all
cells.  Candidate frames and volumes equal the oracle's exactly."""
import numpy as np
import pytest

from common import gpu_mesh
from oracle import frames as ofr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nV,offset,grid", [(3, 0.0, 0.0), (255, 0.0, 0.0), (257, 1e4, 0.0), (2047, -300.0, 0.0), (2048, 0.0, 0.5),
                                            (2049, 1e6, 0.25), (6001, 0.0, 2.0), (21000, 50.0, 0.0)])
def test_candidates_at_the_edges(nV, offset, grid):
    import paper_2609_05467_gb300 as rc
    rng = np.random.default_rng(nV)
    V = rng.uniform(-10, 10, (nV, 3))
    if grid:
        V = np.round(V / grid) * grid                       # many vertices tie for an extreme; normals on cell edges
    V = (V + offset).astype(np.float32)
    T = max(1, nV // 4)
    F = rng.integers(0, nV, (T, 3)).astype(np.int32)
    F[0] = [0, 1, 2]
    bvh = rc.Bvh(*gpu_mesh(V, F))
    fr = rc.rc_frame_candidates(bvh.h, rc.rc_params_default())
    cands = ofr.frame_candidates(V, F)
    assert fr.k == len(cands)
    for c, cand in enumerate(cands):
        assert fr.source[c] == cand["source"]
        assert (fr.box_axis[c], fr.box_step[c]) == (cand["box_axis"], cand["box_step"])
        assert np.array_equal(fr.frame_array(c).view(np.uint32), cand["frame"].view(np.uint32)), c
        assert fr.volume[c] == cand["volume"]
    bvh.close()
