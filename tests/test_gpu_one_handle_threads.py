"""Threads that cast from one handle with different direction counts: each
cast walks the direction table of its own count."""
import threading

import numpy as np
import pytest

import synth
from common import gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_threads_with_their_own_direction_counts():
    import paper_2609_05467_gb300 as rc
    bvh = rc.Bvh(*gpu_mesh(*synth.pocket_block(1)))
    P, N = torch.empty((40, 3), device="cuda"), torch.empty((40, 3), device="cuda")
    face = torch.empty(40, dtype=torch.int32, device="cuda")
    rc.rc_sample_points(bvh.h, 40, rc.rc_params_default(), P, N, face)
    torch.cuda.synchronize()
    kinds = [(32, 0), (257, 0), (1024, 0), (4096, 0), (1024, 1)]

    def cast(dirs, mode, stream, times):
        p = rc.rc_params_default(n_dirs=dirs, tile_mode=mode)
        bits = torch.empty((times, 40, (dirs + 31) // 32), dtype=torch.int32, device="cuda")
        cnt = torch.empty((times, 40), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for k in range(times):
            rc.rc_hemisphere_cast(bvh.h, P, N, p, bits[k], cnt[k], stream=stream)
        stream.synchronize()
        return bits.cpu().numpy(), cnt.cpu().numpy()

    want = [cast(*k, torch.cuda.current_stream(), 1) for k in kinds]
    got = [None] * len(kinds)

    def work(q):
        got[q] = cast(*kinds[q], torch.cuda.Stream(), 200)

    threads = [threading.Thread(target=work, args=(q,)) for q in range(len(kinds))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, g in zip(want, got):
        assert g is not None
        assert (g[0] == w[0]).all() and (g[1] == w[1]).all()
    bvh.close()
