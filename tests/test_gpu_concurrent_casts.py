"""Casts with different direction counts at the same time: the shared memory
that a kernel may have belongs to the kernel, so a launch that asks for much
of it must not fail because another thread's launch asked for less, nor a
batch because another was prepared after it."""
import threading

import numpy as np
import pytest

import synth
from common import gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _points(rc, h, n):
    P, N = torch.empty((n, 3), device="cuda"), torch.empty((n, 3), device="cuda")
    face = torch.empty(n, dtype=torch.int32, device="cuda")
    rc.rc_sample_points(h, n, rc.rc_params_default(), P, N, face)
    return P, N


def test_two_threads():
    import paper_2609_05467_gb300 as rc
    bvh = rc.Bvh(*gpu_mesh(*synth.pocket_block(1)))
    P, N = _points(rc, bvh.h, 3)
    torch.cuda.synchronize()
    errors, results = [], {}

    def work(dirs, width):
        try:
            p = rc.rc_params_default(n_dirs=dirs, tree_width=width)
            s = torch.cuda.Stream()
            bits = torch.empty((3, (dirs + 31) // 32), dtype=torch.int32, device="cuda")
            cnt = torch.empty(3, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for _ in range(400):
                rc.rc_hemisphere_cast(bvh.h, P, N, p, bits, cnt, stream=s)
            s.synchronize()
            results[dirs] = cnt.cpu().numpy()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in ((65536, 4), (16000, 4), (30000, 4))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for dirs, cnt in results.items():
        p = rc.rc_params_default(n_dirs=dirs, tree_width=2)
        bits = torch.empty((3, (dirs + 31) // 32), dtype=torch.int32, device="cuda")
        want = torch.empty(3, dtype=torch.int32, device="cuda")
        rc.rc_hemisphere_cast(bvh.h, P, N, p, bits, want)
        assert np.array_equal(want.cpu().numpy(), cnt)
    bvh.close()


def test_batches_prepared_one_after_the_other():
    import paper_2609_05467_gb300 as rc
    bvh = rc.Bvh(*gpu_mesh(*synth.pocket_block(1)))
    P, N = _points(rc, bvh.h, 5)
    sets = []
    for dirs in (65536, 16000, 40000, 256):
        W = (dirs + 31) // 32
        out = [(torch.zeros((5, W), dtype=torch.int32, device="cuda"), torch.zeros(5, dtype=torch.int32, device="cuda"))
               for _ in range(2)]
        b = rc.rc_batch_create(rc.rc_params_default(n_dirs=dirs))
        rc.rc_batch_add_part(b, bvh.h, P, N, *out[0])
        rc.rc_batch_launch(b)
        rc.rc_hemisphere_cast(bvh.h, P, N, rc.rc_params_default(n_dirs=dirs, tree_width=2), *out[1])
        sets.append((b, out))
    torch.cuda.synchronize()
    for b, out in sets + sets[::-1]:
        out[0][0].zero_()
        rc.rc_batch_launch(b)
        torch.cuda.synchronize()
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    for b, _ in sets:
        rc.rc_batch_destroy(b)
    bvh.close()
