"""Area sampling with few and with many points: the two forms of the kernel
give the same points, those of the oracle, bit for bit, also after a refit
that changes the total area, on parts of one and of many blocks of areas."""
import numpy as np
import pytest

import oracle
from common import gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T", [1, 4096, 4097, 70_000])
@pytest.mark.parametrize("exponent", [-138, 0, 60])
def test_points_of_both_forms(T, exponent):
    import paper_2609_05467_gb300 as rc
    line = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(T)
    A = rng.uniform(0, 10, (T, 1, 3))
    V = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-1, 1, (T, 2, 3))], 1)).reshape(-1, 3)
    F = np.arange(3 * T, dtype=np.int32).reshape(T, 3)
    V = np.ldexp(V, exponent).astype(np.float32)
    h = rc.rc_build_bvh(*gpu_mesh(V, F))
    for turn in range(2):
        for n in (1, line, line + 1):
            P, N = torch.zeros((n, 3), device="cuda"), torch.zeros((n, 3), device="cuda")
            f = torch.zeros(n, dtype=torch.int32, device="cuda")
            rc.rc_sample_points(h, n, rc.rc_params_default(seed=7 + turn), P, N, f)
            oP, oN, of, _ = oracle.sample_area(V, F, n, 7 + turn)
            assert np.array_equal(f.cpu().numpy(), of)
            assert np.array_equal(P.cpu().numpy().view(np.uint32), oP.view(np.uint32))
            assert np.array_equal(N.cpu().numpy().view(np.uint32), oN.view(np.uint32))
        V = (V * rng.uniform(0.5, 1.5, V.shape)).astype(np.float32)
        rc.rc_refit_bvh(h, torch.from_numpy(V).cuda())
    rc.rc_destroy_bvh(h)
