"""The build's block-wide parts at the sizes where they change hands: keys
sorted by one block or by many with 2, 4 or 8 keys a thread, boxes climbed
within a block and across blocks, equal Morton codes, and face data whose
quotients and conversions avoid FP64 at the ends of the fp32 range.  Trees
pass the index checks before and after a refit, and casts and samples equal
the oracle's (bits outside its ambiguous rays; samples bit for bit)."""
import numpy as np
import pytest

import oracle

from common import compare_bits, gpu_cast, gpu_mesh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _soup(T, size, seed, copies=1):
    """T random triangles in a box of 10 mm; with copies > 1 each is there that many times (equal sort keys)."""
    rng = np.random.default_rng(seed)
    k = -(-T // copies)
    A = rng.uniform(0, 10, (k, 1, 3))
    V = (A + np.concatenate([np.zeros((k, 1, 3)), rng.uniform(-size, size, (k, 2, 3))], 1)).reshape(-1, 3)
    F = np.arange(3 * k, dtype=np.int32).reshape(k, 3)
    return V.astype(np.float32), np.tile(F, (copies, 1))[:T].copy()


def _check(rc, h, V, F, seed):
    c = rc.rc_bvh_validate(h)
    assert c["nodes_seen"] >= 1 and sum(v for k, v in c.items() if k != "nodes_seen") == 0, c
    p = rc.rc_params_default(n_dirs=64, sample_mode=rc.RC_SAMPLE_AREA_RANDOM, seed=seed)
    P, Nn = torch.zeros((200, 3), device="cuda"), torch.zeros((200, 3), device="cuda")
    f = torch.zeros(200, dtype=torch.int32, device="cuda")
    rc.rc_sample_points(h, 200, p, P, Nn, f)
    oP, oN, of, _ = oracle.sample_area(V, F, 200, seed)
    assert np.array_equal(f.cpu().numpy(), of)
    assert np.array_equal(P.cpu().numpy().view(np.uint32), oP.view(np.uint32))
    assert np.array_equal(Nn.cpu().numpy().view(np.uint32), oN.view(np.uint32))
    return p, oP[:12], oN[:12]


def _cast_check(rc, h, V, F, p, P, Nn):
    mesh = oracle.Mesh(V, F)
    compare_bits(*gpu_cast(rc, h, P, Nn, p)[:2], *mesh.hemisphere(P, Nn, 64), 64)
    frame = [0.8, -0.6, 0, 0.6, 0.8, 0, 0, 0, 1]
    q = rc.rc_params_default(frame=frame)
    mask = torch.zeros(len(P), dtype=torch.uint8, device="cuda")
    trav = torch.zeros((len(P), 6), dtype=torch.float32, device="cuda")
    rc.rc_orthogonal_cast(h, torch.from_numpy(P).cuda(), torch.from_numpy(Nn).cuda(), q, mask, trav)
    om, oam = mesh.orthogonal(P, Nn, frame=frame)
    assert np.array_equal(mask.cpu().numpy() & ~oam, om & ~oam)


SMS = 152                    # the lines of the many-block sort: 2 and 4 keys a thread up to 1,024 and 2,048 keys an SM


@pytest.mark.parametrize("builder", [0, 1])
@pytest.mark.parametrize("T,copies", [(1, 1), (2, 1), (33, 1), (255, 1), (256, 1), (257, 1), (513, 300), (4095, 1), (4096, 9),
                                      (4097, 1), (2 * SMS * 512 + 1, 1), (2 * SMS * 1024 + 1, 70)])
def test_build_and_refit_at_the_edges(T, copies, builder):
    import paper_2609_05467_gb300 as rc
    if builder and (T > 5000 or copies > 1):
        pytest.skip("the sort is the same for both builders; coincident faces chain too deep in the merge tree")
    size = 3.0 if T < 1000 else 0.2
    V0, F = _soup(T, size, T, copies)
    h = rc.rc_build_bvh_ex(*gpu_mesh(V0, F), builder)
    _cast_check(rc, h, V0, F, *_check(rc, h, V0, F, 3))
    rng = np.random.default_rng(T + 1)
    V1 = (V0 * np.float32(1.5) + rng.uniform(-0.5, 0.5, V0.shape)).astype(np.float32)
    rc.rc_refit_bvh(h, torch.from_numpy(V1).cuda())
    _cast_check(rc, h, V1, F, *_check(rc, h, V1, F, 4))
    info = rc.rc_bvh_get_info(h)
    used = V1[F.reshape(-1)]
    assert np.allclose(info.scene_lo, used.min(0), atol=1e-5) and np.allclose(info.scene_hi, used.max(0), atol=1e-5)
    rc.rc_destroy_bvh(h)


@pytest.mark.parametrize("exponent", [-140, -100, -63, -50, -3, 40, 60])
def test_face_data_across_the_fp32_range(exponent):
    """Normals, areas and points of parts scaled by powers of two, with flat faces (zero and negative-zero components),
    slivers and faces without area."""
    import paper_2609_05467_gb300 as rc
    V, F = _soup(600, 3.0, 5)
    V[:300, 2] = 4.0                                            # normals along z
    V[300:600, 0] = -1.0
    V[3 * 250 + 2] = V[3 * 250 + 1]                             # no area
    V[3 * 400:3 * 500:3] = V[3 * 400 + 1:3 * 500 + 1:3] + np.float32(1e-6)
    V = np.ldexp(V, exponent).astype(np.float32)
    h = rc.rc_build_bvh(*gpu_mesh(V, F))
    _check(rc, h, V, F, 11)
    p = rc.rc_params_default(sample_mode=rc.RC_SAMPLE_FACE_CENTROID)
    P, Nn = torch.zeros((600, 3), device="cuda"), torch.zeros((600, 3), device="cuda")
    f = torch.zeros(600, dtype=torch.int32, device="cuda")
    w = torch.zeros(600, dtype=torch.float64, device="cuda")
    rc.rc_sample_points(h, 600, p, P, Nn, f, w)
    oP, oN, of, ow = oracle.sample_centroid(V, F)
    assert np.array_equal(Nn.cpu().numpy().view(np.uint32), oN.view(np.uint32))
    assert np.array_equal(P.cpu().numpy().view(np.uint32), oP.view(np.uint32))
    assert np.array_equal(w.cpu().numpy(), ow)
    rc.rc_destroy_bvh(h)
