"""The pooled walk of the hemispherical cast where it can go wrong: the
stack nearly full, the frontier with no room, points of one ray, tiles that
are padded, and the two widths of its pairs.  The bits have to be those of
the binary walk (tree_width 2, a ray per lane), which shares neither the
stack nor the triangle test, and the oracle's outside its ambiguous rays."""
import numpy as np
import pytest

import oracle
import synth
from common import compare_bits, gpu_cast, gpu_mesh

pytestmark = pytest.mark.gpu


def _both(h, P, N, dirs, **kw):
    import paper_2609_05467_gb300 as rc
    a = gpu_cast(rc, h, P, N, rc.rc_params_default(n_dirs=dirs, **kw))
    b = gpu_cast(rc, h, P, N, rc.rc_params_default(n_dirs=dirs, tree_width=2, **kw))
    for x in (a, b):
        assert x[2][3] == 0
        assert x[2][0] == len(P) * dirs
    # origins on the surface: the tangent-plane drops leave out pairs that the
    # binary walk counts as ambiguous (the bits are the same)
    if kw.get("origin_offset") != 0.0:
        assert a[2][1] == b[2][1]
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[0], b[0])
    return a


def _soup(T, size, seed):
    """T random triangles with edges up to `size` in a unit box of 10 mm: with large ones every box meets most others."""
    rng = np.random.default_rng(seed)
    A = rng.uniform(0, 10, (T, 1, 3))
    V = (A + np.concatenate([np.zeros((T, 1, 3)), rng.uniform(-size, size, (T, 2, 3))], 1)).reshape(-1, 3)
    return V.astype(np.float32), np.arange(3 * T, dtype=np.int32).reshape(T, 3)


@pytest.mark.parametrize("T,size,n,dirs", [(4000, 12.0, 40, 256), (4000, 0.3, 64, 512), (40, 12.0, 33, 97), (3, 5.0, 5, 33)])
def test_soup_equals_binary_walk_and_oracle(T, size, n, dirs):
    import paper_2609_05467_gb300 as rc
    V, F = _soup(T, size, T + dirs)
    rng = np.random.default_rng(7)
    P = rng.uniform(0, 10, (n, 3)).astype(np.float32)
    N = rng.normal(size=(n, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    g = _both(bvh.h, P, N, dirs)
    ob, oa, oc = oracle.Mesh(V, F).hemisphere(P, N, dirs)
    compare_bits(g[0], g[1], ob, oa, oc, dirs)
    bvh.close()


@pytest.mark.parametrize("dirs", [1, 31, 32, 33, 64, 257, 2100])
@pytest.mark.parametrize("launch_mode", [0, 1])
def test_ragged_directions_on_a_fan(dirs, launch_mode):
    """Points at the tip of a fan of slivers: every sliver's box holds the point, more than the frontier has room for."""
    import paper_2609_05467_gb300 as rc
    k = 150
    a = np.linspace(0, 2 * np.pi, k, endpoint=False)
    ring = np.stack([20 * np.cos(a), 20 * np.sin(a), 6 + 3 * np.cos(5 * a)], 1)
    V = np.concatenate([[[0, 0, 0]], ring]).astype(np.float32)
    F = np.stack([np.zeros(k), 1 + np.arange(k), 1 + (np.arange(k) + 1) % k], 1).astype(np.int32)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    P = np.array([[0, 0, 0], [0.01, 0, 0.004], [0, 0, 1], [5, 5, 2]], np.float32)
    N = np.array([[0, 0, 1], [0, 0, 1], [1, 0, 0], [0, 0, -1]], np.float32)
    g = _both(bvh.h, P, N, dirs, launch_mode=launch_mode)
    ob, oa, oc = oracle.Mesh(V, F).hemisphere(P, N, dirs)
    compare_bits(g[0], g[1], ob, oa, oc, dirs)
    bvh.close()


@pytest.mark.parametrize("builder", [0, 1])
def test_part_options_equal_binary_walk(builder):
    import paper_2609_05467_gb300 as rc
    V, F = synth.prismatic(h=5.0)
    bvh = rc.Bvh(*gpu_mesh(V, F), builder=builder)
    P, N, _, _ = oracle.sample_area(V, F, 301, seed=3)
    for kw in (dict(), dict(point_order=1), dict(tile_mode=1), dict(launch_mode=1), dict(origin_offset=0.0)):
        _both(bvh.h, P, N, 150, **kw)
    _both(bvh.h, P, (N * np.float32(1.7)).astype(np.float32), 150)
    bvh.close()


@pytest.mark.parametrize("rows", [2048, 2049])
def test_pair_width_at_its_line(rows):
    """2^24 triangles still use 32-bit pairs, one row more of the grid 64-bit ones."""
    import torch
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
    n, dirs = 500, 96
    p = rc.rc_params_default(n_dirs=dirs)
    P = torch.empty((n, 3), device="cuda")
    N = torch.empty_like(P)
    face = torch.empty(n, dtype=torch.int32, device="cuda")
    rc.rc_sample_points(bvh.h, n, p, P, N, face)
    g = _both(bvh.h, P.cpu().numpy(), N.cpu().numpy(), dirs)
    assert 0.2 < g[1].mean() / dirs < 0.95
    bvh.close()


def test_batch_of_mixed_parts_equals_single_casts():
    import torch
    import paper_2609_05467_gb300 as rc
    p = rc.rc_params_default(n_dirs=257)
    b = rc.rc_batch_create(p)
    parts = []
    for V, F in (synth.pocket_block(1), synth.prismatic(h=6.0), _soup(4000, 12.0, 1)):
        bvh = rc.Bvh(*gpu_mesh(V, F))
        n = 70
        P = torch.empty((n, 3), device="cuda")
        N = torch.empty_like(P)
        face = torch.empty(n, dtype=torch.int32, device="cuda")
        rc.rc_sample_points(bvh.h, n, p, P, N, face)
        out = [(torch.zeros((n, 9), dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"))
               for _ in range(2)]
        rc.rc_batch_add_part(b, bvh.h, P, N, *out[0])
        rc.rc_hemisphere_cast(bvh.h, P, N, rc.rc_params_default(n_dirs=257, tree_width=2), *out[1])
        parts.append((bvh, P, N, out))
    rc.rc_batch_launch(b)
    torch.cuda.synchronize()
    for bvh, _, _, out in parts:
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        bvh.close()
    rc.rc_batch_destroy(b)


@pytest.mark.parametrize("n,dirs", [(1, 33), (1, 2048), (5, 257), (37, 1000), (200, 2048), (1500, 96), (1600, 96)])
def test_few_points_in_parts_equal_the_same_points_among_many(n, dirs):
    """Few points are cast in parts of a tile or more: their rows and counts are those they get in a large set."""
    import paper_2609_05467_gb300 as rc
    V, F = _soup(3000, 1.0, n)
    rng = np.random.default_rng(dirs)
    P = rng.uniform(0, 10, (8000, 3)).astype(np.float32)
    N = rng.normal(size=(8000, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    p = rc.rc_params_default(n_dirs=dirs)
    many, few = gpu_cast(rc, bvh.h, P, N, p), gpu_cast(rc, bvh.h, P[:n], N[:n], p)
    assert np.array_equal(many[0][:n], few[0]) and np.array_equal(many[1][:n], few[1])
    assert few[2][0] == n * dirs
    bvh.close()


@pytest.mark.parametrize("dirs", [33, 600, 2048])
def test_normals_at_the_gate_of_the_tangent_shortcuts(dirs):
    """Normals whose squared length differs from one by the bound of the tangent shortcuts, a little less and a little more:
    bits equal the binary walk's and the oracle's, also for points on the surface and on its vertices."""
    import paper_2609_05467_gb300 as rc
    V, F = synth.icosphere(10.0, 2)
    V = np.concatenate([V, 0.6 * V]).astype(np.float32)
    F = np.concatenate([F, F[:, ::-1] + len(V) // 2]).astype(np.int32)
    gate = 0.25 * (1.0 / (64.0 * ((dirs + 31) // 32)) - 2e-6)
    P, N, _, _ = oracle.sample_centroid(V, F)
    rng = np.random.default_rng(dirs)
    pick = rng.choice(len(P), 120, replace=False)
    P, N = P[pick], N[pick].astype(np.float64)
    P[::3] = V[F[pick[::3], 0]]                              # on a vertex: planes through the origin's neighbourhood
    d = gate * rng.choice([-1, 1], 120) * (1.0 + rng.choice([-1e-2, -1e-4, 0.0, 1e-4, 1e-2], 120))
    N = (N * np.sqrt(1.0 + d)[:, None]).astype(np.float32)
    bvh = rc.Bvh(*gpu_mesh(V, F))
    g = _both(bvh.h, P, N, dirs)
    ob, oa, oc = oracle.Mesh(V, F).hemisphere(P, N, dirs)
    compare_bits(g[0], g[1], ob, oa, oc, dirs)
    bvh.close()
