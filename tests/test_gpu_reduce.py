"""The directional reduction where its grouping and its fp32 sums can go
wrong: groups of one to 32 points, odd numbers of words, tables in shared
memory and not, points whose two largest sums tie or nearly tie, and the
per-direction sums at the edges of chunks and of groups of four points."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _run(bits, N, dirs, weight=None, **kw):
    import torch
    import paper_2609_05467_gb300 as rc
    n = len(bits)
    p = rc.rc_params_default(n_dirs=dirs, **kw)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    acc, conc = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    dom = torch.empty(n, dtype=torch.int8, device="cuda")
    area = torch.empty(dirs, dtype=torch.float64, device="cuda")
    s = rc.rc_direction_variability(t(bits.view(np.int32)), t(N), p, None if weight is None else t(weight), acc, dom, conc, area)
    return s, acc.cpu().numpy(), dom.cpu().numpy(), conc.cpu().numpy(), area.cpu().numpy()


def _rows(rng, n, dirs, share):
    v = rng.random((n, dirs)) < share[:, None]
    W = (dirs + 31) // 32
    pad = np.zeros((n, 32 * W), bool)
    pad[:, :dirs] = v
    return v, np.packbits(pad, axis=1, bitorder="little").view(np.uint32).copy()


def _normals(rng, n):
    N = rng.normal(size=(n, 3))
    N[: n // 3] = np.eye(3)[rng.integers(0, 3, n // 3)] * rng.choice([-1, 1], (n // 3, 1))   # ties of the other two axes
    return (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("conc_mode", [0, 1])
@pytest.mark.parametrize("n,dirs", [(1, 1), (1, 33), (33, 31), (5000, 64), (9800, 96), (39000, 40), (160001, 33), (300, 3072),
                                    (300, 3073), (40, 4100)])
def test_per_point_indicators(n, dirs, conc_mode):
    rng = np.random.default_rng(n + dirs)
    share = rng.choice([0.0, 0.02, 0.5, 0.97, 1.0], n)
    v, bits = _rows(rng, n, dirs, share)
    N = _normals(rng, n)
    weight = rng.random(n) + 0.25
    s, acc, dom, conc, area = _run(bits, N, dirs, weight, conc_mode=conc_mode)
    M, _, odom, oconc, cnt = oracle.variability(bits, N, dirs, conc_mode)
    assert np.array_equal(dom, odom)
    assert np.array_equal(acc, (cnt / np.float64(dirs)).astype(np.float32))
    assert np.array_equal(conc, np.asarray(oconc, np.float64).astype(np.float32))
    assert s.count_sum == v.sum() and s.n_counted == (cnt > 0).sum()
    assert list(s.dom_count) == [(odom == k).sum() for k in range(3)]
    # FP64 sums of n terms in any order: n u of the sum of their magnitudes at most
    assert np.allclose(area, (v * weight[:, None]).sum(0), rtol=n * 2.3e-16, atol=0)
    assert abs(s.weighted_count - (weight * cnt).sum()) <= n * 2.3e-16 * (weight * cnt).sum()


@pytest.mark.parametrize("n", [1, 3, 4, 511, 512, 513, 2050])
def test_unit_weight_sums_are_exact(n):
    rng = np.random.default_rng(n)
    v, bits = _rows(rng, n, 290, np.full(n, 0.6))
    *_, area = _run(bits, _normals(rng, n), 290)
    assert np.array_equal(area, v.sum(0).astype(np.float64))


def test_near_ties_take_the_exact_sums():
    """Visible sets mirrored in the plane x = y of the normal's frame leave two sums equal up to rounding."""
    import paper_2609_05467_gb300 as rc
    dirs = 256
    h = rc.rc_direction_table(dirs)
    rng = np.random.default_rng(0)
    n = 400
    N = np.tile(np.array([[0, 0, 1]], np.float32), (n, 1))
    v = np.zeros((n, dirs), bool)
    for k in range(n):
        a = rng.uniform(0, 2 * np.pi)
        v[k] = (np.abs(h[:, 0]) > 0.55) ^ (np.abs(h[:, 1]) > 0.55) if k % 2 else h[:, 0] * np.cos(a) + h[:, 1] * np.sin(a) > 0.4
    bits = np.packbits(v, axis=1, bitorder="little").view(np.uint32).copy()
    s, acc, dom, conc, _ = _run(bits, N, dirs)
    M, _, odom, oconc, cnt = oracle.variability(bits, N, dirs)
    assert np.array_equal(dom, odom) and np.array_equal(conc, np.asarray(oconc, np.float64).astype(np.float32))


@pytest.mark.parametrize("n,dirs", [(400_000, 1000), (40_000, 4000)])
def test_largest_components_are_rounded_as_stated(n, dirs):
    """Products and sums of a direction round one by one: a fused multiply-add in their place moves the largest component
    of about 1 direction in 10^8, so many points are needed to see it.  Counts: no tolerance."""
    rng = np.random.default_rng(dirs)
    N = rng.normal(size=(n, 3))
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    row = _rows(rng, 1, dirs, np.ones(1))[1]
    bits = np.repeat(row, n, axis=0)
    s, _, dom, conc, _ = _run(bits, N, dirs)
    _, ac, odom, oconc, _ = oracle.variability(bits, N, dirs, 0)
    assert np.array_equal(dom, odom)
    assert np.array_equal(conc, oconc.astype(np.float32))
    assert s.conc_sum_q == int(np.rint(oconc * 2.0 ** 40).astype(np.int64).sum())
