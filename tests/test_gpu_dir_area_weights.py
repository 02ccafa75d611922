"""Per-direction weights where a chunk of points has equal weights and where
it has not: infinite ones reach only the directions that a point sees."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 512, 513, 1500])
@pytest.mark.parametrize("kind", ["equal", "one chunk", "mixed"])
def test_infinite_weights(n, kind):
    import paper_2609_05467_gb300 as rc
    dirs = 70
    rng = np.random.default_rng(n)
    seen = rng.random((n, dirs)) < 0.3
    seen[:, 5::7] = False                                    # directions nobody sees
    w = np.full(n, np.inf)
    if kind == "one chunk":
        w[512:] = 0.5
    if kind == "mixed":
        w[1::2] = rng.random(n)[1::2]
    row = np.zeros((n, 96), bool)
    row[:, :dirs] = seen
    bits = np.packbits(row, axis=1, bitorder="little").view(np.int32).copy()
    N = np.tile(np.array([0, 0, 1], np.float32), (n, 1))
    area = torch.empty(dirs, dtype=torch.float64, device="cuda")
    rc.rc_direction_variability(torch.from_numpy(bits).cuda(), torch.from_numpy(N).cuda(), rc.rc_params_default(n_dirs=dirs),
                                torch.from_numpy(w).cuda(), dir_area=area, summary=False)
    want = np.array([w[seen[:, j]].sum() for j in range(dirs)])
    got = area.cpu().numpy()
    assert not np.isnan(got).any()
    # sums of at most 1,500 positive terms in any order: relative 1,500 x 2^-53
    assert np.array_equal(np.isinf(got), np.isinf(want))
    fin = np.isfinite(want)
    assert np.all(np.abs(got[fin] - want[fin]) <= 1500 * 2.0 ** -53 * want[fin])
