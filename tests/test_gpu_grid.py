"""The uniform grid of eq. (1) at the edges of its build: cells, scan tiles and
storage. The exact nearest neighbours found through the grid (lsr_stage_nn)
equal a brute-force search with the same FP32 distances, ties to the smaller
index, for one cell, one point per cell, scans that end just before and after
a tile of 2048 cells, and boxes of more cells than the storage holds (wrapped).
"""
import numpy as np
import pytest

gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    c = lsr.Context(0)
    yield c
    c.close()


def _brute(Q, X, r):
    nn, d2 = np.full(len(X), -1, np.int64), np.full(len(X), np.inf)
    for i, x in enumerate(X):
        d = ((Q.astype(np.float64) - x.astype(np.float64)) ** 2).sum(1)
        j = int(d.argmin())
        if d[j] < float(np.float32(r)) ** 2:
            nn[i], d2[i] = j, d[j]
    return nn, d2


@gpu
@pytest.mark.parametrize("n", [1, 2, 33, 2047, 2049, 5003])
@pytest.mark.parametrize("extent", [(0.0, 0.0, 0.0), (0.3, 0.3, 0.3), (2047 * 0.05, 0.0, 0.0), (2049 * 0.05, 0.02, 0.0),
                                    (4.0, 3.5, 1.5), (300.0, 200.0, 90.0)])
def test_grid_search_equals_brute_force(ctx, n, extent):
    rng = np.random.default_rng(n + int(10 * sum(extent)))
    r = 0.05
    Q = (rng.uniform(0, 1, (n, 3)) * extent + [-1.0, 2.0, 0.5]).astype(np.float32)
    if n > 2:
        Q[n // 2:n // 2 + n // 8] = Q[:n // 8]  # duplicates: ties
    X = (Q[rng.integers(0, n, 300)] + rng.normal(0, 0.02, (300, 3))).astype(np.float32)
    X[:5] += 3.0  # some far away
    nn, d2 = ctx.stage_nn(Q, X, r)
    ref, rd2 = _brute(Q, X, r)
    near = np.abs(np.sqrt(np.where(np.isfinite(rd2), rd2, 0.0)) - r) < 1e-6  # at the radius: either way
    ok = near | (nn == ref)
    # another index only at a distance that FP32 cannot tell from the smallest
    for i in np.nonzero(~ok)[0]:
        assert nn[i] >= 0 and ref[i] >= 0
        d = ((Q[nn[i]].astype(np.float64) - X[i]) ** 2).sum()
        assert abs(np.sqrt(d) - np.sqrt(rd2[i])) < 1e-5
        assert not np.array_equal(Q[nn[i]], Q[ref[i]])  # a tie goes to the smaller index
    hit = (ref >= 0) & (nn >= 0)
    assert np.abs(np.sqrt(d2[hit]) - np.sqrt(rd2[hit])).max(initial=0.0) < 1e-5
