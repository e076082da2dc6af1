"""Grids of many thousand cells along an axis without wrapped storage (a map of
hundreds of metres at a radius of a few centimetres). The FP32 rounding of cell
coordinates grows with their number, and the searches leave out cells by a
distance taken from those coordinates: every query here has its nearest point
just behind a face of its cell, in the next row of cells, and a second one in
its own row farther off by 1e-5 m, which is what a search finds that leaves
that cell out. (With a margin of 2e-4 cells whatever the box, 3% of these
queries found the second at 1 km and 12% at 4 km.)
"""
import numpy as np
import pytest

gpu = pytest.mark.gpu
f32 = np.float32
EPS = f32(0.0375)


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    c = lsr.Context(0)
    yield c
    c.close()


def _last_below(coord, lo, hi, face):
    """Per element: the largest float of [lo, hi) whose cell coordinate is below face."""
    lo, hi = lo.copy(), hi.copy()
    for _ in range(60):
        mid = ((lo.astype(np.float64) + hi) / 2).astype(f32)
        below = coord(mid) < face
        lo, hi = np.where(below, mid, lo), np.where(below, hi, mid)
    return lo


def _scene(length, n, rng):
    """(Q, X, per query its nearest point's index and squared distance)."""
    ends = np.array([-length / 2 + 3e-4, length / 2], f32)
    ext = ends[1] - ends[0]
    cell = EPS * (f32(1) + max(f32(1e-4), f32(8 * 5.9604645e-8) * ext / EPS))
    inv = f32(1) / cell
    coord = lambda v: (v - ends[0]) * inv  # as the grid computes it
    # queries 5 cells apart about the middle, where a float is much finer than a cell coordinate
    site = ((np.arange(n) - n / 2) * 5 * float(cell)).astype(f32)
    face = np.floor(coord(site))
    behind = _last_below(coord, site - f32(1.2) * cell, site, face)
    x = (behind.astype(np.float64) + rng.uniform(0.3, 0.9, n) * float(EPS)).astype(f32)
    keep = np.floor(coord(x)) == face
    behind, x = behind[keep], x[keep]
    y_below = _last_below(lambda v: v * inv, np.full(1, 0.5, f32) * cell, np.full(1, 1.5, f32) * cell, f32(1))[0]
    y = np.nextafter(y_below, f32(1))  # the first float of the next row
    m, o = len(x), np.zeros(len(x), f32)
    X = np.stack([x, o + y_below, o], 1)
    near = np.stack([behind, o + y, o], 1)
    d2 = ((near.astype(np.float64) - X) ** 2).sum(1)
    second = X.copy()
    second[:, 2] = (np.sqrt(d2) + 1e-5).astype(f32)
    Q = np.concatenate([second, near, np.array([[ends[0], 0, 0], [ends[1], 1.5 * cell, 0]], f32)]).astype(f32)
    return Q, X, np.arange(m, 2 * m), d2


@gpu
@pytest.mark.parametrize("length", [10.0, 200.0, 1000.0, 4000.0])
def test_nearest_point_behind_a_face(ctx, length):
    Q, X, ref, d2 = _scene(length, min(4000, int(length * 4)), np.random.default_rng(int(length)))
    nn, got = ctx.stage_nn(Q, X, float(EPS))
    assert np.array_equal(nn, ref)
    assert np.abs(got - d2).max() <= 4e-7 * float(EPS) ** 2  # FP32 squares and sums


@gpu
@pytest.mark.parametrize("length", [10.0, 200.0, 1000.0, 4000.0])
def test_consensus_sums_of_a_long_box(ctx, length):
    Q, X, ref, d2 = _scene(length, min(4000, int(length * 4)), np.random.default_rng(int(length)))
    count, total = ctx.stage_consensus(X, Q, np.eye(4)[None, :3].reshape(1, 12).astype(f32), float(EPS))
    assert count[0] == len(X)
    assert abs(total[0] - d2.sum()) <= len(X) * (4e-7 * float(EPS) ** 2 + 2.0 ** -40)


@gpu
@pytest.mark.parametrize("length", [10.0, 200.0, 1000.0, 4000.0])
def test_objective_gradient_reaches_the_nearest_point(ctx, length):
    """The gradient of a pair's objective is scattered to the neighbours' rows."""
    import torch
    Q, X, ref, d2 = _scene(length, min(4000, int(length * 4)), np.random.default_rng(int(length)))
    P, Qd = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda()
    dP, dQ = torch.zeros_like(P), torch.zeros_like(Qd)
    ctx.objective_bwd([P], [Qd], np.zeros((1, 6)), np.eye(4)[None], np.ones(1), [dP], [dQ], float(EPS))
    dQ = dQ.cpu().numpy()
    other = np.ones(len(Q), bool)
    other[ref] = False
    assert not dQ[other].any() and np.abs(dQ[ref]).sum(1).all()
