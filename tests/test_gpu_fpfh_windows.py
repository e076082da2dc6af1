"""FPFH at the edges of its windows: cells of one point, of just under, exactly
and just over 32, 64 and 128 points, alone and beside neighbouring cells, with
invalid normals, and clouds whose cells share storage. Against the oracle on
the same FP32 inputs.
"""
import numpy as np
import pytest

import oracle

gpu = pytest.mark.gpu
R = 0.125


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    c = lsr.Context(0)
    yield c
    c.close()


@gpu
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 129, 200])
@pytest.mark.parametrize("where", ["cell", "two cells", "room", "wrapped"])
def test_fpfh_windows(ctx, n, where):
    rng = np.random.default_rng(n)
    P = rng.uniform(0.0, 0.99 * R, (n, 3))
    if where != "cell":  # the same population again in the next cell, less one point
        P = np.concatenate([P, rng.uniform(0.0, 0.99 * R, (max(n - 1, 1), 3)) + [R, 0.0, 0.0]])
    if where == "room":
        P = np.concatenate([P, rng.uniform(-0.5, 0.5, (400, 3))])
    if where == "wrapped":  # a box of far more cells than are stored
        P = np.concatenate([P, rng.uniform(-1.0, 1.0, (50, 3)) * [150.0, 120.0, 90.0]])
    P = (P + [0.3, -0.2, 1.1]).astype(np.float32)
    N = rng.normal(size=P.shape)
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    N[3::11] = 0.0  # invalid normals
    S = rng.uniform(0.0, 0.2, (len(P), 33)).astype(np.float32)
    F = ctx.stage_fpfh(P, N, S, R)
    ref = oracle.fpfh(P, N, S, R)
    D = np.linalg.norm(P[:, None].astype(np.float64) - P[None], axis=2)
    sure = ~((np.abs(D - R) < 1e-6).any(1))  # a neighbour at the radius: either way
    m = int((D < R).sum(1).max())
    # sums of m positive FP32 terms, each from a distance to 3 ulp, then three divisions
    assert np.abs(F - ref)[sure].max() <= (m + 16) * 2.0 ** -23
