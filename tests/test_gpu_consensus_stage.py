"""Inlier counts and distance sums of given poses (lsr_stage_consensus) at odd
sizes, for host and device inputs, and for boxes of more cells than the grids
store, against a brute-force FP64 evaluation.
"""
import numpy as np
import pytest

gpu = pytest.mark.gpu
EPS = 0.0375


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
@pytest.mark.parametrize("n_p,n_q,poses", [(1, 1, 1), (33, 257, 3), (255, 31, 7), (2049, 1500, 5)])
@pytest.mark.parametrize("extent", [(0.0, 0.0, 0.0), (0.4, 0.3, 0.2), (200.0, 150.0, 100.0)])
@pytest.mark.parametrize("device", [False, True])
def test_consensus_against_brute_force(ctx, n_p, n_q, poses, extent, device):
    import torch
    from scipy.spatial.transform import Rotation
    rng = np.random.default_rng(n_p + n_q)
    Q = (rng.uniform(0, 1, (n_q, 3)) * extent).astype(np.float32)
    P = (Q[rng.integers(0, n_q, n_p)] + rng.normal(0, 0.02, (n_p, 3))).astype(np.float32)
    Rt = np.zeros((poses, 3, 4), np.float32)
    for k in range(poses):
        Rt[k, :, :3] = Rotation.from_rotvec(rng.normal(0, 1e-3 if k else 0.0, 3)).as_matrix()
        Rt[k, :, 3] = rng.normal(0, 0.02, 3) * (k % 3)
    args = (P, Q, Rt.reshape(-1, 12))
    if device:
        args = tuple(torch.from_numpy(x).cuda() for x in args)
    count, sumd2 = (np.asarray(x.cpu() if hasattr(x, "cpu") else x) for x in ctx.stage_consensus(*args, EPS))
    for k in range(poses):
        X = P.astype(np.float64) @ Rt[k, :, :3].T.astype(np.float64) + Rt[k, :, 3]
        d = np.sqrt(np.array([((Q.astype(np.float64) - x) ** 2).sum(1).min() for x in X]))
        tol = 4e-7 * (np.abs(X).max() + 1.0) * 3  # FP32 rounding of the moved coordinates
        near = int((np.abs(d - EPS) < tol).sum())
        assert abs(int(count[k]) - int((d < EPS).sum())) <= near
        ref = (d[d < EPS] ** 2).sum()
        assert abs(float(sumd2[k]) - ref) <= 2 * tol * EPS * n_p + near * EPS ** 2
