"""The objective of several pairs at once: pairs go through every step
together, eight at a time, so batches around that number and of very uneven
sizes (one point to thousands) must give what single-pair calls give. Sums are
FP64 in a fixed order per pair and do not depend on the batch: energies and
pose gradients equal bit for bit; dP is written once per point, so equal too;
dQ adds FP32 atomics in any order (a point closes at most a few pairs): 1e-6.
"""
import numpy as np
import pytest

gpu = pytest.mark.gpu
EPS = 0.0375


@gpu
@pytest.mark.parametrize("sizes", [[(1, 1)], [(5, 4), (3000, 1), (1, 2500), (127, 129)],
                                   [(64 * k + 1, 97 * k + 3) for k in range(8)],
                                   [(33 * k + 7, 511 + k) for k in range(19)]])
def test_objective_batches_equal_single_pairs(sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    rng = np.random.default_rng(len(sizes))
    P, Q = [], []
    for a, b in sizes:
        q = rng.uniform(0, 0.4, (b, 3))
        p = q[rng.integers(0, b, a)] + rng.normal(0, 0.01, (a, 3))
        p[::5] += 2.0  # no neighbour
        P.append(torch.from_numpy(p.astype(np.float32)).cuda())
        Q.append(torch.from_numpy(q.astype(np.float32)).cuda())
    n = len(sizes)
    xi = rng.normal(0, 2e-3, (n, 6))
    T0 = np.tile(np.eye(4), (n, 1, 1))
    dE = rng.uniform(0.5, 2.0, n)
    with lsr.Context(0) as ctx:
        def bwd(i):
            dP = [torch.full_like(P[k], 7.0) for k in i]
            dQ = [torch.full_like(Q[k], 7.0) for k in i]
            dx = ctx.objective_bwd([P[k] for k in i], [Q[k] for k in i], xi[i], T0[i], dE[i], dP, dQ, EPS)
            return dx, dP, dQ
        E = ctx.objective_fwd(P, Q, xi, T0, EPS)
        dxi, dP, dQ = bwd(list(range(n)))
        assert np.isfinite(E).all()
        for k in range(n):
            assert ctx.objective_fwd(P[k:k + 1], Q[k:k + 1], xi[k:k + 1], T0[k:k + 1], EPS)[0] == E[k]
            dx1, dP1, dQ1 = bwd([k])
            assert np.array_equal(dx1[0], dxi[k])
            assert torch.equal(dP1[0], dP[k])
            assert torch.allclose(dQ1[0], dQ[k], rtol=1e-6, atol=1e-6 * float(dQ[k].abs().max()) + 1e-12)


@gpu
@pytest.mark.parametrize("n", [1, 3, 8, 9])
def test_objective_in_a_workspace_that_just_suffices(n):
    """The largest pair that an earlier call's workspace still holds: its plan
    ends inside that workspace (a plan that does not is refused), and the
    energy is that of a workspace of its own."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    rng = np.random.default_rng(n)
    q = torch.from_numpy(rng.uniform(0, 0.4, (500, 3)).astype(np.float32)).cuda()
    big = torch.from_numpy(rng.uniform(0, 0.4, (4_000_000, 3)).astype(np.float32)).cuda()
    last = min(n, 8) - 1  # the last pair of a full chunk grows
    xi, T0 = np.zeros((n, 6)), np.tile(np.eye(4), (n, 1, 1))

    def clouds(points):
        return [big[:points if k == last else 1000] for k in range(n)], [q] * n

    def held(points):
        """(whether the workspace of 1000 points held this many, the energies)"""
        with lsr.Context(0) as ctx:
            ctx.objective_fwd(*clouds(1000), xi, T0, EPS)
            had = ctx.workspace_bytes()
            E = ctx.objective_fwd(*clouds(points), xi, T0, EPS)
            return ctx.workspace_bytes() == had, E

    lo, hi = 1000, len(big)
    assert held(lo)[0] and not held(hi)[0]
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if held(mid)[0]:
            lo = mid
        else:
            hi = mid
    for points in (lo, lo - 1, lo - 13, lo - 50):
        same, E = held(points)
        assert same
        with lsr.Context(0) as ctx:
            assert np.array_equal(E, ctx.objective_fwd(*clouds(points), xi, T0, EPS))
