"""Selection with hypotheses left out by groups of points far from Q: the
winner is one of the oracle's best hypotheses, with its count, and no hypothesis
that the oracle counts higher is missed; for an ordinary pair, a Q whose box is
too large for the coarse bit-set, a P whose normal grid shares storage so that
groups are wide, and clouds away from the origin.
"""
import numpy as np
import pytest

import oracle
from synth import make_pair

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("kind", ["plain", "far Q", "far P", "shifted"])
def test_far_groups_select_the_same(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    H, n = 60_000, 16_384  # (the smallest P that takes the groups)
    fp = make_pair(0, 0, n_p=n, n_q=n)
    P, Q, vpP, vpQ = fp.P, fp.Q, np.asarray(fp.vpP, np.float32), np.asarray(fp.vpQ, np.float32)
    far = (np.random.default_rng(n).uniform(-1, 1, (40, 3)) * [180.0, 150.0, 120.0]).astype(np.float32)
    if kind == "far Q":
        Q = np.concatenate([Q, far])
    if kind == "far P":
        P = np.concatenate([P, far])
    if kind == "shifted":
        P, Q, vpP, vpQ = (x + np.float32(s) for x, s in ((P, 4.0), (Q, -3.0), (vpP, 4.0), (vpQ, -3.0)))
    with lsr.Context(0, n_hypotheses=H, seed=fp.seed) as ctx:
        r = ctx.register_pair(P, Q, vpP, vpQ)
    ref = oracle.register(P, Q, vpP, vpQ, diag=True, seed=fp.seed, n_hypotheses=H)
    assert r.status == ref["status"] == 0
    mine = [t for t in ref["top"] if t["h"] == r.best_h]
    assert mine or ref["top"][0]["touch"]
    # counts of hypotheses whose descriptor matches FP32 may take otherwise are not compared
    for t in mine:
        assert t["touch"] or abs(r.hyp_inliers - t["count"]) <= t["amb"]
    for t in ref["top"]:
        assert t["touch"] or t["count"] - t["amb"] <= r.hyp_inliers
