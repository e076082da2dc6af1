"""The tensor-core matcher over listed tiles (from 2^29 pairs of rows on the
database tiles within a unit's reach are listed from the descriptor order, and
queries without a certificate are searched through the boxes) at the edges of
its units, tiles and items of 64 tiles, with both tile shapes and operand
layouts: the hook LSR_INJECT_MATCH_LIST takes that path at any size. It has to
return the FP32 matcher's indices and distance bits (tests/test_gpu_match_window.py
holds that one against the oracle), for ragged sizes, ties, near-duplicates,
identical rows, queries far outside, and rows that are no finite numbers. Larger
sets that take it (and the FP32 matcher's blocks of 32 tiles) by their size are
held against 64 bits.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

gpu = pytest.mark.gpu
D = 33
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", params=[1, 2], ids=["tile1", "tile2"])
def ctx(request):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    c = lsr.Context(0, match_tile=request.param)
    yield c
    c.close()


def fpfh_like(n, rng):
    g = rng.gamma(0.35, 1.0, size=(n, 3, 11))
    g /= g.sum(2, keepdims=True)
    return g.reshape(n, D).astype(np.float32)


def smooth(n, rng, m=40):
    """Rows near a surface of few dimensions, as descriptors of a scene are."""
    base = fpfh_like(m, rng)
    w = rng.dirichlet(np.full(m, 0.08), n)
    return (w @ base + 2e-3 * rng.standard_normal((n, D))).astype(np.float32)


def listed_equals_fp32(ctx, A, B, precision):
    import paper_1801_01572_gb300 as lsr
    nn32, d32, _ = ctx.stage_match(A, B, precision=0)
    ctx.stage_match(A, B, precision=precision)
    k0 = lsr.launch_count()
    ctx.stage_match(A, B, precision=precision)
    k1 = lsr.launch_count()
    ctx.debug_inject(lsr.INJECT_MATCH_LIST, 1)
    nn, d, fb = ctx.stage_match(A, B, precision=precision)
    if len(A) * len(B) < 2 ** 29:
        assert lsr.launch_count() - k1 > k1 - k0  # the order's launches: the list was taken
    assert np.array_equal(nn, nn32)
    assert np.array_equal(d.view(np.uint32), d32.view(np.uint32))
    return nn, d, fb


@gpu
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("nP,nQ", [(1, 1), (1, 9), (255, 129), (257, 257), (130, 385), (513, 127), (129, 8191),
                                   (129, 8193), (385, 16385), (1000, 3001), (3000, 1000)])
def test_listed_sizes(ctx, nP, nQ, precision):
    rng = np.random.default_rng(nP + 17 * nQ)
    listed_equals_fp32(ctx, fpfh_like(nP, rng), fpfh_like(nQ, rng), precision)
    listed_equals_fp32(ctx, smooth(nP, rng), smooth(nQ, rng), precision)


@gpu
@pytest.mark.parametrize("precision", [1, 2])
def test_listed_ties_and_near_duplicates(ctx, precision):
    """Duplicates thousands of rows apart, pairs 1e-6 apart, and clusters of 12
    rows within 1e-7, over three items."""
    rng = np.random.default_rng(5)
    B = smooth(20000, rng)
    B[15000:15100] = B[100:200]
    B[16000:16100] = B[200:300] + np.float32(1e-6)
    for c in range(20):
        B[17000 + c:17000 + c + 64 * 12:64] = B[300 + c] + 1e-7 * rng.random((12, D), dtype=np.float32)
    A = np.concatenate([B[15000:15100], B[200:300] + np.float32(3e-7), B[300:320] + np.float32(2e-7),
                        smooth(500, rng)])
    nn, d, _ = listed_equals_fp32(ctx, A, B, precision)
    assert np.array_equal(nn[:100], np.arange(100, 200)) and not d[:100].any()


@gpu
@pytest.mark.parametrize("precision", [1, 2])
def test_listed_search_of_every_query(ctx, precision):
    """Identical rows (all projections equal) in more chunks than are kept: no
    query has a certificate, all go through the boxes, the first row wins; and
    a cluster of them among others."""
    rng = np.random.default_rng(6)
    one = fpfh_like(1, rng)
    for n in (700, 9000):
        B = np.repeat(one, n, axis=0)
        A = fpfh_like(400, rng)
        nn, d, fb = listed_equals_fp32(ctx, A, B, precision)
        assert not nn.any() and fb == len(A)
        nn, d, fb = listed_equals_fp32(ctx, B[:300], B, precision)
        assert not nn.any() and not d.any() and fb == 300
    B = np.concatenate([smooth(5000, rng), np.repeat(one, 3000, axis=0), smooth(5000, rng)])
    A = np.concatenate([smooth(700, rng), one + (1e-4 * rng.standard_normal((333, D))).astype(np.float32)])
    nn, d, fb = listed_equals_fp32(ctx, A, B, precision)
    assert np.all(nn[700:] == 5000) and fb >= 333


@gpu
@pytest.mark.parametrize("precision", [1, 2])
def test_listed_far_queries_and_scales(ctx, precision):
    rng = np.random.default_rng(3)
    B = np.concatenate([smooth(9000, rng), 1e-20 * fpfh_like(200, rng)])
    A = np.concatenate([smooth(300, rng), 5 * fpfh_like(100, rng), -3 * fpfh_like(100, rng),
                        np.full((20, D), 40, np.float32), np.zeros((40, D), np.float32), 1e6 * fpfh_like(30, rng),
                        1e-19 * fpfh_like(50, rng)]).astype(np.float32)
    listed_equals_fp32(ctx, A, B.astype(np.float32), precision)


@gpu
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 3e38])
@pytest.mark.parametrize("where", ["queries", "sampled rows", "other rows", "all queries"])
def test_listed_rows_that_are_no_numbers(ctx, precision, bad, where):
    rng = np.random.default_rng(8)
    A, B = smooth(700, rng), smooth(9001, rng)  # every fourth row is sampled for the centre
    if where == "queries":
        A[[0, 131, 699], [0, 32, 16]] = bad
    elif where == "all queries":
        A[:, 5] = bad
    else:
        B[[4, 4000, 8000] if where == "sampled rows" else [1, 4001, 8999], [0, 32, 16]] = bad
    nn, d, fb = listed_equals_fp32(ctx, A, B, precision)
    if where == "queries":
        ok = np.ones(700, bool)
        ok[[0, 131, 699]] = False
        assert np.all(nn[~ok] == -1) and np.all(nn[ok] >= 0)
    elif where == "all queries":
        assert np.all(nn == -1)
    else:
        assert np.all(nn >= 0) and not np.isin(nn, [1, 4, 4000, 4001, 8000, 8999]).any()


@gpu
def test_listed_stall_times_out_and_context_recovers(ctx):
    import paper_1801_01572_gb300 as lsr
    rng = np.random.default_rng(9)
    A, B = smooth(600, rng), smooth(9000, rng)
    want = ctx.stage_match(A, B, precision=0)
    ctx.debug_inject(lsr.INJECT_MATCH_LIST, 1)
    ctx.debug_inject(lsr.INJECT_MATCH_STALL, 1)
    with pytest.raises(lsr.LsrError) as e:
        ctx.stage_match(A, B, precision=1)
    assert e.value.code == lsr.LSR_E_TIMEOUT
    ctx.debug_inject(lsr.INJECT_MATCH_LIST, 1)
    got = ctx.stage_match(A, B, precision=1)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@gpu
@pytest.mark.parametrize("nP,nQ", [(24001, 23001), (700, 800_001), (800_001, 700), (31000, 31007)])
def test_listed_by_size(ctx, nP, nQ):
    """Sets above the threshold, uneven ones among them, with duplicates across
    items; some queries (the special ones among them) against 64 bits."""
    import torch
    rng = np.random.default_rng(nP)
    A, B = smooth(nP, rng), smooth(nQ, rng)
    k = min(nP, nQ) // 10
    B[-k:] = B[:k]
    A[:k] = B[-k:]
    A[k:2 * k] = B[k:2 * k] + (1e-5 * rng.standard_normal((k, D))).astype(np.float32)
    nn, d, _ = listed_equals_fp32(ctx, A, B, 1)
    some = np.unique(np.concatenate([rng.integers(0, 2 * k, 200), rng.integers(0, nP, 300)]))
    Bd = torch.from_numpy(B).cuda().double()
    for i in some:
        dist = ((Bd - torch.from_numpy(A[i]).cuda().double()) ** 2).sum(1)
        two = torch.topk(dist, 2, largest=False)
        j, first, second = int(two.indices[0]), float(two.values[0]), float(two.values[1])
        assert abs(d[i] - first) <= 1e-5 * first + 1e-12
        if second - first > 1e-5 * second + 1e-9:
            assert nn[i] == j
        if i < k:
            assert nn[i] == i and d[i] == 0


CHILD = r"""
import sys
sys.path[:0] = [ROOT, ROOT + "/tests"]
import numpy as np
import paper_1801_01572_gb300 as lsr
from test_gpu_match_list import fpfh_like, listed_equals_fp32, smooth
assert lsr.lib().lsr_checked_build()
rng = np.random.default_rng(2)
for tile in (1, 2):
    with lsr.Context(0, match_tile=tile) as ctx:
        for precision in (1, 2):
            for nP, nQ in ((257, 385), (129, 8193), (700, 9001)):
                listed_equals_fp32(ctx, smooth(nP, rng), smooth(nQ, rng), precision)
            listed_equals_fp32(ctx, fpfh_like(300, rng), np.repeat(fpfh_like(1, rng), 3000, axis=0), precision)
print("CHILD_OK")
"""


@gpu
def test_listed_in_the_checked_build():
    """The bounds checks of the list's re-rank and search report nothing."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_01572_gb300 import _build
    _build.build(checked=True)
    p = subprocess.run([sys.executable, "-c", "ROOT = " + repr(ROOT) + CHILD], env=dict(os.environ, LSR_CHECKED="1"),
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and "CHILD_OK" in p.stdout, p.stderr[-3000:]
