"""The rates that the benchmark states for the FP32 matcher and the consensus
estimate, from made-up kernel times: work and time belong to the same kernels.
"""
from types import SimpleNamespace

import pytest

import bench


def _info(n_p, terms):
    times = {"k_match_seed<false>": (4, 4.0), "k_match_win<32, false>": (4, 8.0)}
    prof = SimpleNamespace(match_terms=terms, survivors=1000, n_normal_ok=500)
    return dict(nP=n_p, nQ=20000, main_kernel=bench.MAIN_KERNEL["fp32"], match="fp32", main_times=times, prof=prof,
                params=SimpleNamespace(n_hypotheses=1000), n_prof=4,
                kernel_times={**times, "k_consensus_count<true>": (4, 2.0), "k_gather<true>": (4, 1.0)})


@pytest.mark.parametrize("terms", [3.0e9, 5.0e10])
def test_matcher_rate_is_both_passes_terms_over_both_passes_time(terms):
    r = bench.roofline(_info(30000, terms))
    assert r["launches_timed"] == 4 and r["launch_ms"] == pytest.approx(3.0)
    assert r["achieved"] == pytest.approx(3 * terms / 3e-3 / 1e12)
    rows = {k["kernel"]: k for k in bench.kernel_table(_info(30000, terms))["kernels"]}
    for name in ("k_match_seed<false>", "k_match_win<32, false>"):
        assert rows[name]["achieved"] == pytest.approx(3 * terms / 3e-3 / 1e12)
    assert rows["k_gather<true>"]["unit"] == "GB/s"


@pytest.mark.parametrize("n_p,read", [(16383, 16383), (16384, 512), (30000, 938)])
def test_consensus_estimate_is_charged_the_points_it_reads(n_p, read):
    rows = {k["kernel"]: k for k in bench.kernel_table(_info(n_p, 1e9))["kernels"]}
    assert rows["k_consensus_count<true>"]["work_per_step"] == 16.0 * read + 56.0 * 500
