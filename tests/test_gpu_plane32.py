"""The forward plane pass at 32 points in both of its forms, either side of the
plan size where they change over (64 blocks: four fields of 16 planes), with
odd rows, full rows, and sources longer than half of the padded line; against
the FP64 oracle at the FP32 path's bar."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import histories, oracle_values, rel_l2, run_library

pytestmark = pytest.mark.gpu
TOL = 1e-6

CASES = {   # nodes per axis of each domain; 4 planes' blocks per point along z
    "blocks8": [(16, 16, 2)],
    "blocks60_odd": [(15, 13, 15)],
    "blocks64": [(16, 16, 16)],
    "blocks68_odd": [(13, 15, 17)],
    "blocks84": [(15, 13, 12), (16, 16, 9)],
    "blocks64_long_source": [(9, 11, 6), (20, 19, 10)],
    "blocks80_long_source": [(9, 11, 8), (19, 20, 12)],
}


@pytest.mark.parametrize("push", ["all", "each"])    # the plan's form, in one launch or one per domain
@pytest.mark.parametrize("name", sorted(CASES))
def test_plane32(name, push):
    ns, h = CASES[name], 0.3
    doms = [synth.Domain((0.0, 0.0, 0.0), ns[0], h)]
    if len(ns) > 1:
        doms.append(synth.Domain((h * ns[0][0] + 1.1, 0.4, -0.2), ns[1], h))
    with rp.RetardedPotentials(doms, synth.C_AU, 0.05, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
        assert plan.pair_info(0, len(ns) - 1)["fft_m"][:2] == (32, 32)
        T = plan.query()["max_lag"] + 3
    hists = histories(synth.seeded_sources(doms), 0, T, 0.05)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [T - 1], push=push)
    if push == "each":
        same = run_library(doms, synth.C_AU, 0.05, hists, 0, [T - 1])
    for t, d in enumerate(doms):
        if push == "each":
            np.testing.assert_array_equal(res[T - 1][t], same[T - 1][t])
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, T - 1, np.arange(d.N))
        errs = rel_l2(res[T - 1][t], want)
        assert max(errs) <= TOL, (name, t, errs)
