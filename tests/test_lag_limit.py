"""The longest lag window of a direct pair: one limit where a context runs, the
planner's where it only plans, each named by the refusal."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

DOMS = [synth.Domain((0.0, 0.0, 0.0), (9, 8, 7), 0.3), synth.Domain((3.5, 0.4, -0.3), (8, 9, 5), 0.25)]


def _refusal(c, flags=0):
    ctx = rp.rp_create(c, 0.05, mode=rp.RP_MODE_DIRECT, flags=flags)
    try:
        for d in DOMS:
            rp.rp_add_domain(ctx, d.origin, d.n, d.h)
        with pytest.raises(rp.RPError) as e:
            rp.rp_finalize(ctx)
        assert e.value.status == rp.RP_ERR_UNSUPPORTED
        return rp.rp_last_error(ctx)
    finally:
        rp.rp_destroy(ctx)


def test_a_plan_takes_up_to_600_steps():
    for c, want in ((0.45, 227), (0.2, 507)):
        with rp.RetardedPotentials(DOMS, c, 0.05, mode=rp.RP_MODE_DIRECT, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
            p = [plan.pair_info(t, s) for t in (0, 1) for s in (0, 1)]
            assert max(q["lag_hi"] - q["lag_lo"] + 1 for q in p) == want
    msg = _refusal(0.1, rp.RP_FLAG_PLAN_ONLY)
    assert "1011" in msg and "600" in msg


@pytest.mark.gpu
@pytest.mark.parametrize("c,steps", [(0.45, 227), (0.2, 507), (0.1, 1011)])
def test_a_running_context_names_its_limit(c, steps):
    msg = _refusal(c)
    assert str(steps) in msg and "226" in msg


@pytest.mark.gpu
def test_the_longest_window_runs():
    from _harness import oracle_values, rel_l2, run_library
    c = 0.4515
    with rp.RetardedPotentials(DOMS, c, 0.05, mode=rp.RP_MODE_DIRECT, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
        p = [plan.pair_info(t, s) for t in (0, 1) for s in (0, 1)]
        assert max(q["lag_hi"] - q["lag_lo"] + 1 for q in p) == 226
        lag = plan.query()["max_lag"]
    rng = np.random.default_rng(9)
    hists = [rng.standard_normal((lag + 2, 4, d.N)).astype(np.float32) for d in DOMS]
    res = run_library(DOMS, c, 0.05, hists, 0, [lag + 1], mode=rp.RP_MODE_DIRECT)
    for t, d in enumerate(DOMS):
        want = oracle_values(DOMS, hists, 0, c, 0.05, t, lag + 1, np.arange(d.N))
        errs = rel_l2(res[lag + 1][t], want)
        # FP32 leaves tau a few roundings of its size, which weigh samples that differ by O(1)
        assert max(errs) <= 1e-6 + 4e-7 * lag, (t, errs)
