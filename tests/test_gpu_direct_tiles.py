"""The direct sum's tiles, shares and parts at the sizes where they end:
white-noise histories (a sample of the wrong lag or node is an O(1) error)
against the FP64 oracle."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import oracle_values, rel_l2, run_library

pytestmark = pytest.mark.gpu

# FP32 leaves tau = R/(c dt) with a few roundings of its size, which the hat
# weights carry into the sum of samples that differ by O(1)
TOL_BASE, TOL_PER_LAG = 1e-6, 4e-7

CASES = {   # domains, speed of light (the lag window), mode
    "one_node": ([synth.Domain((0.0, 0.0, 0.0), (1, 1, 1), 0.3), synth.Domain((2.0, 0.1, 0.2), (3, 2, 2), 0.25)],
                 137.036, rp.RP_MODE_DIRECT),
    "tile_edges": ([synth.Domain((0.0, 0.0, 0.0), (65, 1, 1), 0.3), synth.Domain((1.0, 3.0, 0.5), (43, 3, 1), 0.25)],
                   137.036, rp.RP_MODE_DIRECT),
    "parts": ([synth.Domain((0.0, 0.0, 0.0), (13, 11, 9), 0.3), synth.Domain((5.0, 0.4, -0.3), (10, 9, 8), 0.25)],
              137.036, rp.RP_MODE_FFT),
    "lags50": ([synth.Domain((0.0, 0.0, 0.0), (9, 8, 7), 0.3), synth.Domain((3.5, 0.4, -0.3), (8, 9, 5), 0.25)],
               3.0, rp.RP_MODE_DIRECT),
    "lags130": ([synth.Domain((0.0, 0.0, 0.0), (9, 8, 7), 0.3), synth.Domain((3.5, 0.4, -0.3), (8, 9, 5), 0.25)],
                1.2, rp.RP_MODE_DIRECT),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_direct_sum_against_oracle(name):
    doms, c, mode = CASES[name]
    dt = 0.05
    with rp.RetardedPotentials(doms, c, dt, mode=mode, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
        lag = plan.query()["max_lag"]
    rng = np.random.default_rng(7)
    T = lag + 3
    hists = [rng.standard_normal((T, 4, d.N)).astype(np.float32) for d in doms]
    res = run_library(doms, c, dt, hists, 0, [T - 1], mode=mode)
    for t, d in enumerate(doms):
        want = oracle_values(doms, hists, 0, c, dt, t, T - 1, np.arange(d.N))
        errs = rel_l2(res[T - 1][t], want)
        assert max(errs) <= TOL_BASE + TOL_PER_LAG * lag, (name, t, lag, errs)
