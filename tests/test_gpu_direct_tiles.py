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


@pytest.mark.parametrize("mode", [rp.RP_MODE_FFT, rp.RP_MODE_DIRECT])
def test_direct_sum_reads_each_targets_own_samples(mode):
    """One sample that is not finite reaches exactly the nodes whose lag
    interval holds it (neighbours that share a thread's samples do not)."""
    import torch
    dev = torch.device("cuda", 0)
    c, dt = 20.0, 0.05                                     # one light step per bohr
    doms = [synth.Domain((0.0, 0.0, 0.0), (12, 4, 3), 0.3), synth.Domain((5.0, 0.2, -0.1), (9, 3, 2), 0.25)]
    with rp.RetardedPotentials(doms, c, dt, mode=mode, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
        T = plan.query()["max_lag"] + 3
    rng = np.random.default_rng(11)
    hists = [rng.standard_normal((T, 4, d.N)).astype(np.float32) for d in doms]
    bad, lag = 13, 3                                       # a node of domain 1, this many steps back
    hists[1][T - 1 - lag, 0, bad] = np.inf
    with rp.RetardedPotentials(doms, c, dt, mode=mode) as lib:
        for i in range(T):
            x = [torch.from_numpy(h[i]).to(dev) for h in hists]
            lib.push_all([v[0].contiguous() for v in x], [v[1:].contiguous().reshape(-1) for v in x])
        phi, _ = lib.evaluate()
        got = ~np.isfinite(phi[0].cpu().numpy())
    src = np.array([v[bad] for v in doms[1].coords()])
    tau = np.sqrt(sum((a - b) ** 2 for a, b in zip(doms[0].coords(), src))) / (c * dt)
    assert np.all(np.abs(tau - np.round(tau)) > 1e-4)      # no node on an interval's edge
    m = np.floor(tau).astype(int)
    want = (m == lag) | (m == lag - 1)
    assert want.any() and (~want).any()
    np.testing.assert_array_equal(got, want)
