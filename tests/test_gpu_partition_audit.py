"""The FP64 audit under a source partition: a context keeps the raw history of
its own sources only (rp_push_all gets NULL for the others), and its audit
scores its own share of the potentials."""
import numpy as np
import pytest
import torch

from paper_2311_15429_gb300 import rp, synth

from _harness import oracle_values

DOMS = [synth.cubic((0.0, 0.0, 0.0), 12, 0.25), synth.cubic((8.0, 0.5, -0.3), 12, 0.25)]
T = 12


def test_the_plan_keeps_owned_histories_only():
    size = {}
    for owned in (None, [0]):
        for flags in (0, rp.RP_FLAG_AUDIT):
            with rp.RetardedPotentials(DOMS, synth.C_AU, 0.05, flags=flags | rp.RP_FLAG_PLAN_ONLY,
                                       owned_sources=owned) as plan:
                size[owned is None, flags] = plan.query()["device_bytes"]
    ring = {k: size[k, rp.RP_FLAG_AUDIT] - size[k, 0] for k in (True, False)}
    assert ring[True] == 2 * ring[False] > 0


@pytest.mark.gpu
@pytest.mark.parametrize("own", [0, 1])
def test_audit_of_a_share(own):
    dev = torch.device("cuda", 0)
    hists = [s.history(0, T, 0.05) for s in synth.seeded_sources(DOMS)]
    with rp.RetardedPotentials(DOMS, synth.C_AU, 0.05, owned_sources=[own], flags=rp.RP_FLAG_AUDIT) as lib:
        for i in range(T):
            x = torch.from_numpy(hists[own][i]).to(dev)
            r, J = [None, None], [None, None]
            r[own], J[own] = x[0].contiguous(), x[1:].reshape(-1).contiguous()
            lib.push_all(r, J)
        lib.evaluate()
        rel = rp.rp_audit(lib.ctx, lib.phi, lib.A, 256, seed=2)
        assert np.all(rel <= 1e-6) and np.all(rel > 0), rel
        share = [h if d == own else np.zeros_like(h) for d, h in enumerate(hists)]
        for t, d in enumerate(DOMS):
            nodes = np.arange(0, d.N, 7)
            want = oracle_values(DOMS, share, 0, synth.C_AU, 0.05, t, T - 1, nodes)
            got = rp.rp_audit_values(lib.ctx, t, nodes)
            assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))
