"""The source partition under the ground-state split: contexts that own
complementary sources, pushed together with NULL for the other sources or one
by one, add up to the context that owns every source; so do their static
potentials."""
import numpy as np
import pytest
import torch

from paper_2311_15429_gb300 import rp, synth

pytestmark = pytest.mark.gpu

DOMS = [synth.cubic((0.0, 0.0, 0.0), 12, 0.25), synth.cubic((8.0, 0.5, -0.3), 12, 0.25),
        synth.Domain((-6.0, 3.0, 1.0), (9, 7, 11), 0.3)]       # the third by the direct sum
T = 12


def _run(hists, owned, first_alone):
    dev = torch.device("cuda", 0)
    with rp.RetardedPotentials(DOMS, synth.C_AU, 0.05, owned_sources=owned,
                               flags=rp.RP_FLAG_GROUND_STATE_SPLIT) as lib:
        for i in range(T):
            x = [torch.from_numpy(h[i]).to(dev) if d in owned else None for d, h in enumerate(hists)]
            r = [None if v is None else v[0].contiguous() for v in x]
            J = [None if v is None else v[1:].reshape(-1).contiguous() for v in x]
            if first_alone and i == 0:
                for d in owned:
                    lib.push(d, r[d], J[d])
            else:
                lib.push_all(r, J)
        static = ([torch.empty_like(v) for v in lib.phi], [torch.empty_like(v) for v in lib.A])
        rp.rp_ground_potential(lib.ctx, *static)
        lib.evaluate()
        lib.sync()
        return [np.concatenate([v.cpu().numpy() for v in (lib.phi[t], lib.A[t], static[0][t], static[1][t])])
                for t in range(len(DOMS))]


@pytest.mark.parametrize("first_alone", [False, True])
def test_partitioned_split_adds_up(first_alone):
    hists = [s.history(0, T, 0.05) for s in synth.seeded_sources(DOMS)]
    full = _run(hists, [0, 1, 2], False)
    parts = [_run(hists, p, first_alone) for p in ([0, 2], [1])]
    for t, d in enumerate(DOMS):
        total = sum(p[t].astype(np.float64) for p in parts)
        at = 0
        for n in (d.N, 3 * d.N, d.N, 3 * d.N):
            a, b = total[at:at + n], full[t][at:at + n].astype(np.float64)
            assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b), (t, at)
            at += n
