"""The plane passes of square cross-sections: odd, short and full rows, one
more or one fewer than a round of tasks, sources longer than half of the
padded line (no zero half to skip) and targets longer than it (nothing
cropped), against the FP64 oracle at the FP32 path's bar."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import histories, oracle_values, rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-6

# domains (nodes per axis), and the source the context owns (None: all)
CASES = {
    "m32_odd": ([(15, 13, 9), (16, 16, 7)], None),
    "m64_odd": ([(31, 27, 5), (32, 32, 4)], None),
    "m96_short_rows": ([(33, 48, 5), (48, 35, 4)], None),
    "m128_odd": ([(63, 49, 3), (50, 64, 4)], None),
    "m192_odd": ([(95, 81, 2), (65, 96, 3)], None),
    "m64_long_source": ([(9, 11, 6), (50, 47, 3)], None),
    "m128_long_target": ([(90, 85, 3), (20, 33, 4)], 1),
    "m96_long_both": ([(70, 61, 3), (26, 21, 4)], 1),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_plane_lines(name):
    import torch
    ns, own = CASES[name]
    h, c, dt, T = 0.3, synth.C_AU, 0.05, 20
    doms = [synth.Domain((0.0, 0.0, 0.0), ns[0], h), synth.Domain((h * ns[0][0] + 1.1, 0.4, -0.2), ns[1], h)]
    hists = histories(synth.seeded_sources(doms), 0, T, dt)
    owned = [0, 1] if own is None else [own]
    dev = torch.device("cuda", 0)
    with rp.RetardedPotentials(doms, c, dt, owned_sources=None if own is None else owned) as lib:
        for i in range(T):
            for d in owned:
                x = torch.from_numpy(hists[d][i]).to(dev)
                lib.push(d, x[0].contiguous(), x[1:].contiguous().reshape(-1))
        phi, A = lib.evaluate()
        torch.cuda.synchronize()
        src = hists if own is None else [x if d in owned else np.zeros_like(x) for d, x in enumerate(hists)]
        rng = np.random.default_rng(3)
        for t, d in enumerate(doms):
            nodes = np.sort(rng.choice(d.N, min(d.N, 1500), replace=False))
            want = oracle_values(doms, src, 0, c, dt, t, T - 1, nodes)
            got = np.concatenate([phi[t].cpu().numpy()[None], A[t].cpu().numpy().reshape(3, -1)])
            errs = rel_l2(got[:, nodes], want)
            assert max(errs) <= TOL, (name, t, errs)
