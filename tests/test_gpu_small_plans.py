"""Plans so small that one block a tile is the whole MAC: unsplit tiles of few
entries, split ones of more, with and without the extra FFT warps; against the
FP64 oracle at the FP32 path's bar."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import histories, oracle_values, rel_l2, run_library

pytestmark = pytest.mark.gpu
TOL = 1e-6

CASES = {   # domains, edge, distance between their origins
    "one14": (1, (14, 14, 14), 0.0),            # M = 32
    "two14": (2, (14, 14, 14), 8.2),
    "two16": (2, (16, 16, 16), 8.8),
    "one20": (1, (20, 20, 20), 0.0),            # M = 48
    "one24": (1, (24, 24, 24), 0.0),
    "four19": (4, (19, 19, 19), 300.0),         # several units a block, three entries a tile
    "one_box": (1, (16, 16, 33), 0.0),          # M = 96 along z alone
}


@pytest.mark.parametrize("plain", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_small_plans(name, plain):
    count, n, apart = CASES[name]
    doms = [synth.Domain((apart * i, 0.4 * i, -0.2 * i), n, 0.3) for i in range(count)]
    with rp.RetardedPotentials(doms, synth.C_AU, 0.05, flags=rp.RP_FLAG_PLAN_ONLY) as plan:
        T = plan.query()["max_lag"] + 3
    hists = histories(synth.seeded_sources(doms), 0, T, 0.05)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [T - 1], flags=rp.RP_FLAG_PLAIN_SUM if plain else 0)
    for t, d in enumerate(doms):
        nodes = np.arange(0, d.N, max(1, d.N // 1500))
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, T - 1, nodes)
        errs = rel_l2(res[T - 1][t][:, nodes], want)
        assert max(errs) <= TOL, (name, t, errs)


@pytest.mark.parametrize("warps", [0, 8])
@pytest.mark.parametrize("plain", [False, True])
def test_launches_of_one_column_class(plain, warps):
    """A cube and a box of the same padded length along z are two MAC launches,
    each with warps of its own."""
    if warps and not plain:
        pytest.skip("the compensated sum has one variant")
    doms = [synth.Domain((0.0, 0.0, 0.0), (25, 26, 27), 0.3), synth.Domain((9.0, 0.4, -0.2), (14, 15, 28), 0.3)]
    flags = rp.RP_FLAG_PLAIN_SUM if plain else 0
    with rp.RetardedPotentials(doms, synth.C_AU, 0.05, flags=flags, mac_warps=warps) as lib:
        T = lib.query()["max_lag"] + 3
        used = lib.query()["mac_warps"]
    assert used == (warps or used) and used in ((8, 12, 16) if plain else (12,))
    hists = histories(synth.seeded_sources(doms), 0, T, 0.05)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [T - 1], flags=flags, mac_warps=warps)
    for t, d in enumerate(doms):
        nodes = np.arange(0, d.N, max(1, d.N // 1500))
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, T - 1, nodes)
        errs = rel_l2(res[T - 1][t][:, nodes], want)
        assert max(errs) <= TOL, (t, errs)
