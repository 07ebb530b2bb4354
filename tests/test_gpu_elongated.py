"""Grids that are not cubes on the kernels of their padded length along z: the
column pass and the MAC of every compiled length under cross-sections of one
or several 16-column tiles, square and not, and launches of so few tiles that
a block takes one field or two of a tile.  Against the FP64 oracle at the FP32
path's bar."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import histories, oracle_values, rel_l2, run_library

pytestmark = pytest.mark.gpu
TOL = 1e-6

SHAPES = {   # nodes -> padded (x, y, z)
    "8x16x32": (4, 8, 15),
    "12x16x48": (6, 7, 23),
    "32x32x64": (15, 16, 29),
    "16x16x96": (8, 8, 41),
    "6x32x128": (3, 13, 59),
    "16x48x192": (7, 20, 90),
    "64x16x32_many_tiles": (31, 8, 16),
    "8x12x64_no_class": (4, 6, 30),
}


@pytest.mark.parametrize("plain", [False, True])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_elongated_grids(name, plain):
    n = SHAPES[name]
    doms = [synth.Domain((0.0, 0.0, 0.0), n, 0.3), synth.Domain((0.3 * n[0] + 1.3, 0.4, -0.2), n, 0.3)]
    hists = histories(synth.seeded_sources(doms), 0, 14, 0.05)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [13], flags=rp.RP_FLAG_PLAIN_SUM if plain else 0)
    for t, d in enumerate(doms):
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, 13, np.arange(d.N))
        errs = rel_l2(res[13][t], want)
        assert max(errs) <= TOL, (name, t, errs)
