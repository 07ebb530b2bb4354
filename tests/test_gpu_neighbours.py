"""Neighbouring domains whose targets read the same source slots (the MAC then
takes the same tile of every target in turn): three targets of one padded
size, four fields a block and, with few tiles, fewer; against the FP64 oracle
at the FP32 path's bar."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import histories, oracle_values, rel_l2, run_library

pytestmark = pytest.mark.gpu
TOL = 1e-6


@pytest.mark.parametrize("n", [(16, 16, 16), (8, 8, 30), (17, 20, 33)])
def test_neighbours_share_slots(n):
    doms = [synth.Domain(((0.3 * n[0] + 0.7) * i, 0.3 * i, -0.2 * i), n, 0.3) for i in range(3)]
    hists = histories(synth.seeded_sources(doms), 0, 12, 0.05)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [10, 11])
    for step in (10, 11):
        for t, d in enumerate(doms):
            nodes = np.arange(0, d.N, max(1, d.N // 3000))
            want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, step, nodes)
            errs = rel_l2(res[step][t][:, nodes], want)
            assert max(errs) <= TOL, (n, step, t, errs)
