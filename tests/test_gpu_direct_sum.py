"""The direct sum's precision and its order, against the FP64 oracle: exact
geometry where the grid's numbers are exact, a compensated sum, any unit of
length and speed of light, and the same bits with and without the workspace
of its parts."""
import numpy as np
import pytest

from paper_2311_15429_gb300 import rp, synth

from _harness import oracle_values, run_library

pytestmark = pytest.mark.gpu

UNIT = 2.0 ** -24       # rounding unit of FP32


def _joint(got, want):
    return float(np.linalg.norm(got.T - want) / np.linalg.norm(want))


def _noise(doms, T, seed=3):
    rng = np.random.default_rng(seed)
    return [rng.standard_normal((T, 4, d.N)).astype(np.float32) for d in doms]


@pytest.mark.parametrize("offset", [None, (8.0, 0.5, -0.25), (8.3, 0.47, -0.21)])
def test_geometry_keeps_its_bits(offset):
    """White noise: every node pair's relative error enters the sum's in
    quadrature.  At a spacing of 1/4 the positions and their differences are
    exact, and what is left per pair (R^2, its root, the volume, tau and the
    hat weight of a sample difference) is 2.5 rounding units; positions rounded
    in units of the light step cost three times that."""
    doms = [synth.Domain((0.0, 0.0, 0.0), (24, 24, 24), 0.25)]
    if offset:
        doms.append(synth.Domain(offset, (20, 18, 16), 0.25))
    hists = _noise(doms, 7)
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [6], mode=rp.RP_MODE_DIRECT)
    for t, d in enumerate(doms):
        nodes = np.arange(0, d.N, 17)
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, 6, nodes)
        assert _joint(res[6][t][:, nodes], want) <= 2.5 * UNIT


@pytest.mark.parametrize("n", [(1, 1, 9), (12, 1, 9)])   # targets on their own, four to a thread
def test_sum_is_compensated(n):
    """Two samples of 2^24 and -2^24 at nodes mirrored on the targets' plane
    cancel exactly; a plain FP32 chain between them loses the samples of size
    one, whose sum is the result."""
    h = 0.25
    src = synth.Domain((0.0, 0.0, 0.0), (2, 2, 40), h)
    doms = [src, synth.Domain((1.0 if n[0] > 1 else 5.0, 0.5 * h, 2.0), n, h)]
    rng = np.random.default_rng(5)
    hists = [(0.5 + rng.random((6, 4, d.N))).astype(np.float32) for d in doms]
    hists[0][:, :, 0] = 2.0 ** 24       # node (0, 0, 0)
    hists[0][:, :, 2] = -2.0 ** 24      # node (0, 1, 0): the same warp, two sources later
    res = run_library(doms, synth.C_AU, 0.05, hists, 0, [5], mode=rp.RP_MODE_DIRECT)
    want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, 1, 5, np.arange(doms[1].N))
    assert _joint(res[5][1], want) <= 1e-6


@pytest.mark.parametrize("unit", [1.0, 2.0 ** -35, 2.0 ** 35])     # h^3 stays an FP32 number
@pytest.mark.parametrize("c", [synth.C_AU, 1e21])
def test_any_unit_of_length_and_speed(unit, c):
    """A speed of light without bound (the static limit) and lengths far from
    one: finite, and as accurate as at the usual scale."""
    doms = [synth.Domain((0.0, 0.0, 0.0), (9, 8, 7), 0.3 * unit),
            synth.Domain((3.5 * unit, 0.4 * unit, -0.3 * unit), (8, 9, 5), 0.25 * unit)]
    hists = _noise(doms, 8)
    res = run_library(doms, c * unit, 0.05, hists, 0, [7], mode=rp.RP_MODE_DIRECT)
    for t, d in enumerate(doms):
        want = oracle_values(doms, hists, 0, c * unit, 0.05, t, 7, np.arange(d.N))
        got = res[7][t]
        assert np.isfinite(got).all()
        scale = np.linalg.norm(want[:, :1]), np.linalg.norm(want[:, 1:])   # A carries 1 / c
        assert np.linalg.norm(got.T[:, :1] - want[:, :1]) <= 1e-6 * scale[0]
        assert np.linalg.norm(got.T[:, 1:] - want[:, 1:]) <= 1e-6 * scale[1]


CASES = {   # domains, mode: parts for both targets, for one only (a small one under a large source), for none
    "parts": ([synth.Domain((0.0, 0.0, 0.0), (20, 19, 18), 0.25), synth.Domain((6.0, 0.4, -0.3), (17, 13, 11), 0.3)],
              rp.RP_MODE_DIRECT),
    "one_target": ([synth.Domain((0.0, 0.0, 0.0), (24, 23, 22), 0.25), synth.Domain((7.0, 0.4, -0.3), (5, 4, 3), 0.3)],
                   rp.RP_MODE_FFT),
    "no_parts": ([synth.Domain((0.0, 0.0, 0.0), (9, 8, 5), 0.25), synth.Domain((3.5, 0.4, -0.3), (5, 4, 3), 0.3)],
                 rp.RP_MODE_DIRECT),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_same_bits_without_the_workspace(name):
    """Under a device budget there is no workspace and a block runs its
    targets' parts in turn: the same bits; both against the oracle."""
    import torch
    dev = torch.device("cuda", 0)
    doms, mode = CASES[name]
    hists = _noise(doms, 7)
    got = []
    for budget in (0, 1 << 33):
        with rp.RetardedPotentials(doms, synth.C_AU, 0.05, mode=mode, device_budget=budget) as lib:
            for i in range(7):
                x = [torch.from_numpy(h[i]).to(dev) for h in hists]
                lib.push_all([v[0].contiguous() for v in x], [v[1:].contiguous().reshape(-1) for v in x])
            phi, A = lib.evaluate()
            got.append([np.concatenate([phi[t].cpu().numpy()[None], A[t].cpu().numpy().reshape(3, -1)])
                        for t in range(len(doms))])
    for t, d in enumerate(doms):
        np.testing.assert_array_equal(got[0][t], got[1][t])
        nodes = np.arange(0, d.N, max(1, d.N // 400))
        want = oracle_values(doms, hists, 0, synth.C_AU, 0.05, t, 6, nodes)
        assert _joint(got[0][t][:, nodes], want) <= 2e-6    # FP32 tau at a spacing that is not exact
