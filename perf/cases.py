"""The work a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes what a user's program
holds before a time step (a finalized context with its history pushed, the
step's source slices, output buffers), ``run`` is one time step through the
public calls, ``work`` is what a step cannot do without and ``exact`` is the
step's result in 64 bits from plain torch (FFT convolutions, matrix products
and stencils of its own).

Sizes are those of the method's evaluation (two domains at 20 or 2000 bohr,
tens of domains far apart), of the elongated boxes of its cost model, and of
the tests' ragged and unequal grids.  The geometry is fixed by the case; the
sources (three Gaussians per domain with a continuity-consistent current, as
in the package's synthetic workloads) come from the seed.
"""
from __future__ import annotations

import math
import random
from collections import namedtuple

import numpy as np
import torch

from paper_2311_15429_gb300 import rp

C_AU = 137.036
COMING = 8          # slices of the coming steps a program has in hand; passes cycle through them
GROUP = 16          # history slices made and pushed at a time

Box = namedtuple("Box", "origin n h N")


def _box(origin, n, h):
    return Box(tuple(float(v) for v in origin), tuple(int(v) for v in n), float(h), int(n[0] * n[1] * n[2]))


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The smallest step: two molecules 20 bohr apart, both near, four launches.
        dict(name="pair16", kind="near", count=2, nx=16, ny=16, nz=16, h=0.3, apart=20.0, dt=0.05, how="calls"),
        # Four odd-sized neighbours with a large static density: the induced
        # response alone is propagated (ground-state split).
        dict(name="four27_split", kind="near", count=4, nx=27, ny=27, nz=27, h=0.3, apart=13.0, dt=0.05, how="split"),
        # Two elongated wires as in the method's cost model: boxes that are
        # not cubes, a fine time step and so many lags per pair.
        dict(name="wires16x96", kind="near", count=2, nx=16, ny=16, nz=96, h=0.25, apart=8.0, dt=0.01, how="calls"),
        # Neighbours whose grids have different spacings: not a convolution,
        # the cross pairs go through the direct sum.
        dict(name="spacings32", kind="unequal", count=2, n=32, h=0.25, n2=27, h2=0.3, apart=12.0, dt=0.05, how="calls"),
        # The headline: two 48^3 domains 2000 bohr apart, a 320-step history
        # on the device, pushes overlapped with the evaluation before them.
        dict(name="pair48", kind="near", count=2, nx=48, ny=48, nz=48, h=0.25, apart=2000.0, dt=0.05, how="event"),
        # The same between a host program's pinned buffers, copies included.
        dict(name="pair48_host", kind="near", count=2, nx=48, ny=48, nz=48, h=0.25, apart=2000.0, dt=0.05, how="host"),
        # The same with the history kept in host memory.
        dict(name="pair48_spill", kind="near", count=2, nx=48, ny=48, nz=48, h=0.25, apart=2000.0, dt=0.05,
             how="spill"),
        # Eight larger domains, every cross pair far (low-rank factors).
        dict(name="cells8x64", kind="far", count=8, n=64, h=0.25, dt=0.05, apart=300.0, how="event"),
        # Thirty-two medium domains, every cross pair far.
        dict(name="cells32x48", kind="far", count=32, n=48, h=0.25, dt=0.05, apart=300.0, how="event"),
        # The largest: domains of mixed sizes and spacings up to 96^3, plain calls.
        dict(name="mixed20", kind="mixed", count=20, geometry=3, dt=0.05, apart=320.0, how="calls"),
        # Far pairs by moments and the learned map instead of factors (a
        # hundredth of the memory).
        dict(name="learned16x48", kind="learned", count=16, n=48, h=0.25, dt=0.05, apart=600.0, how="calls"),
        # E and B on the grids of two domains from the potentials of three steps.
        dict(name="fields2x64", kind="fields", count=2, nx=64, ny=64, nz=64, h=0.25, dt=0.05, B=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["near", "deep", "wires", "unequal", "far", "mixed", "learned", "fields"])
    h = round(rng.uniform(0.2, 0.35), 3)
    if kind == "near":
        n = [_log_int(rng, 9, 64) for _ in range(3)]
        if rng.random() < 0.6:
            n = [n[0]] * 3
        count = rng.randint(1, 5)
        return dict(kind="near", count=count, nx=n[0], ny=n[1], nz=n[2], h=h,
                    apart=round(max(n) * h + rng.uniform(1.0, 12.0), 2), dt=0.05,
                    how=rng.choice(["calls", "calls", "event", "host", "split", "graph"]))
    if kind == "deep":
        n = _log_int(rng, 16, 48)
        return dict(kind="near", count=2, nx=n, ny=n, nz=n, h=h, apart=round(rng.uniform(300.0, 2000.0), 1), dt=0.05,
                    how=rng.choice(["calls", "event", "host", "spill", "graph"]))
    if kind == "wires":
        w, length = _log_int(rng, 6, 24), _log_int(rng, 32, 96)
        return dict(kind="near", count=rng.randint(1, 2), nx=w, ny=w, nz=length, h=h,
                    apart=round(w * h + rng.uniform(1.0, 10.0), 2), dt=0.01, how=rng.choice(["calls", "event"]))
    if kind == "unequal":
        n, n2, h2 = _log_int(rng, 9, 36), _log_int(rng, 9, 30), round(rng.uniform(0.2, 0.35), 3)
        return dict(kind="unequal", count=2, n=n, h=h, n2=n2, h2=h2 + (0.011 if abs(h2 - h) < 1e-9 else 0.0),
                    apart=round(0.5 * (n * h + n2 * h2) + rng.uniform(1.0, 8.0), 2), dt=0.05,
                    how=rng.choice(["calls", "event", "graph"]))
    if kind == "far":
        n = _log_int(rng, 24, 64)
        return dict(kind="far", count=rng.randint(4, 8 if n > 48 else 28), n=n, h=h, dt=0.05, apart=300.0,
                    how=rng.choice(["calls", "event", "event", "graph"]))
    if kind == "mixed":
        return dict(kind="mixed", count=rng.randint(6, 14), geometry=rng.randint(10, 9999), dt=0.05, apart=320.0,
                    how=rng.choice(["calls", "event"]))
    if kind == "learned":
        return dict(kind="learned", count=rng.randint(4, 14), n=_log_int(rng, 24, 48), h=h, dt=0.05, apart=600.0,
                    how="calls")
    return dict(kind="fields", count=rng.randint(2, 5), nx=_log_int(rng, 9, 96), ny=_log_int(rng, 9, 96),
                nz=_log_int(rng, 9, 96), h=h, dt=0.05, B=rng.random() < 0.7)


# ------------------------------------------------------------------ geometry

def _scatter(count, apart, seed):
    """Centres in a cube, at least `apart` from one another."""
    g = random.Random(seed)
    side = 2.0 * apart * count ** (1.0 / 3.0)
    pts = []
    while len(pts) < count:
        p = [g.uniform(-side / 2, side / 2) for _ in range(3)]
        if all(math.dist(p, q) >= apart for q in pts):
            pts.append(p)
    return pts


def _cubic(centre, n, h):
    return _box([v - h * (n - 1) / 2.0 for v in centre], (n, n, n), h)


def _domains(case):
    kind = case["kind"]
    if kind == "near":      # a row along x, nudged off the lattice
        n = (case["nx"], case["ny"], case["nz"])
        return [_box((case["apart"] * i, 0.37 * i, -0.21 * i), n, case["h"]) for i in range(case["count"])]
    if kind == "unequal":
        return [_cubic((0.0, 0.0, 0.0), case["n"], case["h"]),
                _cubic((case["apart"], 0.4, -0.3), case["n2"], case["h2"])]
    if kind in ("far", "learned"):
        return [_cubic(p, case["n"], case["h"]) for p in _scatter(case["count"], case["apart"], 7)]
    if kind == "mixed":
        g = random.Random(case["geometry"])
        ns = [24, 32, 48, 64, 96]
        return [_cubic(p, ns[i % 5] if i < 15 else g.choice(ns[:4]), g.uniform(0.2, 0.35))
                for i, p in enumerate(_scatter(case["count"], case["apart"], case["geometry"]))]
    return [_box((100.0 * i, 0.0, 0.0), (case["nx"], case["ny"], case["nz"]), case["h"]) for i in range(case["count"])]


def _distances(t, s):
    gap = far = 0.0
    for a in range(3):
        t0, t1 = t.origin[a], t.origin[a] + t.h * (t.n[a] - 1)
        s0, s1 = s.origin[a], s.origin[a] + s.h * (s.n[a] - 1)
        gap += max(0.0, t0 - s1, s0 - t1) ** 2
        far += max(abs(t1 - s0), abs(s1 - t0)) ** 2
    return math.sqrt(gap), math.sqrt(far)


def _lags(t, s, dt):
    lo, hi = _distances(t, s)
    return int(math.floor((0.0 if t is s else lo) / (C_AU * dt))), int(math.floor(hi / (C_AU * dt))) + 1


# ------------------------------------------------------------------ sources

class _Sources:
    """rho = sum_k A_k(t) g_k and J = sum_k A_k'(t) grad(erf(r/(sqrt2 s))/r)/(4 pi)
    of three Gaussians per domain, as float32 slices [4][N] at any step."""

    def __init__(self, boxes, seed, dt):
        g = np.random.default_rng(seed)
        self.dt, self.items = dt, []
        dev = torch.device("cuda", 0)
        for b in boxes:
            ax = [torch.arange(b.n[a], dtype=torch.float64, device=dev) * b.h for a in range(3)]
            sigma, a, phase = g.uniform(0.5, 1.0, 3), g.uniform(0.5, 1.5, 3), g.uniform(0.0, 2 * math.pi, 3)
            basis = torch.empty((3, 4, b.N), dtype=torch.float32, device=dev)
            for k in range(3):
                c = [g.uniform(0.25, 0.75) * b.h * (b.n[i] - 1) for i in range(3)]
                x, y, z = (ax[0] - c[0])[None, None, :], (ax[1] - c[1])[None, :, None], (ax[2] - c[2])[:, None, None]
                r2 = x * x + y * y + z * z
                r = r2.sqrt().clamp_min(1e-9)
                s = float(sigma[k])
                e = torch.exp(-r2 / (2 * s * s))
                basis[k, 0] = (e / (2 * math.pi * s * s) ** 1.5).reshape(-1)
                over_r = (math.sqrt(2 / math.pi) / s * e * r - torch.erf(r / (math.sqrt(2.0) * s))) / (r * r * r)
                for i, d in enumerate((x, y, z)):
                    basis[k, 1 + i] = (d * over_r).reshape(-1)
            self.items.append((basis, a, phase))

    def slice(self, d, j):
        basis, a, phase = self.items[d]
        arg = 0.3 * j * self.dt + phase
        w = torch.from_numpy(np.stack([a * (1 + 0.1 * np.sin(arg))] +
                                      [a * 0.03 * np.cos(arg) / (4 * math.pi)] * 3, 1).astype(np.float32))
        return (w.to(basis.device)[:, :, None] * basis).sum(0)

    def step(self, j):
        """One [4][N] tensor per domain at step j."""
        return [self.slice(d, j) for d in range(len(self.items))]


def _rho_J(xs):
    return [x[0] for x in xs], [x[1:].reshape(-1) for x in xs]


# ------------------------------------------------------------------ a time step

def prepare(case, seed):
    dev = torch.device("cuda", 0)
    boxes = _domains(case)
    if case["kind"] == "fields":
        lib = rp.RetardedPotentials(boxes, C_AU, case["dt"])
        f = _potentials(boxes, seed)
        return dict(kind="fields", lib=lib, phi=[v[0].contiguous() for v in f],
                    A=[[v[1 + 3 * i:4 + 3 * i].reshape(-1) for i in range(3)] for v in f],
                    E=[torch.empty(3 * b.N, device=dev) for b in boxes],
                    B=[torch.empty(3 * b.N, device=dev) if case["B"] else None for b in boxes])
    src = _Sources(boxes, seed, case["dt"])
    how, far = case["how"], case["kind"] in ("far", "mixed", "learned")
    flags = {"event": rp.RP_FLAG_OVERLAP_PUSH, "host": rp.RP_FLAG_OVERLAP_PUSH, "split": rp.RP_FLAG_GROUND_STATE_SPLIT,
             "spill": rp.RP_FLAG_HISTORY_SPILL}.get(how, 0)
    kw = dict(mode=rp.RP_MODE_LOWRANK, far_distance=200.0, far_batch=32, far_source_points=4) if far else {}
    if case["kind"] == "learned":
        flags |= rp.RP_FLAG_DEFER_FAR
    lib = rp.RetardedPotentials(boxes, C_AU, case["dt"], flags=flags, **kw)
    if case["kind"] == "learned":
        # a short fit: the step's work is the same as after a long one
        lib.train_far_model(300.0, gate=0.5, histories=64, samples=16, iterations=200, batch=512, validation=1,
                            seed=int(seed) % 1000 + 1)
    for j0 in range(-_history(case), 0, GROUP):
        xs = [src.step(j) for j in range(j0, min(j0 + GROUP, 0))]
        for x in xs:
            lib.push_all(*_rho_J(x))
        lib.sync()
    coming = [src.step(j) for j in range(COMING)]
    state = dict(kind=case["kind"], how=how, lib=lib, k=0, keep=coming)
    if how == "host":
        coming = [[x.cpu().pin_memory() for x in xs] for xs in coming]
        out = [[torch.zeros((4, b.N), pin_memory=True) for b in boxes] for _ in range(2)]
        state.update(keep=(coming, out), outputs=out,
                     pout=[tuple(rp.pointer_array(v) for v in _rho_J(o)) for o in out])
    if how in ("event", "host"):
        state["pin"] = [tuple(rp.pointer_array(v) for v in _rho_J(xs)) for xs in coming]
        if how == "event":
            state["pout"] = (rp.pointer_array(lib.phi), rp.pointer_array(lib.A))
    else:
        state["in"] = [_rho_J(xs) for xs in coming]
    if how == "graph":      # one recorded step on fixed buffers; the program copies each slice in
        state["flat"] = [torch.cat([x.reshape(-1) for x in xs]) for xs in coming]
        buf = torch.zeros_like(state["flat"][0])
        at, fixed = 0, []
        for b in boxes:
            fixed.append(buf[at:at + 4 * b.N].view(4, b.N))
            at += 4 * b.N
        rp.rp_graph_capture(lib.ctx, *_rho_J(fixed), lib.phi, lib.A)
        state["buf"] = buf
    if len(boxes) > 32:
        raise ValueError("more domains than a case returns")
    torch.cuda.synchronize()
    return state


def _potentials(boxes, seed):
    """phi and A of three steps on each grid: [10][N] around 1."""
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev).manual_seed(int(seed))
    return [torch.randn((10, b.N), generator=g, device=dev).mul_(0.05).add_(1.0) for b in boxes]


def run(state):
    if state["kind"] == "fields":
        E, B = state["E"], state["B"]
        for d in range(len(E)):
            rp.rp_fields(state["lib"].ctx, d, state["phi"][d], *state["A"][d], E[d], B[d])
        return [E, B] if B[0] is not None else [E]
    k = state["k"]
    state["k"] = k + 1
    how, lib = state["how"], state["lib"]
    if how == "event":
        rp.rp_push_all_event(lib.ctx, *state["pin"][k % COMING])
        rp.rp_evaluate(lib.ctx, *state["pout"])
        return [lib.phi, lib.A]
    if how == "host":       # results are read two steps later at the latest: two sets of buffers
        rp.rp_push_all_host(lib.ctx, *state["pin"][k % COMING])
        rp.rp_evaluate_host(lib.ctx, *state["pout"][k % 2])
        return [list(v) for v in _rho_J(state["outputs"][k % 2])]
    if how == "graph":
        state["buf"].copy_(state["flat"][k % COMING])
        rp.rp_graph_step(lib.ctx)
        return [lib.phi, lib.A]
    lib.push_all(*state["in"][k % COMING])
    phi, A = lib.evaluate()
    return [phi, A]


def _history(case):
    """Slices before the first timed step: what the deepest pair reads (the
    learned map also reads a window of delays around it), and some."""
    boxes = _domains(case)
    deepest = max(_lags(t, s, case["dt"])[1] for t in boxes for s in boxes)
    return deepest + (20 if case["kind"] == "learned" else 3)


# ------------------------------------------------------------------ what a step cannot do without

def _padded(n):
    for m in (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192):
        if m >= n:
            return m
    return n


def work(case):
    boxes = _domains(case)
    if case["kind"] == "fields":
        n = sum(b.N for b in boxes)
        return dict(bytes=4.0 * n * (10 + 3 + (3 if case["B"] else 0)), flops=(60.0 if case["B"] else 30.0) * n)
    far = case["kind"] in ("far", "mixed", "learned")
    nbytes = flops = 0.0
    for s in boxes:
        nbytes += 2 * 16.0 * s.N                      # the new slice in, the potentials out
        lags = set()
        for t in boxes:
            if far and t is not s:
                flops += 4 * 2.0 * 64 * 64 * (_lags(t, s, case["dt"])[1] - _lags(t, s, case["dt"])[0] + 1)
                continue
            lo, hi = _lags(t, s, case["dt"])
            lags.update(range(lo, hi + 1))
            if t.h != s.h:
                flops += 34.0 * t.N * s.N             # the direct sum
            else:
                m = math.prod(_padded(t.n[a] + s.n[a] - 1) for a in range(3))
                flops += (hi - lo + 1) * 4 * (2.0 if t is s else 4.0) * m
        nbytes += 16.0 * s.N * (len(lags) - (0 in lags))   # the older slices its near pairs read
        m = math.prod(_padded(2 * v - 1) for v in s.n)
        flops += 2 * 4 * 2.5 * m * math.log2(m)       # one forward and one inverse transform per field
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------ the step in 64 bits

def exact(case, seed):
    boxes = _domains(case)
    dev = torch.device("cuda", 0)
    dt = case["dt"]
    if case["kind"] == "fields":
        f = [_exact_fields(case, b, v) for b, v in zip(boxes, _potentials(boxes, seed))]
        return [[v[0] for v in f], [v[1] for v in f]] if case["B"] else [[v[0] for v in f]]
    if case["kind"] == "mixed":     # unequal spacings far apart: 1e12 pairs of nodes, minutes in 64 bits
        return None
    src = _Sources(boxes, seed, dt)
    first = -_history(case)
    still = [x.double() for x in src.step(first)] if case["how"] == "split" else None

    def sample(s, j):
        x = src.slice(s, max(j, first)).double()
        return x - still[s] if still is not None else x

    phi, A = [], []
    for ti, t in enumerate(boxes):
        total = torch.zeros((4, t.N), dtype=torch.float64, device=dev)
        for si, s in enumerate(boxes):
            if t.h == s.h:
                total += _by_fft(t, s, ti == si, lambda m: sample(si, -m), dt)
            else:
                total += _by_sum(t, s, lambda m: sample(si, -m), dt)
        phi.append(total[0])
        A.append((total[1:] / C_AU).reshape(-1))
    return [phi, A]


def _by_fft(t, s, same, sample, dt):
    dev = torch.device("cuda", 0)
    size = [_padded(t.n[a] + s.n[a] - 1) for a in range(3)]
    d2 = 0.0
    for a, shape in zip(range(3), ((1, 1, -1), (1, -1, 1), (-1, 1, 1))):
        i = torch.arange(size[a], dtype=torch.float64, device=dev)
        i = torch.where(i < t.n[a], i, i - size[a])   # displacement in nodes, cyclic
        d2 = d2 + ((t.origin[a] - s.origin[a]) + t.h * i).reshape(shape) ** 2
    R = d2.sqrt()
    tau = R / (C_AU * dt)
    inv = t.h ** 3 / R
    if same:
        inv[0, 0, 0] = (3 * math.log(2 + math.sqrt(3)) - math.pi / 2) * t.h ** 2
    acc = None
    lo, hi = _lags(t, s, dt)
    for m in range(0 if same else lo, hi + 1):
        G = torch.fft.rfftn((1.0 - (m - tau).abs()).clamp_min(0.0) * inv)
        x = sample(m).reshape(4, s.n[2], s.n[1], s.n[0])
        y = torch.fft.rfftn(x, s=(size[2], size[1], size[0]), dim=(1, 2, 3)) * G
        acc = y if acc is None else acc + y
    out = torch.fft.irfftn(acc, s=(size[2], size[1], size[0]), dim=(1, 2, 3))
    return out[:, :t.n[2], :t.n[1], :t.n[0]].reshape(4, t.N)


def _nodes(b):
    dev = torch.device("cuda", 0)
    z, y, x = torch.meshgrid(*[b.origin[a] + b.h * torch.arange(b.n[a], dtype=torch.float64, device=dev)
                               for a in (2, 1, 0)], indexing="ij")
    return [v.reshape(-1) for v in (x, y, z)]


def _by_sum(t, s, sample, dt):
    tn, sn = _nodes(t), _nodes(s)
    lo, hi = _lags(t, s, dt)
    S = [sample(m) for m in range(lo, hi + 1)]
    out = torch.empty((4, t.N), dtype=torch.float64, device=tn[0].device)
    step = max(1, 100_000_000 // s.N)
    for a in range(0, t.N, step):
        R = sum((tn[i][a:a + step, None] - sn[i][None, :]) ** 2 for i in range(3)).sqrt()
        tau, inv = R / (C_AU * dt), s.h ** 3 / R
        out[:, a:a + step] = sum(S[m - lo] @ ((1.0 - (m - tau).abs()).clamp_min(0.0) * inv).T
                                 for m in range(lo, hi + 1))
    return out


def _exact_fields(case, b, f):
    f = f.double().reshape(10, b.n[2], b.n[1], b.n[0])

    def d(v, axis):         # second order, one-sided on the faces; axis 0 is x
        v = v.movedim(2 - axis, 0)
        o = torch.empty_like(v)
        o[1:-1] = v[2:] - v[:-2]
        o[0] = -3 * v[0] + 4 * v[1] - v[2]
        o[-1] = 3 * v[-1] - 4 * v[-2] + v[-3]
        return (o / (2 * b.h)).movedim(0, 2 - axis)

    phi, A, A1, A2 = f[0], f[1:4], f[4:7], f[7:10]
    E = torch.stack([-d(phi, i) - (3 * A[i] - 4 * A1[i] + A2[i]) / (2 * case["dt"] * C_AU) for i in range(3)])
    B = torch.stack([d(A[(i + 2) % 3], (i + 1) % 3) - d(A[(i + 1) % 3], (i + 2) % 3) for i in range(3)])
    return E.reshape(-1), B.reshape(-1)
