"""FP64 decisions beside their threshold: for chosen sites of the first and of
the last colour class, one sweep at beta = -ln P / dH (1 -+ 1e-8), just on
either side of acceptance.  The FP32 form of beta dH is off by 1e-7 or so, ten
times as far, so it cannot decide these sites right; the oracle's FP64 can
(its rounding is below 1e-11 of dH).  Once for any spins, where beta is about 1
and the allowance for the hardware 2^x is the wider part of the bound, and once
for spins within 1e-3 of their trials, where beta is about 1000 and the bound
is nearly all decision_band's.  On every launch that decides from FP32 values:
stencil, pipelined and z-march passes, the launches of a group of sweeps, the
neighbour tables (6, 8, 12 and more than 12 neighbours) and the batches.
"""
import math

import numpy as np
import pytest
import torch

from helpers import make_gpu, oracle_graph
from paper_2106_11286_gb300 import hs, inputs

pytestmark = pytest.mark.gpu

SEED, OFF, SITES = 31, 1e-8, 10


def second_shells(L, width):
    """A periodic bcc crystal's first `width` neighbours: 8, then 6, then 12 (CSR)."""
    near = {0: [(x - 1, y - 1, z - 1, 1) for z in (0, 1) for y in (0, 1) for x in (0, 1)],
            1: [(x, y, z, 0) for z in (0, 1) for y in (0, 1) for x in (0, 1)]}
    cube = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    far = sorted((d for d in cube if any(d)), key=lambda d: sum(map(abs, d)))[:18]
    rows = []
    for z in range(L):
        for y in range(L):
            for x in range(L):
                for b in (0, 1):
                    offs = near[b] + [(*d, b) for d in far]
                    rows.append([((((z + r) % L) * L + (y + q) % L) * L + (x + p) % L) * 2 + c
                                 for p, q, r, c in offs[:width]])
    return np.arange(len(rows) + 1, dtype=np.int64) * width, np.array(rows, dtype=np.int32).ravel()


GRAPHS = {"sc16": ("sc", (16, 16, 16), True), "sc_flat": ("sc", (20, 16, 6), True), "sc32": ("sc", (32, 32, 16), True),
          "sc_open": ("sc", (11, 9, 8), False), "bcc": ("bcc", (10, 9, 8), True), "fcc": ("fcc", (6, 5, 4), False),
          "csr14": ("csr", 8, 14), "csr26": ("csr", 8, 26)}
PARAMS = [dict(J=1.0, K=0.0, e=(0, 0, 1)), dict(J=-1.5, K=0.4, e=(1, -2, 0.5)), dict(J=0.8, K=1.2, e=(0, 0, 1))]


def _graph(orc, name):
    kind, dims, periodic = GRAPHS[name]
    if kind != "csr":
        return oracle_graph(orc, kind, dims, periodic), dict(kind=kind, dims=dims, periodic=periodic)
    rp, col = second_shells(dims, periodic)
    return oracle_graph(orc, "csr", row_ptr=rp, col=col), dict(kind="csr", row_ptr=rp, col=col)


def _trial(orc, site, colour):
    z, v, P = orc.trial_uniforms(0, seed=SEED, replica=0, site=site, rank=0, sweep_index=0, colour=colour)
    z, v = 2.0 * z - 1.0, 2.0 * v - 1.0
    r = math.sqrt((1.0 - z) * (1.0 + z))
    return np.array([r * math.cos(math.pi * v), r * math.sin(math.pi * v), z]), P


def _thresholds(orc, g, S0, params, near):
    """(site, beta) of sites of the first and the last class; near: their spins in S0 set beside their trials."""
    e = np.array(params["e"], dtype=np.float64)
    e /= np.linalg.norm(e)
    J, K = params["J"], params["K"]

    def swept(beta):
        S = S0.copy()
        orc.sweep(g, S, beta=beta, seed=SEED, sweep_index=0, mode=0, **params)
        return S

    chosen = []
    for colour in (0, g.n_colours - 1):
        sites = np.nonzero(g.colour == colour)[0]
        sites = sites[np.random.default_rng(colour).permutation(len(sites))][:6 * SITES]
        chosen.append((colour, sites))
        if near:
            for i, d in zip(sites, inputs.random_unit_spins(len(sites), 19)):
                S0[i] = _trial(orc, int(i), colour)[0] + 1e-3 * d
                S0[i] /= np.linalg.norm(S0[i])
    low, high, least = (10.0, 1e5, 1e-5) if near else (0.02, 5.0, 0.05)
    found = []
    for colour, sites in chosen:
        many = 0
        for i in sites:
            t, P = _trial(orc, int(i), colour)
            beta = low + 0.5
            for _ in range(6):  # the last class's neighbours are swept at the same beta
                S = S0 if colour == 0 else swept(beta)
                h = S[g.col[g.row_ptr[i]:g.row_ptr[i + 1]]].sum(0)
                dH = J * float((S0[i] - t) @ h) + K * (float(S0[i] @ e) ** 2 - float(t @ e) ** 2)
                if dH <= least or not low < -math.log(P) / dH < high:
                    break
                before, beta = beta, -math.log(P) / dH
                if colour == 0 or beta == before:
                    break
            else:
                continue
            if dH <= least or not low < -math.log(P) / dH < high:
                continue
            sides = [swept(beta * (1 - OFF)), swept(beta * (1 + OFF))]
            if np.any(sides[0][i] != S0[i]) and np.all(sides[1][i] == S0[i]):
                found.append((int(i), beta))
                many += 1
            if many == SITES:
                break
    assert len(found) >= SITES
    return found


def _check(S0, found, sweep):
    for i, beta in found:
        for side in (-1, 1):
            spin = sweep(beta * (1 + side * OFF), i)
            assert np.any(spin != S0[i]) == (side < 0), (i, beta, side)


LAUNCHES = [("sc16", None, None), ("sc_flat", None, None), ("sc32", None, None), ("sc32", "stencil", 0),
            ("sc32", "stencil", 3), ("sc32", "pipe", 0), ("sc32", "march", 0), ("sc_open", None, None),
            ("sc_open", "table", 0), ("bcc", None, None), ("bcc", "table", 0), ("fcc", None, None), ("csr14", None, None),
            ("csr26", None, None)]


@pytest.mark.parametrize("graph,kernel,prefetch", LAUNCHES)
@pytest.mark.parametrize("near", [False, True])
@pytest.mark.parametrize("params", PARAMS)
def test_decisions_beside_the_threshold(orc, graph, kernel, prefetch, params, near):
    g, kw = _graph(orc, graph)
    S0 = inputs.random_unit_spins(g.n, 17)
    found = _thresholds(orc, g, S0, params, near)
    first = torch.from_numpy(S0).cuda()
    for meas in (False, True):
        with make_gpu(precision="fp64", seed=SEED, **kw, **params) as lat:
            if kernel:
                lat.set_launch(kernel=kernel, prefetch=prefetch)
            lat.accumulate(meas)

            def sweep(beta, i):
                hs.hs_set_spins_device(lat.h, first)
                lat.set_sweep_counter(0)
                lat.sweep(beta, 1)
                return lat.get_spins()[i]
            _check(S0, found, sweep)


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("near", [False, True])
@pytest.mark.parametrize("params", PARAMS)
def test_batch_decisions_beside_the_threshold(orc, schedule, params, near):
    g, kw = _graph(orc, "sc16")
    S0 = inputs.random_unit_spins(g.n, 17)
    found = _thresholds(orc, g, S0, params, near)
    first = torch.from_numpy(S0).cuda()
    with make_gpu(precision="fp64", seed=SEED, **kw, **params) as lat, \
            make_gpu(precision="fp64", seed=SEED + 1, **kw, **params) as other:
        other.init()
        lat.accumulate(True)
        b = hs.hs_batch_create([lat.h, other.h])
        try:
            hs.hs_batch_set_layout(b, 1, 2, 0, schedule)

            def sweep(beta, i):
                hs.hs_set_spins_device(lat.h, first)
                lat.set_sweep_counter(0)
                hs.hs_batch_run(b, [beta, 0.5], 1)
                return lat.get_spins()[i]
            _check(S0, found, sweep)
        finally:
            hs.hs_batch_destroy(b)
