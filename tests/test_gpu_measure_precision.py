"""hs_measure keeps FP64's precision inside a thread, however many sites it
sums: a state whose energy (or (S.e)^2, or magnetisation) comes from the work
items of one thread of the measurement's grid, against exact rational sums.

Bound: a thread's sum rounds to FP64 three times as its parts are added and
once by J or K; its parts, in FP32, are off by less than 2^-60 of the largest
partial sum.  The sums over the grid add zeros, but for the table, where each
bond counts at both ends: there the other ends' threads add at most ten
roundings each.  So 4 and 16 units of 2^-53 of the sum of the sizes.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2106_11286_gb300 import hs, inputs

pytestmark = pytest.mark.gpu

THREAD = 12345
BLOCK = 256


def _items(n):
    """Work items of thread THREAD, of n in the whole measurement."""
    blocks = min(-(-n // BLOCK), 6 * torch.cuda.get_device_properties(0).multi_processor_count)
    return np.arange(THREAD, n, blocks * BLOCK)


def _ordered(n, seed):
    """Unit vectors near z, as an ordered magnet's, in FP32."""
    S = np.random.default_rng(seed).normal(0.0, 0.25, (n, 3))
    S[:, 2] += 1.0
    return (S / np.linalg.norm(S, axis=1, keepdims=True)).astype(np.float32)


def _exact(values):
    return sum((Fraction(float(v)) for v in values), Fraction(0))


DIMS = (256, 256, 512)


def _thread_sites(colour):
    Lx, Ly, _ = DIMS
    nxv = Lx // 8  # four sites of one colour an item
    t = _items(DIMS[0] * DIMS[1] * DIMS[2] // 8)
    row, xv = t // nxv, t % nxv
    z, y = row // Ly, row % Ly
    x = 2 * (4 * xv[:, None] + np.arange(4)) + ((colour + y + z) % 2)[:, None]
    return x.ravel(), np.repeat(y, 4), np.repeat(z, 4)


def _measure(S, precision, **kw):
    with hs.Lattice("sc", dims=DIMS, precision=precision, **kw) as lat:
        hs.hs_set_spins_device(lat.h, torch.from_numpy(S).to("cuda", torch.float64).contiguous())
        return lat.measure()


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_bonds_of_one_thread(precision):
    Lx, Ly, Lz = DIMS
    S = np.zeros((Lz, Ly, Lx, 3), np.float32)
    z, y, x = np.ogrid[:Lz, :Ly, :Lx]
    even = (x + y + z) % 2 == 0
    S[even] = _ordered(int(even.sum()), 1)
    tx, ty, tz = _thread_sites(1)
    S[tz, ty, tx] = _ordered(len(tx), 2)
    if precision == "fp16":
        S = S.astype(np.float16).astype(np.float32)
    got = _measure(S, precision, K=0.0)
    terms = []
    for a, b, c in zip(tx, ty, tz):
        for p, q, r in ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)):
            n = S[(c + r) % Lz, (b + q) % Ly, (a + p) % Lx]
            terms += [Fraction(float(u)) * Fraction(float(v)) for u, v in zip(S[c, b, a], n)]
    assert len(tx) >= 64
    assert abs(Fraction(got["E"]) + sum(terms)) <= 4 * Fraction(1, 2**53) * sum(map(abs, terms))


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
def test_squares_and_components_of_one_thread(precision):
    S = np.zeros((DIMS[2], DIMS[1], DIMS[0], 3), np.float32)
    own = []
    for colour in (0, 1):
        tx, ty, tz = _thread_sites(colour)
        S[tz, ty, tx] = _ordered(len(tx), 3 + colour)
        if precision == "fp16":
            S[tz, ty, tx] = S[tz, ty, tx].astype(np.float16)
        own.append(S[tz, ty, tx])
    own = np.concatenate(own)
    got = _measure(S, precision, J=0.0, K=1.0)
    k = sum(Fraction(float(v)) ** 2 for v in own[:, 2])
    assert abs(Fraction(got["E"]) + k) <= 4 * Fraction(1, 2**53) * k
    n = DIMS[0] * DIMS[1] * DIMS[2]
    for q in range(3):
        size = _exact(np.abs(own[:, q])) / n
        assert abs(Fraction(float(got["M"][q])) - _exact(own[:, q]) / n) <= 4 * Fraction(1, 2**53) * size


def test_table_bonds_of_one_thread():
    L = 128
    n = 2 * L**3
    S = np.zeros((L**3, 2, 3), np.float32)  # natural order: corner, centre; renumbered: corners, then centres
    S[:, 0] = _ordered(L**3, 5)
    t = _items(n)
    cells = t[t >= L**3] - L**3
    S[cells, 1] = _ordered(len(cells), 6)
    with hs.Lattice("bcc", dims=(L, L, L), precision="fp32", K=0.0) as lat:
        lat.set_spins(S.reshape(-1, 3).astype(np.float64))
        got = lat.measure()
    terms = []
    for c in cells:
        x, y, z = c % L, c // L % L, c // L**2
        for d in range(8):
            m = S[(((z + (d >> 2)) % L) * L + (y + (d >> 1 & 1)) % L) * L + (x + (d & 1)) % L, 0]
            terms += [Fraction(float(u)) * Fraction(float(v)) for u, v in zip(S[c, 1], m)]
    assert abs(Fraction(got["E"]) + sum(terms)) <= 16 * Fraction(1, 2**53) * sum(map(abs, terms))


@pytest.mark.parametrize("kind,dims", [("sc", (6, 4, 2)), ("sc", (16, 10, 4)), ("bcc", (4, 4, 4))])
@pytest.mark.parametrize("K", [0.0, 0.3])
def test_measure_below_fp32_products(kind, dims, K):
    """Components whose products FP32 cannot hold (no unit vectors): summed in FP64."""
    with hs.Lattice(kind, dims=dims, K=K, precision="fp32") as lat, \
            hs.Lattice(kind, dims=dims, K=K, precision="fp64") as wide:
        n = lat.info.n_sites
        S = (inputs.random_unit_spins(n, 4) * 1e-25).astype(np.float32).astype(np.float64)
        for m in (lat, wide):
            m.set_spins(S)
        got, want = lat.measure(), wide.measure()
    assert abs(got["E"] - want["E"]) <= 1e-13 * 8e-50 * n
    np.testing.assert_allclose(got["M"], want["M"], rtol=1e-13)
