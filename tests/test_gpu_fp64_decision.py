"""FP64 decisions taken from FP32 values within an error bound: equal to the
oracle's outside |beta dH + ln P| < 1e-9 over several sweeps' worth of sites,
for spins that the bound covers (unit vectors, exact zeros among their
components) and for ones it does not (longer or mixed lengths, where FP64
decides), for couplings of either sign and far from 1, and beta from 0 up."""
import numpy as np
import pytest

from helpers import check_sweep_parity, make_gpu, oracle_graph
from paper_2106_11286_gb300 import hs, inputs

pytestmark = pytest.mark.gpu

GRAPHS = {"sc": ("sc", (12, 10, 8), True), "sc_v1": ("sc", (2, 6, 4), True), "bcc": ("bcc", (5, 4, 3), True),
          "fcc_open": ("fcc", (4, 3, 5), False)}


def _spins(kind, n):
    S = inputs.random_unit_spins(n, 17)
    if kind == "axis":      # along the coordinate axes: zeros, ties of dH
        S = np.eye(3)[np.arange(n) % 3] * np.where(np.arange(n) % 2, 1.0, -1.0)[:, None]
    elif kind == "long":
        S *= 3.0
    elif kind == "mixed":   # a few huge ones, whose neighbours' fields cancel
        S[::7] *= 1e12
        S[1::7] *= 1e-200
    return S


@pytest.mark.parametrize("graph", list(GRAPHS))
@pytest.mark.parametrize("kind", ["unit", "axis", "long", "mixed"])
@pytest.mark.parametrize("J,K,e,beta", [(1.0, 0.0, (0, 0, 1), 1.0), (-2.5, 0.4, (1, -2, 0.5), 0.7),
                                        (1e-3, 40.0, (0, 0, 1), 0.05), (1.0, 0.1, (0, 0, 1), 0.0),
                                        (3e40, 0.0, (0, 0, 1), 1e-40), (1.0, 0.2, (0, 1, 1), 5e3)])
def test_fp64_decisions(orc, graph, kind, J, K, e, beta):
    lat_kind, dims, periodic = GRAPHS[graph]
    g = oracle_graph(orc, lat_kind, dims, periodic)
    S0 = _spins(kind, g.n)
    params = dict(J=J, K=K, e=e)
    with make_gpu(lat_kind, dims, periodic, precision="fp64", seed=23, **params) as lat:
        lat.set_spins(S0)
        lat.accumulate(True)
        lat.sweep(beta, 1)
        got, (moments, _) = lat.get_spins(), lat.read_accumulator()
    want = S0.copy()
    band = np.zeros(g.n, dtype=np.uint8)
    orc.sweep(g, want, beta=beta, seed=23, sweep_index=0, mode=0, band=1e-9, band_site=band, **params)
    check_sweep_parity(g, S0, got, want, band, 1e-12)
    ref = orc.measure(g, got, **params)
    # every site's and bond's share rounded a few times at the size of the largest terms
    size = (abs(J) * 6 + abs(K)) * np.abs(got).max() ** 2 * g.n
    assert abs(moments[0] - ref["E"]) <= 1e-14 * size
