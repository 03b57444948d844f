"""The automatic launch of small lattices (a whole group of sweeps in one
cluster, or in one cooperative launch) against the launch chain: the same
spins bit for bit, the same accepted moves, and moments that differ by FP64
rounding at most -- FP32 / FP16 sums are grouped alike, FP64 ones are added in
another order, 10^4 terms of equal sign: below 1e-12.

Sizes about the edges of the choice (2500 to 4800 work items a pass, 3.0 and 1.0 million sites),
of the warps and CTAs, of one or several items per thread, and of the vector
widths; 70 sweeps, more than one group of 64, then one more call.
"""
import numpy as np
import pytest

from paper_2106_11286_gb300 import hs

pytestmark = pytest.mark.gpu

A6 = (0.1, -0.2, 0.05, 0.03, -0.04, 0.02)
DIMS = [(2, 2, 2), (8, 4, 10), (20, 12, 18), (16, 32, 90), (30, 16, 16), (36, 16, 64), (18, 20, 16), (40, 32, 24), (10, 6, 4), (12, 10, 14), (16, 16, 16), (18, 16, 18), (32, 16, 16), (48, 10, 50), (64, 32, 16),
        (72, 64, 66)]
LARGE = [(250, 62, 64), (128, 128, 182), (256, 184, 64)]


def _run(dims, precision, e, K, tensor, meas, chain, sweeps):
    with hs.Lattice("sc", dims=dims, precision=precision, seed=5, K=K, e=e, A=A6 if tensor else None) as lat:
        if chain:
            lat.set_launch(kernel="stencil")
        lat.init()
        lat.accumulate(meas)
        for n in sweeps:
            lat.sweep(0.8, n)
        moments, count = lat.read_accumulator()
        return lat.get_spins(), moments, count, lat.measure()["accept_rate"], lat.info.sweep


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("dims", DIMS + LARGE)
@pytest.mark.parametrize("e,K,tensor,meas", [((0, 0, 1), 0.0, False, True), ((0.3, -0.2, 1.0), 0.3, False, True),
                                             ((0, 0, 1), 0.1, True, True), ((0, 0, 1), 0.1, False, False)])
def test_group_equals_the_launch_chain(precision, dims, e, K, tensor, meas):
    sweeps = (3, 1) if dims in LARGE else (70, 1)
    got = _run(dims, precision, e, K, tensor, meas, False, sweeps)
    want = _run(dims, precision, e, K, tensor, meas, True, sweeps)
    np.testing.assert_array_equal(got[0], want[0])
    assert got[2:] == want[2:]
    np.testing.assert_allclose(got[1], want[1], rtol=0, atol=1e-12 * max(1.0, np.abs(want[1]).max()))


def _table(kind, precision, chain, sweeps, meas):
    from paper_2106_11286_gb300 import inputs
    kw = dict(precision=precision, seed=7, K=0.2, e=(1, 1, 1))
    if kind == "csr":
        rp, col, mask = inputs.bcc_nanoparticle(radius=9.3, box=22, vacancy_fraction=0.05, seed=3)
        lat = hs.Lattice("csr", row_ptr=rp, col_idx=col, site_mask=mask, **kw)
    elif kind == "sc_open":
        lat = hs.Lattice("sc", dims=(31, 17, 23), periodic=False, **kw)
    elif kind == "fcc_masked":
        lat = hs.Lattice("fcc", dims=(7, 5, 9), site_mask=inputs.vacancy_mask(7 * 5 * 9 * 4, 0.1, 5), **kw)
    elif kind == "bcc_large":
        lat = hs.Lattice("bcc", dims=(60, 56, 50), **kw)
    else:
        lat = hs.Lattice("bcc", dims=(2, 2, 1), **kw)
    with lat:
        if chain:
            lat.set_launch(kernel="table", blocks_per_sm=8)
        lat.init()
        lat.accumulate(meas)
        for n in sweeps:
            lat.sweep(0.9, n)
        moments, count = lat.read_accumulator()
        return lat.get_spins(), moments, count, lat.measure()["accept_rate"], lat.info.sweep


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("kind", ["csr", "sc_open", "fcc_masked", "bcc_large", "bcc_tiny"])
@pytest.mark.parametrize("meas", [True, False])
def test_table_group_equals_the_launch_chain(precision, kind, meas):
    """The neighbour-table lattices' group launch, likewise (widths 8, 6, 12; greedy classes; vacancies)."""
    sweeps = (3, 1) if kind == "bcc_large" else (66, 1)
    got, want = (_table(kind, precision, chain, sweeps, meas) for chain in (False, True))
    np.testing.assert_array_equal(got[0], want[0])
    assert got[2:] == want[2:]
    np.testing.assert_allclose(got[1], want[1], rtol=0, atol=1e-12 * max(1.0, np.abs(want[1]).max()))
