"""Which launch runs a small lattice's sweeps (hs_get_group_launch), and that
the configuration calls leave it as it was where they say that they change
nothing."""
import threading

import numpy as np
import pytest
import torch

from paper_2106_11286_gb300 import hs

pytestmark = pytest.mark.gpu

SMALL = [("sc", (16, 16, 16), "fp64"), ("sc", (24, 24, 24), "fp32"), ("sc", (18, 20, 16), "fp16"),
         ("sc", (64, 64, 64), "fp32"), ("sc", (32, 32, 32), "fp64"), ("bcc", (20, 20, 20), "fp32"),
         ("fcc", (12, 12, 12), "fp64")]


@pytest.mark.parametrize("kind,dims,precision", SMALL)
def test_a_refused_configuration_changes_nothing(kind, dims, precision):
    with hs.Lattice(kind, dims=dims, precision=precision) as lat:
        launch, group = lat.launch, lat.group_launch
        assert group["kind"] != "none" and group["ctas"] > 0
        refused = [dict(prefetch=3)] if kind != "sc" else [dict(kernel="march", tile_y=7), dict(kernel="table")]
        if precision == "fp16" and kind == "sc":
            refused.append(dict(kernel="pipe", vec_width=1))  # 2 bytes a vector
        for bad in refused:
            with pytest.raises(hs.HSError):
                lat.set_launch(**bad)
            assert (lat.launch, lat.group_launch) == (launch, group)


@pytest.mark.parametrize("kind,dims,precision", SMALL + [("sc", (200, 200, 200), "fp32"), ("sc", (20, 16, 6), "fp64")])
def test_a_saved_configuration_restores_the_launch(kind, dims, precision):
    with hs.Lattice(kind, dims=dims, precision=precision) as lat:
        launch, group = lat.launch, lat.group_launch
        lat.set_launch(**launch)
        assert (lat.launch, lat.group_launch) == (launch, group)
        lat.set_launch(**dict(kernel="stencil", order=1) if kind == "sc" else dict(kernel="table", blocks_per_sm=1))
        assert lat.group_launch["kind"] == "none"
        lat.set_launch(**launch)
        assert (lat.launch, lat.group_launch) == (launch, group)
        lat.set_launch(kernel="stencil" if kind == "sc" else "table")
        assert lat.group_launch["kind"] == "none"  # a kernel named: its launch chain
        lat.set_launch()
        assert (lat.launch, lat.group_launch) == (launch, group)


@pytest.mark.parametrize("kind,dims,precision,own", [
    ("sc", (16, 16, 16), "fp64", "slabs"), ("sc", (24, 24, 24), "fp32", "cluster"), ("sc", (48, 48, 48), "fp32", "grid"),
    ("sc", (24, 24, 24), "fp64", "grid"), ("bcc", (20, 20, 20), "fp32", "grid"), ("fcc", (12, 12, 12), "fp64", "grid"),
    ("sc", (64, 64, 64), "fp32", "none"), ("sc", (96, 96, 96), "fp32", "none"), ("sc", (96, 96, 96), "fp16", "none"),
    ("sc", (64, 64, 64), "fp64", "none"), ("bcc", (40, 40, 40), "fp32", "none"), ("fcc", (36, 36, 36), "fp32", "none")])
def test_a_stream_of_its_own_leaves_room(kind, dims, precision, own):
    """Four cooperative launches fit the device at once, or the sweeps stay a chain; the default stream's lattices,
    which run one after another, take what one fits."""
    with hs.Lattice(kind, dims=dims, precision=precision) as lat, \
            hs.Lattice(kind, dims=dims, precision=precision, stream=torch.cuda.Stream()) as beside:
        assert beside.group_launch["kind"] == own
        assert lat.group_launch["kind"] == (own if own != "none" else "grid")
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        if own == "grid":  # 128 registers a thread at most, 65536 an SM
            g = beside.group_launch
            assert 4 * g["ctas"] <= sms * (2048 // g["threads"])


@pytest.mark.parametrize("kind,dims,precision,group", [
    # work items about the clusters' lines: 4096 and 4608 of four sites, 2816 and 3840 of one
    ("sc", (32, 32, 32), "fp32", "slabs"), ("sc", (32, 32, 36), "fp32", "grid"), ("sc", (32, 32, 32), "fp16", "slabs"),
    ("sc", (32, 32, 36), "fp16", "grid"), ("sc", (22, 16, 16), "fp32", "slabs"), ("sc", (30, 16, 16), "fp32", "grid"),
    ("sc", (28, 28, 18), "fp32", "cluster"), ("sc", (28, 28, 24), "fp32", "grid"),
    ("sc", (16, 16, 18), "fp64", "slabs"), ("sc", (20, 16, 16), "fp64", "grid"), ("sc", (20, 16, 6), "fp64", "cluster"),
    # about the cooperative launch's: by width in FP32 and FP16
    ("sc", (144, 144, 144), "fp32", "grid"), ("sc", (152, 144, 144), "fp32", "none"),
    ("sc", (124, 116, 116), "fp32", "grid"), ("sc", (70, 54, 70), "fp32", "grid"), ("sc", (70, 70, 72), "fp32", "none"),
    ("sc", (136, 136, 128), "fp16", "grid"), ("sc", (136, 136, 144), "fp16", "none"),
    ("sc", (92, 92, 90), "fp16", "grid"), ("sc", (100, 100, 98), "fp16", "none"),
    ("sc", (70, 54, 70), "fp16", "grid"), ("sc", (70, 70, 72), "fp16", "none"),
    ("sc", (96, 96, 96), "fp64", "grid"), ("sc", (100, 102, 100), "fp64", "none"),
    # neighbour tables: what is resident at once in FP32 and FP16, the stated number of sites in FP64
    ("bcc", (48, 48, 48), "fp32", "grid"), ("bcc", (50, 50, 50), "fp32", "none"), ("bcc", (48, 48, 48), "fp16", "grid"),
    ("bcc", (50, 50, 50), "fp16", "none"), ("fcc", (42, 42, 42), "fp32", "grid"), ("fcc", (43, 43, 43), "fp32", "none"),
    ("bcc", (66, 66, 66), "fp64", "grid"), ("bcc", (67, 67, 67), "fp64", "none")])
def test_the_launch_by_size(kind, dims, precision, group):
    """Each kind of launch on both sides of its lines, so that the comparisons with the chain compare what they say."""
    with hs.Lattice(kind, dims=dims, precision=precision) as lat:
        assert lat.group_launch["kind"] == group, lat.group_launch


@pytest.mark.parametrize("kind,dims,precision", [
    ("sc", (70, 54, 70), "fp32"), ("sc", (70, 54, 70), "fp16"), ("sc", (92, 92, 90), "fp16"),  # several items a thread
    ("bcc", (48, 48, 48), "fp32"), ("bcc", (48, 48, 48), "fp16"), ("fcc", (42, 42, 42), "fp32"),  # every SM full
    ("bcc", (66, 66, 66), "fp64")])
def test_the_largest_groups_equal_the_chain(kind, dims, precision):
    """As in test_gpu_group.py: spins and accepted moves bit for bit, moments within the FP64 rounding of their sums."""
    got = []
    for chain in (False, True):
        with hs.Lattice(kind, dims=dims, precision=precision, seed=8, K=0.2, e=(0.3, -0.2, 1.0)) as lat:
            if chain:
                lat.set_launch(kernel="stencil" if kind == "sc" else "table")
            assert (lat.group_launch["kind"] == "none") == chain
            lat.init()
            lat.accumulate(True)
            lat.sweep(0.8, 3)
            got.append((lat.get_spins(), lat.read_accumulator()[0], lat.measure()["accept_rate"]))
    (a, m, r), (b, n, s) = got
    np.testing.assert_array_equal(a, b)
    assert r == s
    np.testing.assert_allclose(m, n, rtol=0, atol=1e-12 * max(1.0, np.abs(n).max()))


def test_lattices_side_by_side():
    """Every kind of launch at once, each lattice on a thread and a stream of its own: the chains that they have alone."""
    made = [("sc", (16, 16, 16), "fp64"), ("sc", (20, 16, 6), "fp64"), ("sc", (48, 48, 48), "fp32"), ("sc", (96, 96, 96), "fp32"),
            ("bcc", (20, 20, 20), "fp32"), ("fcc", (12, 12, 12), "fp64"), ("sc", (32, 32, 32), "fp16"), ("bcc", (40, 40, 40), "fp32")]

    def swept(lat):
        lat.init()
        lat.accumulate(True)
        lat.sweep(0.8, 130)
        return lat.get_spins(), lat.read_accumulator()

    def lattice(k, **kw):
        kind, dims, precision = made[k]
        return hs.Lattice(kind, dims=dims, precision=precision, seed=k, K=0.1, **kw)

    got, lats = [None] * len(made), [lattice(k, stream=torch.cuda.Stream()) for k in range(len(made))]

    def work(k):
        got[k] = swept(lats[k])

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(made))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(len(made)):
        lats[k].close()
        with lattice(k) as lat:
            spins, (moments, count) = swept(lat)
        np.testing.assert_array_equal(got[k][0], spins)
        assert got[k][1][1] == count == 130
        np.testing.assert_allclose(got[k][1][0], moments, rtol=0, atol=1e-12 * np.abs(moments).max())
