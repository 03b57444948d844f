"""Which launch runs a small lattice's sweeps (hs_get_group_launch), and that
the configuration calls leave it as it was where they say that they change
nothing."""
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
