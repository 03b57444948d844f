"""hs_get_spins_device over every vector width, partial tiles, slabs' plane
offsets, a buffer that is only 8-byte aligned, and values at the edges of the
integer widening: each value comes back as the FP64 number it is stored as."""
import numpy as np
import pytest
import torch

from paper_2106_11286_gb300 import hs, inputs

pytestmark = pytest.mark.gpu

STORE = {"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}


@pytest.mark.parametrize("precision", list(STORE))
@pytest.mark.parametrize("dims", [(2, 2, 2), (6, 4, 2), (4, 6, 8), (8, 2, 6), (16, 10, 4), (64, 34, 38)])
@pytest.mark.parametrize("offset", [0, 1])
def test_export_returns_the_stored_values(precision, dims, offset):
    n = dims[0] * dims[1] * dims[2]
    S = inputs.random_unit_spins(n, 7).astype(STORE[precision])
    edge = np.array([0.0, -0.0, 1e-45, -3e-39, 1.1754944e-38, np.inf, -np.inf, np.nan, 1.0, -1.0, 6e-8, 3e-5],
                    dtype=np.float64)
    with np.errstate(over="ignore"):
        S.reshape(-1)[:12] = edge.astype(STORE[precision])
    want = S.astype(np.float64)
    with hs.Lattice("sc", dims=dims, precision=precision) as lat:
        lat.set_spins(want)
        buf = torch.full((3 * n + 2,), 7.0, dtype=torch.float64, device="cuda")
        hs.hs_get_spins_device(lat.h, buf[offset:offset + 3 * n])
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
    assert (got[:offset] == 7.0).all() and (got[offset + 3 * n:] == 7.0).all()
    back = got[offset:offset + 3 * n]
    np.testing.assert_array_equal(back, want.reshape(-1))
    np.testing.assert_array_equal(np.signbit(back), np.signbit(want.reshape(-1)))


@pytest.mark.parametrize("z0,nz", [(0, 3), (3, 5), (7, 1)])
def test_export_of_a_slab(z0, nz):
    dims = (24, 6, 8)
    S = inputs.random_unit_spins(24 * 6 * nz, 9).astype(np.float32).astype(np.float64)
    with hs.Slab(dims, z0, nz, precision="fp32") as slab:
        slab.set_spins(S)
        np.testing.assert_array_equal(slab.get_spins(), S)
