"""hs_measure against plain FP64 numpy sums of the state it measures, over
every vector width of the sc kernel (Lx/2 odd, and divisible by 2, 4 and 8),
axes with the FP32-pair and the FP64 on-site terms, the tensor, and states
outside FP32's range.

Tolerance: FP32 / FP16 sums run in pairs of floats (48 bits), so a site's
share of at most 6 + |K| + |A| < 8 is off by at most 40 operations x 2^-48 x 8
< 1.2e-12, FP64 by 40 x 2^-53 x 8; both stay below 1.2e-12 per site.
"""
import numpy as np
import pytest

from paper_2106_11286_gb300 import hs, inputs

pytestmark = pytest.mark.gpu

A6 = (0.1, -0.2, 0.05, 0.03, -0.04, 0.02)
FULL = np.array([[A6[0], A6[3], A6[4]], [A6[3], A6[1], A6[5]], [A6[4], A6[5], A6[2]]])


def _numpy(S, dims, K, e, tensor):
    Lx, Ly, Lz = dims
    s = S.reshape(Lz, Ly, Lx, 3)
    bonds = sum((s * np.roll(s, 1, axis=a)).sum() for a in range(3))
    e = np.asarray(e) / np.linalg.norm(e)
    onsite = K * ((S @ e) ** 2).sum()
    if tensor:
        onsite += np.einsum("ia,ab,ib->", S, FULL, S)
    return -bonds - onsite, S.sum(axis=0) / len(S)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("dims", [(2, 2, 2), (6, 4, 2), (4, 6, 8), (8, 2, 6), (16, 10, 4), (48, 34, 38)])
@pytest.mark.parametrize("K,e,tensor", [(0.0, (0, 0, 1), False), (0.3, (0, 0, 1), False),
                                        (0.3, (0.3, -0.2, 1.0), False), (0.1, (0, 0, 1), True)])
def test_measure_matches_fp64_sums(precision, dims, K, e, tensor):
    n = dims[0] * dims[1] * dims[2]
    S = inputs.random_unit_spins(n, 3)
    with hs.Lattice("sc", dims=dims, K=K, e=e, precision=precision, A=A6 if tensor else None) as lat:
        lat.set_spins(S)
        got, stored = lat.measure(), lat.get_spins()
    E, M = _numpy(stored, dims, K, e, tensor)
    assert abs(got["E"] - E) <= 1.2e-12 * n
    np.testing.assert_allclose(got["M"], M, rtol=0, atol=1.2e-12)


@pytest.mark.parametrize("dims", [(6, 4, 2), (16, 10, 4)])
def test_measure_beyond_fp32_products(dims):
    """Components whose products overflow FP32 (no unit vectors): summed in FP64."""
    n = dims[0] * dims[1] * dims[2]
    S = (inputs.random_unit_spins(n, 4) * 1e25).astype(np.float32).astype(np.float64)
    with hs.Lattice("sc", dims=dims, K=0.3, precision="fp32") as lat:
        lat.set_spins(S)
        got = lat.measure()
    E, M = _numpy(S, dims, 0.3, (0, 0, 1), False)
    assert got["E"] == pytest.approx(E, rel=1e-12, abs=1e-12 * 8e50 * n)
    np.testing.assert_allclose(got["M"], M, rtol=0, atol=1e13)
