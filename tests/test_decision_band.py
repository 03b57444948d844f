"""The bound within which FP64 lattices leave a decision to FP64 (host only):
finite at every number of neighbours, infinite where the parameters leave
FP32's range, and above the error of the FP32 form of beta dH, emulated in
numpy for spins whose fields are as large as they can be (aligned ones) and for
random ones.  numpy rounds every product and sum by itself, the kernels fuse
some: their error is no larger."""
import numpy as np
import pytest

from paper_2106_11286_gb300 import hs, inputs


def _trunc(v):
    """A double's value cut to FP32, as the kernels' bit-field conversion does."""
    f = v.astype(np.float32)
    over = np.abs(f.astype(np.float64)) > np.abs(v)
    return np.where(over, np.nextafter(f, np.float32(0)), f)


def _dot(a, b):
    return (a[:, 0] * b[:, 0] + a[:, 1] * b[:, 1]) + a[:, 2] * b[:, 2]


@pytest.mark.parametrize("width", [1, 2, 4, 6, 8, 12, 13, 14, 18, 26, 64, 300])
@pytest.mark.parametrize("J,K", [(1.0, 0.0), (-2.5, 0.7), (0.01, 3.0)])
@pytest.mark.parametrize("kind", ["aligned", "random"])
def test_band_covers_the_fp32_form(width, J, K, kind):
    n = 4000
    beta, e = 0.7, np.array([1.0, -2.0, 0.5]) / np.sqrt(5.25)
    near = inputs.random_unit_spins(n * width, 3).reshape(n, width, 3)
    s = inputs.random_unit_spins(n, 4)
    t = inputs.random_unit_spins(n, 5)
    if kind == "aligned":
        near = near * 1e-3 + s[:, None]
        near /= np.linalg.norm(near, axis=2, keepdims=True)
    h = near.sum(1)
    want = beta * (J * ((s - t) * h).sum(1) + K * ((s @ e) ** 2 - (t @ e) ** 2))
    f = np.float32
    fs, ft, fh = _trunc(s), _trunc(t), _trunc(near[:, 0])
    for k in range(1, width):
        fh = fh + _trunc(near[:, k])
    fe = e.astype(f)[None]
    se, te = _dot(fs, fe), _dot(ft, fe)
    dH = f(K) * ((se - te) * (se + te)) + f(J) * (_dot(fs, fh) - _dot(ft, fh))
    assert dH.dtype == np.float32
    band = hs.hs_decision_band(beta, J, K, width)
    assert np.isfinite(band)
    # the factor beta and its product round once more each, which decide64 covers by its factors
    assert np.abs((f(beta) * dH).astype(np.float64) - want).max() <= band + 2.4e-7 * np.abs(want).max()
    assert band < 1e-3 * beta * (abs(J) * (1 + width) ** 2 + abs(K))


def test_band_is_infinite_beyond_fp32():
    for beta, J, K in ((1.0, 1e-36, 0.0), (1.0, 1e36, 0.0), (1e-20, 1e-20, 0.0), (1.0, 1.0, 1e-35)):
        assert hs.hs_decision_band(beta, J, K, 6) == np.inf
    assert np.isfinite(hs.hs_decision_band(0.0, 1.0, 0.0, 14))
