"""The grid barrier between the passes of a small lattice's group launch is
bounded (hs_sweep; the batch's is in test_gpu_failure.py).  The hook makes the
first wait of a call run out; the call's other launches, queued behind it, must
then leave at once with their folds: the error comes after about one wait, not
one for every 64 sweeps, and once; no sweep is counted; and the handle sweeps
on as a new one does.
"""
import time

import numpy as np
import pytest

from paper_2106_11286_gb300 import hs

pytestmark = pytest.mark.gpu

LATTICES = [("sc", (64, 64, 64), "fp32"), ("sc", (64, 64, 64), "fp64"), ("sc", (64, 64, 64), "fp16"),
            ("fcc", (12, 12, 12), "fp64"), ("fcc", (12, 12, 12), "fp32")]


@pytest.mark.parametrize("kind,dims,precision", LATTICES)
def test_sweep_barrier_timeout_drains_and_recovers(kind, dims, precision):
    make = lambda: hs.Lattice(kind, dims=dims, precision=precision, seed=4, K=0.1)  # noqa: E731
    with make() as lat, make() as new:
        lat.init()
        lat.accumulate(True)
        lat.sweep(0.8, 2)
        lat.read_accumulator()
        hs.hs_inject_timeout(lat.h)
        t0 = time.time()
        lat.sweep(0.8, 10 * 64)  # ten launches: one wait each would be ten seconds
        with pytest.raises(hs.HSError) as ei:
            lat.read_accumulator()
        assert ei.value.code == -5
        assert time.time() - t0 < 4
        assert lat.read_accumulator()[1] == 2  # reported once; the first call's sweeps alone
        # the next call runs as on a new handle
        for m in (lat, new):
            m.init()
            m.accumulate(True)
            m.reset_accumulator()
            m.set_sweep_counter(0)
            m.sweep(0.8, 70)
        (a, n), (b, k) = lat.read_accumulator(), new.read_accumulator()
        assert n == k == 70 and np.array_equal(a, b)
        assert np.array_equal(lat.get_spins(), new.get_spins())
