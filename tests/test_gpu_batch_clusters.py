"""FP64 batches of few small members, each swept by a cluster of its own:
uneven sizes (one work item per thread and several, partial warps, empty
CTAs), tilted and z axes, K = 0 and not, equilibration counted apart, runs
longer than one group of 32 sweeps -- the members' spins equal hs_sweep's bit
for bit, their moments to FP64 rounding (10^4 terms of equal sign: 1e-12)."""
import numpy as np
import pytest

from paper_2106_11286_gb300 import hs

pytestmark = pytest.mark.gpu


def _members(dims):
    axes = [(0, 0, 1), (0.3, -0.2, 1.0), (1, 1, 1)]
    return [hs.Lattice("sc", dims=d, precision="fp64", seed=3, replica=r, K=0.1 * (r % 3), e=axes[r % 3])
            for r, d in enumerate(dims)]


@pytest.mark.parametrize("dims", [[(4, 2, 2)], [(8, 8, 8)] * 3, [(24, 24, 24), (4, 2, 2), (12, 10, 6)],
                                  [(16, 16, 16)] * 48, [(12, 12, 12)] * 76, [(24, 24, 28)] * 20])
@pytest.mark.parametrize("n_sweeps,n_equil", [(1, 0), (40, 33), (0, 5)])
def test_cluster_batch_equals_single_lattices(dims, n_sweeps, n_equil):
    betas = [0.5 + 0.7 * r / len(dims) for r in range(len(dims))]
    a, c = _members(dims), _members(dims)
    for m in a + c:
        m.init()
    batch = hs.hs_batch_create([m.h for m in a])
    try:
        assert hs.hs_batch_get_layout(batch)["schedule"] == (2 if len(dims) > 1 else 0)  # one warp: no cluster
        hs.hs_batch_run(batch, betas, n_sweeps, n_equil)
        for x, z, beta in zip(a, c, betas):
            z.sweep(beta, n_equil)
            z.accumulate(True)
            z.sweep(beta, n_sweeps)
            assert np.array_equal(x.get_spins(), z.get_spins())
            (mx, cx), (mz, cz) = x.read_accumulator(), z.read_accumulator()
            assert cx == cz == n_sweeps
            np.testing.assert_allclose(mx, mz, rtol=0, atol=1e-12 * max(1.0, np.abs(mz).max()))
            assert x.info.sweep == z.info.sweep == n_sweeps + n_equil
    finally:
        hs.hs_batch_destroy(batch)
        for m in a + c:
            m.close()
