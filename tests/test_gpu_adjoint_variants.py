"""The reverse step's two variants (by the number of 32-slot slices: spare capacity takes the same
system to the one for large contexts) give the same gradients, for checkpoints at every step, in
segments with a remainder, and one segment."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("every", [1, 4, 9])
def test_gradients_do_not_depend_on_the_variant(every):
    wl = workloads.dense_block(8, 8, 6, seed=95, squeeze=2e-4, vel=0.05)
    out = []
    for capacity in (wl.n, 80_000):
        sim = dem.from_workload(wl, max_neighbors=16, capacity=capacity)
        sim.rollout_forward(9, every)
        out.append(sim.rollout_adjoint(np.ones((1, 2)), np.array([[0.0, 0.0]])))
    assert np.isfinite(out[0]).all() and (out[0] != 0).all()
    # the same float arithmetic; the sums over particles are in double, in the order of the slots
    np.testing.assert_allclose(out[1], out[0], rtol=1e-12)
