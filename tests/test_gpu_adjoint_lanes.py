"""Rollouts with several lanes per particle: the states that the reverse pass recomputes are the forward
ones bit for bit, so the gradients do not depend on the checkpoint interval, nor on a change of the
context's lanes after the forward pass."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu

STEPS = 40


def _grad(wl, lanes, every, block=0, then=None):
    sim = dem.from_workload(wl, max_neighbors=16)
    sim.set_step_lanes(lanes)
    sim.set_step_block(block)
    sim.rollout_forward(STEPS, every)
    if then is not None:
        sim.set_step_lanes(then)
    return sim.rollout_adjoint(np.ones((1, 2)), np.array([[0.0, 0.0]]))


# an interval of one step recomputes nothing; 7: a shorter last segment; 40: one segment
@pytest.mark.parametrize("lanes,block", [(1, 64), (1, 128), (1, 256), (1, 896), (2, 0), (4, 0), (8, 0)])
def test_gradients_do_not_depend_on_the_checkpoint_interval(lanes, block):
    # jostling spheres: contacts open and close within the rollout
    wl = workloads.dense_block(8, 8, 6, seed=95, squeeze=2e-4, vel=0.05)
    ref = _grad(wl, lanes, 1, block)
    assert np.isfinite(ref).all() and (ref != 0).all()
    for every in (4, 7, STEPS):
        assert np.array_equal(_grad(wl, lanes, every, block), ref), every


def test_lanes_set_after_the_forward_pass_do_not_change_the_gradients():
    wl = workloads.dense_block(8, 8, 6, seed=95, squeeze=2e-4, vel=0.05)
    assert np.array_equal(_grad(wl, 4, 10, then=1), _grad(wl, 4, 1))
