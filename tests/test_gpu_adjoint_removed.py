"""A rollout of a context that still holds a removed particle (parked until the next list build drops
it): the particle neither moves nor contributes, so the gradients are finite, do not depend on the
checkpoint interval, and are those of the same state without it."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu


def _rollout(every, lanes, far):
    # a block of colliding spheres, and below it a pair in contact whose lower sphere passes the removal
    # height while it touches; far: the pair's spheres apart, so that nothing touches the removed one
    b = workloads.dense_block(4, 4, 4, seed=5, squeeze=2e-4, vel=0.05)
    r, z0 = float(b.r.max()), 6e-3
    x = np.concatenate([b.x - b.x.min(0) + [5e-3, 5e-3, 12e-3],
                        [[8e-3, 8e-3, z0 + (2.5 if far else 1.999) * r], [8e-3, 8e-3, z0]]])
    z = np.zeros((2, 3))
    v, w, rr = np.concatenate([b.v, z + [0, 0, -1.0]]), np.concatenate([b.w, z]), np.concatenate([b.r, [r, r]])
    sim = dem.DEM([dem.desc(n=len(x), lo=(0, 0, 0), hi=(0.03, 0.03, 0.06), periodic=(False, False, False), dt=b.dt,
                            skin=0.5e-3, r_max=r, E=1e7, nu=0.25, e=0.9, mu=0.5, rho=2500.0, floor=False)],
                  max_neighbors=16)
    sim.write_state(x, v, w, rr)
    sim.set_step_lanes(lanes)
    sim.set_walls(z_remove=z0 - 1.5e-6)
    sim.step(int(2.0e-6 / b.dt) + 2)
    assert sim.wall_removed()[0] == 1
    sim.set_walls()                             # no removal height: rollouts are allowed again
    sim.rollout_forward(12, every)
    assert sim.counts()[0][0] == len(x)         # still among the slots
    return sim.rollout_adjoint(np.array([[1.0, 0.0]]), np.array([[0.0, 0.0]]))


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("far", [False, True])
def test_a_removed_particle_does_not_enter_the_gradients(lanes, far):
    ref = _rollout(1, lanes, far)
    assert np.isfinite(ref).all() and (ref != 0).all()
    for every in (4, 12):
        assert np.array_equal(_rollout(every, lanes, far), ref), every


def test_the_gradients_are_those_of_the_rest():
    # the block's spheres touch neither of the pair, whose upper sphere falls freely after the removal
    # (its KE does not depend on the material): near and far pairs give the block's gradients, up to
    # the order of the slots in the sums (float states, sums in double)
    np.testing.assert_allclose(_rollout(4, 1, False), _rollout(4, 1, True), rtol=1e-12)


def test_particles_marked_at_a_drain_face_do_not_enter_the_gradients():
    # a coupling call marks the top half-layer of the fine level, which touches the layer below it
    A, _, fine_wl, spec = workloads.coupling_case()
    out = []
    for every in (1, 5, 12):
        coarse = dem.from_workload(A)
        fine = dem.DEM([dem.desc_from_workload(fine_wl, capacity=fine_wl.n + 4000)])
        fine.write_state(fine_wl.x, fine_wl.v, fine_wl.w, fine_wl.r, fine_wl.m)
        cp = dem.Coupler(coarse, fine, **dict(spec, hi=(0.024, 0.024, 0.016), feed_faces=1, drain_faces=1 << 5))
        fine.step(20)
        cp.couple()
        gone = int(np.isnan(fine.read(dem.RADIUS)).sum())
        assert gone > 20
        fine.rollout_forward(12, every)
        out.append(fine.rollout_adjoint(np.array([[1.0, 0.0]]), np.array([[0.0, 0.0]])))
    assert np.isfinite(out[0]).all() and (out[0] != 0).all()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
