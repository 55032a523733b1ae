"""A written state's slots are ordered by contact count before many steps (a second list build):
the results are those of the same steps taken in calls too short for it, bit for bit, with overlaps
written before the first step, and the build is not counted."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import autotune, dem, workloads

pytestmark = pytest.mark.gpu


def _run(make, calls):
    sim = make()
    for n in calls:
        sim.step(n)
    return [sim.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA)], sim.stats()["rebuilds"]


@pytest.mark.parametrize("instances", [1, 3])
@pytest.mark.parametrize("resume", [False, True])
def test_ordered_slots_change_no_result(instances, resume):
    if resume and instances > 1:
        pytest.skip("contacts are written to single-instance contexts")
    wls = [workloads.dense_block(9, 8, 5 + k, seed=90 + k, squeeze=2e-4, vel=0.2) for k in range(instances)]
    ch = autotune.Choice(skin_factor=0.05, cell_factor=1.0, graph_steps=0, max_neighbors=32)
    first = autotune.make_context(wls, ch)
    first.step(20)
    state = [first.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA, dem.RADIUS, dem.MASS)]
    contacts = first.read_contacts(12) if resume else None

    def make():
        sim = autotune.make_context(wls, ch)
        sim.write_state(*state)
        if resume:
            sim.write_contacts(*contacts)
        return sim
    a, ra = _run(make, [80])            # ordered first
    b, rb = _run(make, [40, 40])        # too short for it
    assert ra == rb
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
