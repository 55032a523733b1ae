"""A step graph that was switched off leaves nothing behind: no fused steps are reported, and settings
changed later do not build it again."""
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
def test_a_graph_switched_off_stays_off(mode):
    sim = dem.from_workload(workloads.dense_block(6, 6, 4, seed=3))
    sim.set_graph_mode(mode)
    sim.set_graph(20)
    assert sim.stats()["graph_fused"] == (mode == 2)
    sim.step(41)
    assert sim.graph_step_kernel_ms()[1] > 0
    sim.set_graph(0)
    for change in (lambda: None, lambda: sim.set_step_lanes(2), lambda: sim.set_list_build(1),
                   lambda: sim.set_graph_mode(1), lambda: sim.set_step_lanes(1), lambda: sim.set_step_block(64)):
        change()
        assert sim.stats()["graph_fused"] == 0
        with pytest.raises(dem.DemError):
            sim.graph_step_kernel_ms()
    sim.set_graph_mode(0).set_step_block(0)
    sim.set_graph(20)                           # and comes back when asked for
    sim.step(41)
    assert sim.stats()["graph_fused"] == 1 and sim.stats()["steps"] == 82
