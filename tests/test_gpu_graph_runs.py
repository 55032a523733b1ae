"""Step graphs with a conditional list build per run of several steps, and graphs run for fewer
steps than they were built for, compute exactly what launches of their own compute, with list
builds falling anywhere within a run and reads (which need valid lists) in between."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import autotune, dem, workloads

pytestmark = pytest.mark.gpu


# 1, 4, 5, 6 steps per graph: below, at and above a run; 23: a last run of three.  The step counts
# leave remainders that the graph runs in part (13 of 23) and that are launched alone (1 of 23).
@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("graph", [1, 4, 5, 6, 23])
def test_graph_runs_and_remainders_equal_single_launches(graph, mode):
    # a skin of 1/200 d: a list build every few steps
    wls = [workloads.dense_block(*sh, seed=70 + k, vel=0.4) for k, sh in enumerate([(9, 7, 5), (5, 6, 4)])]
    ch = autotune.Choice(skin_factor=0.005, cell_factor=1.0, graph_steps=graph, max_neighbors=32)
    a, b = autotune.make_context(wls, ch), autotune.make_context(wls, ch)
    b.set_graph_mode(mode)
    b.set_graph(graph)
    for n in (30, 24, 13, 1, 46):
        for sim in (a, b):
            sim.step(n)
        for f in (dem.POS, dem.VEL, dem.OMEGA):
            assert np.array_equal(a.read(f), b.read(f)), (n, f)
    sa, sb = a.stats(), b.stats()
    assert sa["rebuilds"] == sb["rebuilds"] > 10
    assert sb["graph_fused"] == (mode == 2)


def test_step_kernel_times_cover_the_steps_of_the_last_launch():
    sim = dem.from_workload(workloads.dense_block(8, 8, 6, seed=73))
    sim.set_graph_mode(1)
    sim.set_graph(20)
    sim.step(41)                                # 1 alone, then 20 and 20
    ms, count = sim.graph_step_kernel_ms()
    assert count == 4 and 0 < ms < 100
    sim.step(7)                                 # 7 of 20: the runs of steps 0-4 and 5-9
    ms, count = sim.graph_step_kernel_ms()
    assert count == 2 and 0 < ms < 100


# one warp to several units per block: 40 and 512 slots (blocks of 64 threads), 12,000 and 40,000
# (wide blocks; with 8 lanes more slices than the resident warps), and spare capacity
@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("shape,spare", [((5, 4, 2), 0), ((8, 8, 8), 5000), ((30, 20, 20), 0), ((40, 40, 25), 30000)])
def test_fused_blocks_of_every_width_equal_one_launch_per_step(shape, spare, lanes):
    wl = workloads.dense_block(*shape, seed=80, vel=0.4)
    wl.skin = 0.02e-3
    runs = []
    for mode in (1, 2):
        sim = dem.from_workload(wl, capacity=wl.n + spare, max_neighbors=20)
        sim.set_step_lanes(lanes)
        sim.set_graph_mode(mode)
        sim.set_graph(40)
        sim.step(121)
        runs.append(sim)
    a, b = runs
    assert a.stats()["rebuilds"] == b.stats()["rebuilds"] > 2
    for f in (dem.POS, dem.VEL, dem.OMEGA):
        assert np.array_equal(a.read(f), b.read(f)), f
