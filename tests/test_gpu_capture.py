"""Calls captured by the caller into a CUDA graph of its own: a few steps and reads of a context with a
captured step graph, replayed, give what the calls themselves give, list builds included."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
def test_steps_and_reads_in_a_callers_graph(mode):
    import torch
    wl = workloads.dense_block(9, 8, 6, seed=97, vel=0.4)
    wl.skin = 0.01e-3                                   # a list build every few steps
    side = torch.cuda.Stream()
    sims = [dem.from_workload(wl, stream=side) for _ in range(2)]
    for sim in sims:
        sim.set_graph_mode(mode)
        sim.set_graph(20)
        sim.step(1)
        sim.sync()
    a, b = sims
    x, v = (torch.empty((wl.n, 3), dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        a.step(7)
        a.read(dem.POS, out=x, host=False)
        a.read(dem.VEL, out=v, host=False)
    for _ in range(6):
        g.replay()
        torch.cuda.synchronize()
        b.step(7)
        assert np.array_equal(x.cpu().numpy(), b.read(dem.POS))
        assert np.array_equal(v.cpu().numpy(), b.read(dem.VEL))
        # and a read of its own between replays, for which the lists have to be valid
        assert np.array_equal(a.read(dem.FORCE), b.read(dem.FORCE))
        assert np.array_equal(a.read_neighbors(), b.read_neighbors())
    assert b.stats()["rebuilds"] > 4
