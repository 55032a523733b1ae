"""Fused steps after very many of them: the barrier's step tag has 32 bits, and a run across its wrap
equals one launch per step, list builds included."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem

pytestmark = pytest.mark.gpu


def _falling():
    # spheres at rest that fall freely, apart: the largest displacement of a step grows all the time, so
    # that one kept from an earlier step shows in the number of list builds
    g = (np.arange(12) + 0.5) * 3e-3
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    n = len(x)
    sim = dem.DEM([dem.desc(n=n, lo=(0, 0, 0), hi=(0.036, 0.036, 0.036), periodic=(True, True, False), dt=1e-5,
                            skin=0.2e-3, r_max=1e-3, E=1e7, nu=0.25, e=0.9, mu=0.5, rho=2500.0, g=(0, 0, -9.81),
                            floor=False)], max_neighbors=16)
    sim.write_state(x, np.zeros((n, 3)), np.zeros((n, 3)), np.full(n, 1e-3))
    return sim


# the wrap within the first launch, at a launch's first and last step, and in the graph's next launch
@pytest.mark.parametrize("before", [0, 1, 5, 50, 51, 70])
def test_the_barrier_tag_wraps(before):
    a, b = _falling(), _falling()
    for sim, mode in ((a, 1), (b, 2)):
        sim.set_graph_mode(mode)
        sim.set_graph(50)
        sim.step(1)
    b.test_barrier_tag(2**32 - 1 - before)
    for sim in (a, b):
        sim.step(1000)
    assert a.stats()["rebuilds"] == b.stats()["rebuilds"] > 3
    for f in (dem.POS, dem.VEL):
        assert np.array_equal(a.read(f), b.read(f)), f
