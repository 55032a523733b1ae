"""Neighbour lists of spheres far above and below the box: z is kept to +-2e9 units of a grid that gives
the box 2^30, so differences along z need more than 32 signed bits."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem

pytestmark = pytest.mark.gpu


# a box of height 1 and z = +-h: apart by 2 h, which is 2^32 units at h = 2; radius 0.26
@pytest.mark.parametrize("build", [0, 1])
@pytest.mark.parametrize("h,touching", [(0.2, True), (0.3, False), (0.99, False), (1.01, False), (1.5, False),
                                        (1.74, False), (1.76, False), (1.86, False)])
def test_spheres_far_apart_along_z_are_not_listed(h, touching, build):
    sim = dem.DEM([dem.desc(n=3, lo=(0, 0, 0), hi=(1, 1, 1), periodic=(False, False, False), dt=1e-6, skin=0.01,
                            r_max=0.27, E=1e7, nu=0.25, e=0.9, mu=0.5, rho=2500.0, floor=False)], max_neighbors=4)
    sim.set_list_build(build)
    x = [[0.5, 0.5, h], [0.5, 0.5, -h], [9.0, 0.5, 0.5]]
    sim.write_state(x, np.zeros((3, 3)), np.zeros((3, 3)), [0.26, 0.26, 0.26])
    assert sim.read(dem.NBR_COUNT).tolist() == ([1, 1, 0] if touching else [0, 0, 0])
    assert (sim.read(dem.FORCE)[:2, 2] != 0).all() == touching
