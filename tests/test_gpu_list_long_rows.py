"""Rows at the edges of the list build's variants by length (9, 13 and 17 candidates in registers, longer
ones ordered in shared memory) and at the list's width: clusters of k mutually near spheres, at distinct
and at equal distances, against the build that orders every row the same way and against brute force."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu

R = 1.0e-3


def _clusters(k, equal):
    # 150 clusters of k spheres within a quarter radius of each other (every row has k - 1 entries), on a
    # lattice far apart; equal: their centres on distinct points of a small grid, so that many keys are the same
    rng = np.random.default_rng(k)
    g = np.stack(np.meshgrid(np.arange(6), np.arange(5), np.arange(5), indexing="ij"), -1).reshape(-1, 3)
    pts = np.stack(np.meshgrid(np.arange(4), np.arange(4), np.arange(4), indexing="ij"), -1).reshape(-1, 3) * 0.05 * R
    off = (np.stack([pts[rng.permutation(64)[:k]] for _ in g]) if equal else
           rng.uniform(0, 0.15 * R, (len(g), k, 3)))
    x = workloads.qgrid(((g[:, None] + 0.5) * 6 * R + off).reshape(-1, 3))
    return x[rng.permutation(len(x))], np.array([6, 5, 5]) * 6 * R


def _sim(x, box, lmax, build):
    n = len(x)
    sim = dem.DEM([dem.desc(n=n, lo=(0, 0, 0), hi=box, periodic=(False, False, False), dt=1e-9, skin=0.1 * R, r_max=R,
                            E=1e5, nu=0.25, e=0.9, mu=0.5, rho=2500.0, floor=False)], max_neighbors=lmax)
    sim.set_list_build(build)
    v = np.random.default_rng(n).normal(0, 0.05, (2, n, 3))
    sim.write_state(x, v[0], v[1], np.full(n, R))
    return sim


@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("k,lmax", [(8, 16), (9, 16), (10, 16), (13, 16), (14, 16), (17, 16), (17, 17), (17, 32), (18, 17),
                                    (18, 32), (19, 18), (26, 25), (32, 32), (33, 32)])
def test_rows_of_every_length(k, lmax, equal):
    x, box = _clusters(k, equal)
    out = []
    for build in (0, 1):
        sim = _sim(x, box, lmax, build)
        got = sim.read_neighbors(32)
        assert ((got >= 0).sum(1) == k - 1).all()
        sim.step(3)
        # contacts in the rows' order, overlaps carried over a second build of the same rows
        sim.sync()
        sim.write(dem.POS, x)
        sim.step(2)
        out.append([got] + [sim.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA, dem.FORCE)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    d = x[:, None] - x[None] if len(x) < 2600 else None
    if d is not None:
        near = (d * d).sum(-1) < (2.1 * R - 1e-9) ** 2
        np.fill_diagonal(near, False)
        for i in range(0, len(x), 37):
            assert np.array_equal(out[0][0][i][out[0][0][i] >= 0], np.nonzero(near[i])[0])


@pytest.mark.parametrize("k,lmax", [(18, 16), (20, 17), (33, 20)])
@pytest.mark.parametrize("build", [0, 1])
def test_rows_wider_than_the_list_are_reported(k, lmax, build):
    x, box = _clusters(k, False)
    sim = _sim(x, box, lmax, build)
    sim.step(1)
    assert sim.status() == 2                    # DEM_ERR_CAPACITY
