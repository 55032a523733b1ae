"""The list build by cubes of cells against brute force in exact integers, over grids and occupancies
where its windows, images and cube shapes change; and rows of equal keys in the same order whatever
the scan order."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu


def _sim(x, r, box, periodic, r_max, skin, lmax=32):
    n = len(r)
    sim = dem.DEM([dem.desc(n=n, lo=(0, 0, 0), hi=box, periodic=periodic, dt=1e-6, skin=skin, r_max=r_max, E=1e7,
                            nu=0.25, e=0.9, mu=0.5, rho=2500.0, floor=False)], max_neighbors=lmax)
    sim.write_state(x, np.zeros((n, 3)), np.zeros((n, 3)), r)
    return sim


def _brute(sim, x, r, box, periodic, skin):
    q = sim.info()["q"]
    X, R, S = np.rint(x / q).astype(np.int64), np.rint(r / q).astype(np.int64), int(round(skin / q))
    rows = []
    for i in range(len(r)):
        d = X - X[i]
        for a in range(3):
            if periodic[a]:
                L = int(round(box[a] / q))
                h = L // 2
                d[:, a] = np.where(d[:, a] > h, d[:, a] - L, np.where(d[:, a] < -h, d[:, a] + L, d[:, a]))
        cut = R + R[i] + S
        near = (d * d).sum(1) < cut * cut
        near[i] = False
        rows.append(np.nonzero(near)[0])
    return rows


# box in cells of 2 r_max + skin (a little more, so that the count is as given), periodic in x, y;
# particles per cell.  (3, 3, 3): a cube wider than the grid, images on both sides.  (70, 1, 1): cubes
# of 64 cells in a row.  (1, 1, 1): one cell.  (4, 5, 2) at 40 a cell: several windows and more
# particles in a cube than have their cell noted.  (9, 9, 9): several cubes with partial ones.
@pytest.mark.parametrize("cells,per,fill", [
    ((3, 3, 3), (True, True, False), 6), ((70, 1, 1), (True, False, False), 3), ((1, 1, 1), (False, False, False), 30),
    ((4, 5, 2), (True, True, False), 40), ((9, 9, 9), (False, True, False), 2), ((2, 70, 1), (False, True, False), 2)])
def test_cube_lists_equal_brute_force(cells, per, fill):
    rng = np.random.default_rng(7)
    r_max, skin = 1.0e-3, 0.25e-3
    w = 2 * r_max + skin
    box = tuple(workloads.qgrid(np.array(cells) * w * 1.01))
    n = int(np.prod(cells) * fill)
    x = workloads.qgrid(rng.uniform(0, 1, (n, 3)) * np.array(box) * 0.999)
    x[rng.integers(0, n, n // 20 + 1), 2] += 0.3 * box[2]                       # above the box: the top cell layer
    small = 0.25e-3 if fill > 10 else 0.45e-3                                   # rows within 32 entries
    r = workloads.qgrid(rng.uniform(0.5 * small, small, n))
    if fill > 10:
        skin = workloads.qgrid(0.05e-3)
        r_max = 0.5 * (w - skin)
    sim = _sim(x, r, box, per, r_max, float(workloads.qgrid(skin)))
    assert sim.info()["ncell"] == cells
    want = _brute(sim, x, r, box, per, float(workloads.qgrid(skin)))
    assert 20 < sum(len(v) for v in want) and max(len(v) for v in want) <= 32
    for build in (0, 1):
        sim.set_list_build(build)
        sim.write(dem.POS, x)
        got = sim.read_neighbors()
        for i in range(n):
            assert np.array_equal(got[i][got[i] >= 0], want[i]), (build, i)


# a perfect lattice: every key of a shell equal, so the row's order is the IDs'; 6, 12 and 26 entries
@pytest.mark.parametrize("skin", [0.2e-3, 1.0e-3, 1.6e-3])
def test_rows_of_equal_keys_do_not_depend_on_the_scan_order(skin):
    g = np.arange(8) * 1.999e-3 + 1.0e-3
    x = workloads.qgrid(np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3))
    rng = np.random.default_rng(3)
    x = x[rng.permutation(len(x))]
    v, w = rng.normal(0, 0.05, x.shape), rng.normal(0, 20, x.shape)
    out = []
    for build in (0, 1):
        sim = _sim(x, np.full(len(x), 1.0e-3), (0.02, 0.02, 0.02), (False, False, False), 1.0e-3, skin)
        sim.set_list_build(build)
        sim.write(dem.VEL, v).write(dem.OMEGA, w)
        sim.step(30)
        out.append([sim.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_row_wider_than_the_list_is_reported():
    rng = np.random.default_rng(5)
    x = workloads.qgrid(rng.uniform(0, 2e-3, (60, 3)) + 1e-3)
    sim = _sim(x, np.full(60, 1.0e-3), (0.01, 0.01, 0.01), (False, False, False), 1.0e-3, 0.2e-3, lmax=8)
    sim.step(1)
    assert sim.status() == 2                    # DEM_ERR_CAPACITY
