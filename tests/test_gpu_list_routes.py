"""The list build's routes: cubes of cells in shared memory, and a thread per particle for crowded cubes,
for sparse ones where there are many, and for cubes with too much around them.  Rows against brute force in exact integers, and runs with
list builds (tangential overlaps carried over) against the build that takes one route for all."""
import numpy as np
import pytest

from paper_1705_03850_gb300 import dem, workloads

pytestmark = pytest.mark.gpu

D = 1.0e-3


def _system(kind):
    """x, r, box, periodic, r_max: spheres of diameter about D."""
    rng = np.random.default_rng(11)

    def lattice(k, s, jit):
        g = np.stack(np.meshgrid(*[np.arange(m) for m in k], indexing="ij"), -1).reshape(-1, 3)
        return (g + 0.5 + rng.uniform(-jit, jit, g.shape)) * s

    r_max = 0.5 * D
    if kind == "sparse":                # about one particle a cube, some 20,000 cubes
        x, box = lattice((28, 27, 26), 4 * D, 0.4), (28 * 4 * D, 27 * 4 * D, 26 * 4 * D)
        x[::3] = x[1::3][:len(x[::3])] + rng.normal(0, 0.5 * D, (len(x[::3]), 3))     # and close pairs
    elif kind == "few sparse":          # as that, too few cubes for the other route
        x, box = lattice((9, 8, 7), 4 * D, 0.4), (9 * 4 * D, 8 * 4 * D, 7 * 4 * D)
        x[::3] = x[1::3][:len(x[::3])] + rng.normal(0, 0.5 * D, (len(x[::3]), 3))
    elif kind == "crowded":             # cells of three diameters: 27 particles a cell
        x, box, r_max = lattice((24, 24, 20), D, 0.1), (24 * D, 24 * D, 20 * D), 1.4 * D
    else:                               # "mixed": a dense bed, a crowded clump and a sparse cloud above
        bed = lattice((40, 40, 10), D, 0.1)
        cloud = lattice((26, 26, 24), 3.0 * D, 0.4) + [0, 0, 14 * D]
        clump = lattice((24, 24, 24), 0.3 * D, 0.3) + [16 * D, 16 * D, 90 * D]
        x, box = np.concatenate([bed, cloud, clump]), (79 * D, 79 * D, 110 * D)
    x = np.clip(x, 0, np.array(box) * (1 - 1e-9))
    x = workloads.qgrid(x[rng.permutation(len(x))])
    small = 0.15 * D if kind == "mixed" else 0.5 * D
    r = np.where(x[:, 2] > 88 * D, 0.1 * D, rng.uniform(0.45 * D, 0.5 * D, len(x))) if kind == "mixed" else \
        rng.uniform(0.9 * small, small, len(x))
    return x, workloads.qgrid(r), box, (True, True, False), r_max


def _sim(s, skin=0.1 * D, dt=1e-6):
    x, r, box, per, r_max = s
    n = len(r)
    sim = dem.DEM([dem.desc(n=n, lo=(0, 0, 0), hi=box, periodic=per, dt=dt, skin=skin, r_max=r_max, E=1e6, nu=0.25,
                            e=0.9, mu=0.5, rho=2500.0, floor=False)], max_neighbors=32)
    sim.write_state(x, np.zeros((n, 3)), np.zeros((n, 3)), r)
    return sim


KINDS = ["sparse", "few sparse", "crowded", "mixed"]


@pytest.mark.parametrize("kind", KINDS)
def test_rows_equal_brute_force(kind):
    s = _system(kind)
    x, r, box, per, _ = s
    sim = _sim(s)
    got = sim.read_neighbors()
    q = sim.info()["q"]
    X, R, S = np.rint(x / q).astype(np.int64), np.rint(r / q).astype(np.int64), int(round(0.1 * D / q))
    L = [int(round((h - l) / q)) for l, h in zip(sim.info()["lo"], sim.info()["hi"])]
    rows = np.random.default_rng(1).integers(0, len(r), 300)
    total = 0
    for i in rows:
        d = X - X[i]
        for a in range(3):
            if per[a]:
                d[:, a] = (d[:, a] + L[a] // 2) % L[a] - L[a] // 2
        cut = R + R[i] + S
        near = (d * d).sum(1) < cut * cut
        near[i] = False
        want = np.nonzero(near)[0]
        total += len(want)
        assert np.array_equal(got[i][got[i] >= 0], want), i
    assert total > 100


@pytest.mark.parametrize("kind", KINDS)
def test_runs_across_list_builds_equal_the_other_build(kind):
    s = _system(kind)
    n = len(s[1])
    v = np.random.default_rng(2).normal(0, 0.3, (n, 3))
    out = []
    for build in (0, 1):
        sim = _sim(s, dt=2e-6)
        sim.set_list_build(build)
        sim.write(dem.VEL, v)
        sim.step(60)
        assert sim.stats()["rebuilds"] > 1 and sim.stats()["contacts"] > 20
        partner, xi = sim.read_contacts()
        out.append([sim.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA)] + [partner, xi])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_instances_of_every_kind_in_one_context_equal_the_other_build():
    # the routes are chosen for the context as a whole
    systems = [_system(k) for k in ("few sparse", "crowded", "mixed")] + [_system("few sparse") for _ in range(9)]
    out = []
    for build in (0, 1):
        ds = [dem.desc(n=len(r), lo=(0, 0, 0), hi=box, periodic=per, dt=2e-6, skin=0.1 * D, r_max=r_max, E=1e6, nu=0.25,
                       e=0.9, mu=0.5, rho=2500.0, floor=False) for x, r, box, per, r_max in systems]
        sim = dem.DEM(ds, max_neighbors=32)
        sim.set_list_build(build)
        x, r = np.concatenate([s[0] for s in systems]), np.concatenate([s[1] for s in systems])
        v = np.random.default_rng(3).normal(0, 0.3, x.shape)
        sim.write_state(x, v, np.zeros_like(x), r)
        sim.step(60)
        assert sim.stats()["rebuilds"] > len(systems) and sim.stats()["contacts"] > 20
        out.append([sim.read(f) for f in (dem.POS, dem.VEL, dem.OMEGA, dem.NBR_COUNT)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
