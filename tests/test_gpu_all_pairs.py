"""Lennard-Jones forces by all pairs (GPU), which stand in wherever the Verlet
lists do not hold: after lbmd_set_particles until the next re-ordering, once a
particle has moved by half the skin, and for a particle with more neighbours
than a list takes.  Same bits as with the lists.

In the first test the lists that exist belong to other positions (the sites
are dealt out anew among the ids), so using them in place of all pairs would
give other forces altogether."""
import numpy as np
import pytest

from paper_1610_02733_gb300 import inputs, lbmd

pytestmark = pytest.mark.gpu

SHAPE = (17, 16, 14)
# ids in one block, in a cluster of blocks, in a grid of blocks (a warp per
# particle, 8 per block), more than one tile of staged ids (FP32 1024, FP64 512)
SIZES = {"fp32": [5, 60, 300, 1300], "fp64": [5, 60, 300, 700]}
CASES = [(p, n) for p in ("fp32", "fp64") for n in SIZES[p]]


def _sites(n, seed, spacing=1.3, jitter=0.1):
    axes = [np.arange(int(L / spacing)) * (L / int(L / spacing)) for L in SHAPE]
    grid = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, 3)
    rng = np.random.default_rng(seed)
    return grid[rng.permutation(grid.shape[0])[:n]] + jitter * rng.random((n, 3))


def _context(pos, vel, **kw):
    n = pos.shape[0]
    a = dict(variant="B", n_sub=6, kT=1e-4, zeta=0.3, seed=9, max_particles=n, max_bonds=n)
    a.update(kw)
    g = lbmd.LBMD(*SHAPE, **a)
    g.add_particles(pos, vel)
    return g


def _forces(g, n, sigma=1.0, r_cut=1.6):
    g.set_lj(2e-3, sigma, r_cut)
    if n >= 4:
        g.add_fene_bonds([(i, i + 1) for i in range(0, n - 1, 4)], 1e-4, 60.0)


def _state(g):
    out = (g.populations(), g.node_field(), *g.particles())
    g.close()
    assert all(np.isfinite(x).all() for x in out)
    return out


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("variant,integrator", [("A", "start"), ("B", "start"), ("B", "half_step"), ("C", "start")])
@pytest.mark.parametrize("precision,n", CASES)
def test_lists_of_other_positions(precision, n, variant, integrator):
    # two positions far apart in id: the sites of seed 1 and of seed 2
    kw = dict(precision=precision, variant=variant, integrator=integrator)
    vel = inputs.maxwell_velocities(n, 1e-3, 5)
    runs = []
    for spread, fresh, graph in (("rows", True, False), ("auto", False, True), ("rows", False, False),
                                 ("atomic", False, True)):
        g = _context(_sites(n, 2 if fresh else 1), vel, spread=spread, **kw)
        _forces(g, n)
        if not fresh:  # the lists of the sites of seed 1, void from here to the end of the cycle
            g.set_particles(_sites(n, 2), vel)
        g.run_cycles(1) if graph else g.cycle(1)
        runs.append(_state(g))
    for r in runs[1:]:
        _same(r, runs[0])


@pytest.mark.parametrize("precision,n", CASES)
def test_skin_spent_within_a_cycle(precision, n):
    # layers of particles in z that slide past one another by 1.2 in a cycle:
    # the lists are void after 0.4 of it, and pairs come within the cut-off that
    # no list holds
    pos = _sites(n, 3, jitter=0.0)
    layer = np.round(pos[:, 2] / (SHAPE[2] / int(SHAPE[2] / 1.3))).astype(int)
    pos = pos + np.random.default_rng(4).uniform(-0.03, 0.03, (n, 3))
    vel = np.zeros((n, 3))
    vel[:, 0] = np.where(layer % 2 == 0, 0.6, -0.6)
    runs = []
    for spread, void, graph in (("rows", True, False), ("auto", False, True), ("rows", False, False),
                                ("auto", True, True)):
        g = _context(pos, vel, spread=spread, precision=precision, n_sub=8, zeta=0.01)
        _forces(g, n)
        for c in range(3):
            if void and (c == 0 or precision == "fp32"):
                # all pairs from the cycle's first step on (the particles' own
                # positions: in FP64 exact only as they were given)
                g.set_particles(pos=g.particles()[0] if c else pos)
            g.run_cycles(1) if graph else g.cycle(1)
        runs.append(_state(g))
    for r in runs[1:]:
        _same(r, runs[0])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("variant", ["A", "B"])
def test_more_neighbours_than_a_list_takes(precision, variant):
    # 150 particles within the range of one another, among others with lists
    k = np.stack(np.meshgrid(np.arange(6), np.arange(5), np.arange(5), indexing="ij"), -1).reshape(-1, 3)
    ball = 7.0 + 0.25 * k + np.random.default_rng(6).uniform(-0.02, 0.02, k.shape)
    rest = _sites(400, 7)
    rest = rest[np.abs(rest - 7.6).max(axis=1) > 2.0]
    pos = np.concatenate([rest[:50], ball, rest[50:]])
    n = pos.shape[0]
    vel = inputs.maxwell_velocities(n, 1e-4, 8)
    runs = []
    for spread, void, graph in (("rows", True, False), ("auto", False, True), ("rows", False, False),
                                ("auto", True, True)):
        g = _context(pos, vel, spread=spread, precision=precision, variant=variant)
        _forces(g, n, sigma=0.2, r_cut=1.6)
        for c in range(2):
            if void and (c == 0 or precision == "fp32"):
                g.set_particles(pos=g.particles()[0] if c else pos)
            g.run_cycles(1) if graph else g.cycle(1)
        runs.append(_state(g))
    for r in runs[1:]:
        _same(r, runs[0])
