"""Several MD steps in one launch (GPU): the same bits as one step at a time
with the row gather, whatever the particles do meanwhile."""
import numpy as np
import pytest

from gpu_common import assert_pops_close, assert_vec_close, pair
from paper_1610_02733_gb300 import inputs, lbmd

pytestmark = pytest.mark.gpu


def _run(shape, n, kT_init, steps, **kw):
    """steps: 'g' one captured cycle, 'e' one cycle call by call."""
    g = lbmd.LBMD(*shape, kT=1e-3, zeta=1.0, seed=11, max_particles=max(n, 1), **kw)
    if n:
        mass = inputs.uniform((n,), 0.8, 2.0, 4)
        g.add_particles(inputs.uniform_positions(n, shape, 6), inputs.maxwell_velocities(n, kT_init, 6), mass)
    for s in steps:
        g.run_cycles(1) if s == "g" else g.cycle(1)
    out = (g.populations(), g.node_field(), *g.particles())
    g.close()
    return out


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("integrator", ["start", "half_step"])
@pytest.mark.parametrize("shape,n,m", [((7, 5, 6), 1, 1), ((40, 6, 5), 129, 4), ((20, 9, 8), 1500, 10),
                                       ((30, 29, 27), 4000, 3)])
def test_variant_a_phase(precision, integrator, shape, n, m):
    # slow particles (they stay in their cells) and ones that cross several
    # cells per cycle; captured cycles, single steps, and both in turn
    for kT_init in (1e-4, 0.2):
        kw = dict(variant="A", precision=precision, integrator=integrator, n_sub=m)
        want = _run(shape, n, kT_init, "eeee", spread="rows", **kw)
        for steps, spread in (("gggg", "auto"), ("gege", "auto"), ("egge", "atomic")):
            _same(_run(shape, n, kT_init, steps, spread=spread, **kw), want)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("integrator", ["start", "half_step"])
@pytest.mark.parametrize("variant", ["B", "C"])
@pytest.mark.parametrize("shape,n,m", [((7, 5, 6), 1, 3), ((40, 6, 5), 33, 4), ((20, 19, 18), 330, 3), ((33, 32, 31), 19000, 2)])
def test_coupled_phase(precision, integrator, variant, shape, n, m):
    # one block, a cluster of blocks (33 particles: one team in the second
    # block), and more than one block of the larger size per SM
    for kT_init in (1e-4, 0.2):
        kw = dict(variant=variant, precision=precision, integrator=integrator, n_sub=m)
        want = _run(shape, n, kT_init, "eee", spread="rows", **kw)
        for steps, spread in (("ggg", "auto"), ("geg", "atomic")):
            _same(_run(shape, n, kT_init, steps, spread=spread, **kw), want)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("integrator", ["start", "half_step"])
@pytest.mark.parametrize("variant", ["A", "B", "C"])
def test_coupled_phase_with_bonds(precision, integrator, variant):
    # chains longer than a block, a particle with the largest number of
    # bonds, and unbonded ones
    shape, m = (16, 15, 14), 5
    out = []
    for spread, steps in (("rows", "eee"), ("auto", "ggg"), ("atomic", "egg")):
        pos, bonds = inputs.bead_spring_chains(3, 150, shape, 5)
        g = lbmd.LBMD(*shape, kT=1e-3, zeta=1.0, seed=11, max_particles=460, max_bonds=1000, variant=variant,
                      precision=precision, integrator=integrator, n_sub=m, spread=spread)
        g.add_particles(pos, inputs.maxwell_velocities(450, 1e-3, 5))
        g.add_particles(inputs.uniform_positions(10, shape, 1), inputs.maxwell_velocities(10, 1e-3, 1))
        g.add_bonds(bonds, 1.0, 1.0)
        g.add_fene_bonds([(451, 452 + k) for k in range(8)], 0.5, 60.0)
        for s in steps:
            g.run_cycles(1) if s == "g" else g.cycle(1)
        out.append((g.populations(), g.node_field(), *g.particles()))
        g.close()
    _same(out[1], out[0])
    _same(out[2], out[0])


@pytest.mark.parametrize("n", [4864, 4900])
def test_fp64_bonds_at_the_limit_of_the_teams(n):
    # 8 lanes a particle, one block of 256 per SM: both sides of the line on 152 SMs
    shape, m, out = (20, 19, 18), 2, []
    for spread, steps in (("rows", "ee"), ("auto", "gg"), ("auto", "eg")):
        g = lbmd.LBMD(*shape, kT=1e-3, zeta=1.0, seed=11, max_particles=n, max_bonds=n, precision="fp64", n_sub=m,
                      spread=spread)
        g.add_particles(inputs.uniform_positions(n, shape, 6), inputs.maxwell_velocities(n, 1e-3, 6))
        g.add_bonds([(i, i + 1) for i in range(0, n - 1, 2)], 1e-3, 1.0)
        for s in steps:
            g.run_cycles(1) if s == "g" else g.cycle(1)
        out.append((g.populations(), g.node_field(), *g.particles()))
        g.close()
    _same(out[1], out[0])
    _same(out[2], out[0])


@pytest.mark.parametrize("variant", ["A", "B", "C"])
@pytest.mark.parametrize("empty", [1, 2, 3])
def test_particles_added_after_empty_cycles(variant, empty):
    # both active sets are empty until the first particle, whichever the cycle
    # that it comes in takes
    o, g = pair((14, 9, 10), variant=variant, n_sub=3, kT=1e-4, zeta=0.7, seed=5, max_particles=60,
                body_force=(1e-4, 0.0, 0.0))
    o.cycle(empty)
    g.run_cycles(empty)
    pos, vel = inputs.uniform_positions(60, (14, 9, 10), 2), inputs.maxwell_velocities(60, 1e-3, 2)
    for s in (o, g):
        s.add_particles(pos, vel)
        s.cycle(2)
    assert_pops_close(g.populations(), o.populations(), "fp32")
    assert_vec_close(g.particles()[1], o.particles()[1], "fp32", "velocities")
    g.close()
    o.close()
