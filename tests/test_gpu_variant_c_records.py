"""Variant C on the compact records (GPU): its transfers stay in variant B's
node records until the LB step, so every spread path gives the same bits, and
reading the populations inside a cycle (where the transfers so far are added on
the way out) agrees with the oracle and changes nothing."""
import numpy as np
import pytest

from gpu_common import assert_pops_close, pair
from paper_1610_02733_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape,n", [((33, 5, 7), 1), ((8, 6, 10), 400)])
def test_reads_inside_a_cycle(precision, shape, n):
    pos, vel = inputs.uniform_positions(n, shape, 8), inputs.maxwell_velocities(n, 1e-3, 8)
    ends = []
    for read in (True, False):
        o, g = pair(shape, precision=precision, variant="C", n_sub=3, kT=1e-3, zeta=1.0, seed=13, max_particles=n,
                    nu_bulk=0.3)
        for s in (o, g):
            s.add_particles(pos, vel)
        for _ in range(2):
            for _ in range(3):
                g.md_substep()
                o.md_substep()
                if read:
                    assert_pops_close(g.populations(), o.populations(), precision)
                    assert not g.transfer().any()
            g.lb_step()
            o.lb_step()
        ends.append((g.populations(), *g.particles()))
        g.close()
    for a, b in zip(*ends):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16dev"])
@pytest.mark.parametrize("integrator", ["start", "half_step"])
def test_spread_paths_agree_bitwise(precision, integrator):
    shape, n = (34, 9, 6), 700
    runs = {}
    for spread in ("rows", "atomic", "auto"):
        o, g = pair(shape, precision=precision, variant="C", n_sub=4, kT=1e-3, zeta=1.0, seed=3, max_particles=n,
                    spread=spread, integrator=integrator)
        # fast particles: some leave their row within a cycle
        g.add_particles(inputs.uniform_positions(n, shape, 2), inputs.maxwell_velocities(n, 0.05, 2))
        g.run_cycles(4)
        runs[spread] = (g.populations(), *g.particles())
        g.close()
    for spread in ("atomic", "auto"):
        for a, b in zip(runs["rows"], runs[spread]):
            assert np.array_equal(a, b)
