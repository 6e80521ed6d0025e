"""FP64 collision in 64-bit integers (GPU) against the oracle: densities on both
sides of a power of two, fluids near rest, and nodes outside the integers'
range, which take the FP64 form -- also within one lattice."""
import numpy as np
import pytest

from gpu_common import assert_pops_close, pair
from paper_1610_02733_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,noise", [("A", "uniform"), ("B", "gauss"), ("C", "uniform"), ("C", "gauss")])
@pytest.mark.parametrize("rho0", [1.0, 0.51, 2.0 ** -41, 3.0e9])
@pytest.mark.parametrize("state", ["near rest", "mixed", "far"])
def test_lb_step_fp64(variant, noise, rho0, state):
    # thermal speeds relative to the lattice, whatever the density
    shape, n, kT = (10, 4, 7), 40, 1e-3 * rho0
    o, g = pair(shape, precision="fp64", variant=variant, n_sub=2, rho0=rho0, kT=kT, zeta=0.5 * rho0 if rho0 < 1 else 0.5,
                nu=0.1, body_force=(1e-4 * rho0, 0.0, -2e-5 * rho0), seed=31, max_particles=n, noise=noise)
    f = inputs.perturbed(o.populations(), 0.2, 7)
    if state == "mixed":  # every third node: a rest population beyond the range, or a negative one
        f[0, ::3] = 0.9 * rho0
        f[5, 1::3] = -0.2 * rho0
    elif state == "far":
        f *= 9.0
    pos, vel = inputs.uniform_positions(n, shape, 3), inputs.maxwell_velocities(n, 1e-4, 3)
    for s in (o, g):
        s.set_populations(f)
        s.add_particles(pos, vel)
        s.cycle(2)
    assert_pops_close(g.populations() / rho0, o.populations() / rho0, "fp64")
    if variant != "C":
        assert np.abs(g.transfer()).max() == 0.0
    nf, no = g.node_field() / rho0, o.node_field() / rho0
    assert np.abs(nf - no).max() <= 1e-12
    g.close()
    o.close()
