"""Harmonic bonds with rest lengths of every sign and size (GPU) against the
oracle: U = (k/2)(|r| - r0)^2 is defined for any finite r0, and near
|r| = -r0 the difference of squares over r + r0 is not."""
import numpy as np
import pytest

from gpu_common import assert_vec_close, pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("lj,spread", [(False, "auto"), (False, "rows"), (True, "auto"), (True, "rows")])
@pytest.mark.parametrize("k,r0", [(0.02, -1.0), (0.02, -0.25), (0.02, 0.0), (0.02, 1e-15), (0.02, 1.0), (1e-6, 3e4),
                                  (1e-27, 1e25), (1e-27, -1e25)])
def test_one_md_step(precision, lj, spread, k, r0):
    # pairs whose length is |r0| up to a few rounding steps, and others; the
    # force's own conditioning is of order one (r - r0 does not cancel for
    # r0 <= 0, and for r0 = 1 the pairs keep 1e-2 from it), so the parity
    # tolerance of one step holds
    shape = (12, 11, 10)
    length = [1.0, 1.0 + 2.0 ** -20, 1.0001, 1.01, 0.25, 0.2501, 2.5, 0.75]
    if r0 == 1.0:
        length = [0.5, 0.98, 1.02, 1.5]
    o, g = pair(shape, precision=precision, n_sub=2, zeta=0.0, max_particles=40, max_bonds=20, spread=spread)
    pos, bonds = [], []
    for i, d in enumerate(length):
        a = np.array([11.5 + d if i % 2 else 1.25, 1.5 + i, 2.5 + (i % 3)])  # every other pair across the face
        pos += [a % shape, (a - np.array([d, 0, 0])) % shape]
        bonds.append((2 * i, 2 * i + 1))
    pos = np.array(pos)
    for s in (o, g):
        s.add_particles(pos, np.zeros_like(pos))
        if lj:
            s.set_lj(0.0, 0.2, 0.3)  # the pair kernels, without a force of their own
        s.add_bonds(np.array(bonds), k, r0)
        s.md_substep()
    assert np.abs(o.particles()[1]).max() > 0
    assert_vec_close(g.particles()[1], o.particles()[1], precision, "velocities")
    g.close()
    o.close()
