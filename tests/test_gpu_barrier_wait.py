"""A wait between the blocks of one launch that runs out (GPU): with the limit
at 0 every such wait gives up, no block goes on, every later launch of the
context stops at its first wait too, and the calls report it.  The buffers keep
values of before, so what runs on them stays in range; the GPU, and other
contexts, go on."""
import numpy as np
import pytest

from paper_1610_02733_gb300 import inputs, lbmd

pytestmark = pytest.mark.gpu

SHAPE = (24, 20, 18)


def _context(kind, precision, limit):
    n, kw = 1500, {}  # 47 blocks of a team per particle
    if kind == "lj":
        n = 300
    elif kind == "frozen":  # variant A, no wait in the MD phase: the re-ordering's only
        n, kw = 4000, {"variant": "A"}
    elif kind in ("rows", "tiles"):
        n, kw = 4000, {"spread": kind}
    elif kind in ("A", "C"):
        kw = {"variant": kind}
    g = lbmd.LBMD(*SHAPE, precision=precision, n_sub=3, kT=1e-4, zeta=0.5, seed=3, max_particles=n, max_bonds=n, **kw)
    if kind == "lj":  # a lattice of spacing 2, none within the cut-off of another
        grid = np.stack(np.meshgrid(*[np.arange(0, L, 2.0) for L in SHAPE], indexing="ij"), -1).reshape(-1, 3)
        pos = grid[:n] + 0.5
    else:
        pos = inputs.uniform_positions(n, SHAPE, 3)
    g.add_particles(pos, inputs.maxwell_velocities(n, 1e-4, 3))
    if kind == "lj":
        g.set_lj(1e-4, 1.0, 1.5)
    if kind == "bonds" or kind == "A":
        g.add_bonds([(2 * i, 2 * i + 1) for i in range(n // 2)], 1e-3, 1.0)
    g.set_barrier_wait(limit)
    return g


def _raises(call):
    with pytest.raises(lbmd.LbmdError) as ei:
        call()
    assert ei.value.status == lbmd.LBMD_ERR_CUDA, ei.value


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["B", "C", "A", "bonds", "lj", "frozen", "rows", "tiles"])
def test_wait_runs_out(kind, precision):
    want = _context(kind, precision, -1)
    want.run_cycles(3)
    want = want.particles()
    g = _context(kind, precision, 0)
    pos0 = g.particles()[0]
    g.run_cycles(4)  # queued before the failure is known
    _raises(g.synchronize)
    for call in (g.particles, g.populations, g.node_field, g.transfer, g.save_state, g.observables, g.md_substep,
                 lambda: g.run_cycles(1), lambda: g.cycle(1), g.synchronize):
        _raises(call)
    assert pos0.shape[0] == g.n_particles
    g.close()
    # another context is not affected, and neither is one whose limit was put back
    h = _context(kind, precision, 0)
    h.set_barrier_wait(-1)
    h.run_cycles(3)
    for a, b in zip(h.particles(), want):
        assert np.array_equal(a, b)
    h.close()


def test_found_by_the_observables_and_between_calls():
    g = _context("B", "fp32", -1)
    g.run_cycles(1)
    g.observables()
    g.set_barrier_wait(0)
    g.run_cycles(1)  # (a call after it may already know)
    obs = g.observables_async()
    _raises(g.synchronize)
    assert obs is not None
    with pytest.raises(lbmd.LbmdError) as ei:
        g.set_barrier_wait(-2)
    assert ei.value.status == lbmd.LBMD_ERR_ARG
    g.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_adjoint(precision):
    shape, n = (8, 9, 7), 300  # 19 blocks of 16 particles
    pos, vel = inputs.uniform_positions(n, shape, 4), inputs.maxwell_velocities(n, 1e-4, 4)
    ad = lbmd.Adjoint(*shape, n_particles=n, n_cycles=3, n_sub=4, precision=precision, kT=1e-4, seed=4)
    ad.set_barrier_wait(0)
    with pytest.raises(lbmd.LbmdError) as ei:  # the first pass: nothing was ever written
        ad.forward(0.5, pos, vel)
    assert ei.value.status == lbmd.LBMD_ERR_CUDA
    with pytest.raises(lbmd.LbmdError) as ei:
        ad.backward()
    assert ei.value.status == lbmd.LBMD_ERR_SEQUENCE
    ad.set_barrier_wait(-1)
    loss = ad.forward(0.5, pos, vel)
    want = ad.backward()
    ad.set_barrier_wait(0)
    with pytest.raises(lbmd.LbmdError):
        ad.backward()
    ad.set_barrier_wait(-1)
    assert ad.forward(0.5, pos, vel) == loss
    got = ad.backward()
    tol = {"fp32": 1e-5, "fp64": 1e-12}[precision]  # (the adjoint's atomics add in any order)
    assert abs(got[0] - want[0]) <= tol * abs(want[0])
    assert np.abs(got[1] - want[1]).max() <= tol * np.abs(want[1]).max()
    ad.close()
