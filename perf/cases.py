"""The work that users of this framework have it do, as cases to be timed.

A case is a dict of plain numbers and texts; ``listed()`` gives the fixed ones
and ``draw(rng)`` one more of the same ranges.  ``prepare`` builds what a
program holds before it calls (contexts with their particles), ``run`` makes
one pass through the public entry points, ``work`` counts the bytes and
operations that pass cannot do without, and ``exact`` gives the same outputs
from a plain torch computation in 64 bits.

Every random number of the method comes from a counter-based generator under
the context's seed, so a pass is a fixed function of its inputs, noise
included.  A storage form with 32-bit arithmetic returns its results as
32-bit tensors, the FP64 form as 64-bit ones.
"""
import math

import numpy as np
import torch

from paper_1610_02733_gb300 import inputs, lbmd, lj_units, sweep

KT = 1e-4  # thermal energy of the ideal-particle and bead-spring systems
SPRING = (1.0, 1.0)  # stiffness and rest length of the harmonic bonds


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def _box(nx, ny, nz, n, m, cycles, **kw):
    case = {"kind": "box", "nx": nx, "ny": ny, "nz": nz, "n": n, "m": m, "cycles": cycles, "variant": "B",
            "precision": "fp32", "noise": "uniform", "integrator": "start", "zeta": 1.0, "force": 0.0, "io": "device"}
    case.update(kw)
    return case


def listed():
    cases = [
        # the smallest system: ten particles in an 8^3 box in FP64, one LB
        # cycle per call, as a program does that looks at every cycle
        ("box8_fp64", _box(8, 8, 8, 10, 5, 1, precision="fp64")),
        # bead-spring polymer solution: 64 chains of 64 beads in 64^3 (springs
        # whose thermal extension is a hundredth of their length)
        ("chains64", _box(64, 64, 64, 4096, 10, 10, kind="chains", beads=64, zeta=2.0)),
        # the paper's Kremer-Grest system, 10 chains of 256 beads in (20 sigma)^3
        # with Lennard-Jones forces and FENE springs, a point of its sweep
        ("kremer_grest", {"kind": "kg", "chains": 10, "beads": 256, "box": 20, "m": 10, "cycles": 2, "dt": 0.005,
                          "zeta": 20.0, "variant": "B", "integrator": "half_step"}),
        # variant C (the transfers enter the populations every MD step) on a
        # mid-size suspension
        ("suspension_c", _box(96, 80, 112, 51200, 5, 2, variant="C")),
        # driven flow in a ragged box with a few tracers, normal variates, the
        # flow field read back for analysis after every ten cycles
        ("flow_field", _box(61, 47, 53, 500, 4, 10, variant="A", noise="gauss", force=1e-5, io="field")),
        # an external program hands over and takes back the particles every
        # cycle through pinned host arrays, with the observables
        ("host_coupled", _box(96, 96, 96, 53000, 10, 1, io="host")),
        # the double-precision form at a mid-size suspension
        ("suspension_fp64", _box(128, 128, 128, 131072, 10, 1, precision="fp64")),
        # variant A on a large box with odd sides
        ("suspension_a", _box(250, 201, 181, 545000, 10, 2, variant="A")),
        # the headline workload: 256^3 nodes, 10^6 ideal particles, variant B
        ("suspension_b", _box(256, 256, 256, 1000000, 10, 2)),
        # ... with the populations stored as FP16 deviations
        ("suspension_fp16", _box(256, 256, 256, 1000000, 10, 2, precision="fp16dev")),
        # temperature statistics: 512 independent boxes of uneven sizes, every
        # replica's kinetic energy and momentum sampled every 10 MD steps
        ("replicas512", {"kind": "replicas", "replicas": 512, "largest": 32, "most": 400, "steps": 100}),
        # gradient of the mean particle drag (200 MD steps), forward and backward
        ("drag_gradient", {"kind": "gradient", "edge": 32, "n": 64, "m": 10, "cycles": 20, "precision": "fp32"}),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "chains", "kg", "replicas", "gradient"])
    m = rng.choice([1, 2, 4, 5, 10])
    if kind == "kg":
        box = rng.randint(16, 30)
        beads = rng.choice([32, 64, 256, 320])
        return {"kind": "kg", "chains": max(1, int(0.32 * box ** 3) // beads), "beads": beads, "box": box,
                "m": rng.choice([5, 10]), "cycles": 2, "dt": rng.choice([0.001, 0.005]),
                "zeta": rng.choice([1.0, 5.0, 20.0]), "variant": rng.choice(["A", "B", "C"]),
                "integrator": rng.choice(["start", "half_step"])}
    if kind == "replicas":
        return {"kind": "replicas", "replicas": _log_int(rng, 8, 512), "largest": rng.choice([16, 24, 32]),
                "most": rng.randint(20, 400), "steps": rng.choice([50, 100])}
    if kind == "gradient":
        return {"kind": "gradient", "edge": rng.randint(8, 32), "n": _log_int(rng, 1, 300), "m": rng.choice([5, 10]),
                "cycles": rng.randint(2, 20), "precision": rng.choice(["fp32", "fp64"])}
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp16dev"])
    side = _log_int(rng, 8, 128 if precision == "fp64" else 240)
    nx, ny, nz = (max(4, int(side * rng.uniform(0.8, 1.06))) for _ in range(3))
    N = nx * ny * nz
    if kind == "chains":
        beads = rng.choice([16, 64])
        n = beads * max(1, int(N * rng.uniform(0.004, 0.03)) // beads)
        return _box(nx, ny, nz, n, max(m, 4), 2, kind="chains", beads=beads, precision=precision,
                    zeta=rng.uniform(0.5, 2.0),
                    variant=rng.choice(["A", "B"]), integrator=rng.choice(["start", "half_step"]))
    n = max(1, int(N * math.exp(rng.uniform(math.log(0.001), math.log(0.1)))))
    # variant C is studied in the plain storage forms
    variant = rng.choice(["A", "B", "B", "B" if precision == "fp16dev" else "C"])
    noise = "gauss" if precision in ("fp32", "fp64") and rng.random() < 0.25 else "uniform"
    io = rng.choice(["device", "device", "field", "host"]) if N < 1500000 else "device"
    return _box(nx, ny, nz, n, m, 1 if N > 4000000 else 2, variant=variant, precision=precision, noise=noise, io=io,
                integrator=rng.choice(["start", "start", "half_step"]), zeta=rng.uniform(0.3, 0.8) * min(m, 2),
                force=rng.choice([0.0, 1e-5]))


# ---------------------------------------------------------------------------
# Inputs, the same on the GPU side and in exact()
# ---------------------------------------------------------------------------
def _particles(case, seed):
    """Positions, velocities and bonds of a box or chains case."""
    shape = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "chains":
        pos, bonds = inputs.bead_spring_chains(case["n"] // case["beads"], case["beads"], shape, seed)
    else:
        pos, bonds = inputs.uniform_positions(case["n"], shape, seed), None
    return pos, inputs.maxwell_velocities(pos.shape[0], KT, seed), bonds


def _replicas(case, seed):
    edges = [e for e in (12, 16, 24, 32) if e <= case["largest"]]
    c = inputs.replica_configs(case["replicas"], seed, edges=edges, max_particles=case["most"])
    # the explicit friction step is stable well below zeta dt = 2
    c["zeta"] = np.minimum(c["zeta"], 0.7 * c["n_sub"])
    c["seed"] = [seed * 1000 + r for r in range(case["replicas"])]
    c["pos"] = [inputs.uniform_positions(n, d, seed * 1000 + r)
                for r, (n, d) in enumerate(zip(c["n_particles"], c["dims"]))]
    c["vel"] = [inputs.maxwell_velocities(n, KT, seed * 1000 + r) for r, n in enumerate(c["n_particles"])]
    return c


def _gradient(case, seed):
    shape = (case["edge"],) * 3
    return (shape, inputs.uniform_positions(case["n"], shape, seed), inputs.maxwell_velocities(case["n"], KT, seed))


GRADIENT_ZETA, GRADIENT_FORCE = 1.5, (1e-5, 0.0, 0.0)
SAMPLE_EVERY = 10  # MD steps between two kinetic samples of the replicas

_STREAM = None


def _stream():
    """One stream that torch and the contexts share, so that results written
    by a context are ordered with the caller's use of them."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
        torch.cuda.set_stream(_STREAM)
    return _STREAM.cuda_stream


def prepare(case, seed):
    stream = _stream()
    kind = case["kind"]
    if kind == "replicas":
        c = _replicas(case, seed)
        b = lbmd.Batch(c["dims"], n_sub=c["n_sub"], variant=c["variant"], zeta=c["zeta"], seed=c["seed"],
                       max_particles=c["n_particles"], precision="fp32", kT=KT, stream=stream)
        for r in range(case["replicas"]):
            b.add_particles(r, c["pos"][r], c["vel"][r])
        return {"case": case, "batch": b}
    if kind == "gradient":
        shape, pos, vel = _gradient(case, seed)
        ad = lbmd.Adjoint(*shape, n_particles=case["n"], n_cycles=case["cycles"], n_sub=case["m"],
                          precision=case["precision"], kT=KT, body_force=GRADIENT_FORCE, seed=seed, stream=stream)
        return {"case": case, "adjoint": ad, "pos": pos, "vel": vel}
    if kind == "kg":
        sim, _ = sweep.build_system(case["variant"], case["m"], case["dt"], case["zeta"], n_chains=case["chains"],
                                    n_beads=case["beads"], box=case["box"], seed=seed,
                                    integrator=case["integrator"], stream=stream)
        return {"case": case, "sim": sim, "n": sim.n_particles}
    pos, vel, bonds = _particles(case, seed)
    n = pos.shape[0]
    sim = lbmd.LBMD(case["nx"], case["ny"], case["nz"], variant=case["variant"], precision=case["precision"],
                    n_sub=case["m"], kT=KT, zeta=case["zeta"], seed=seed, max_particles=n,
                    max_bonds=0 if bonds is None else bonds.shape[0], noise=case["noise"],
                    integrator=case["integrator"], body_force=(case["force"], 0.0, 0.0), stream=stream)
    sim.add_particles(pos, vel)
    if bonds is not None:
        sim.add_bonds(bonds, *SPRING)
    state = {"case": case, "sim": sim, "n": n}
    if case["io"] == "host":  # page-locked arrays: up, and down again
        state["up"] = [torch.from_numpy(a).pin_memory() for a in (pos, vel)]
        state["down"] = [torch.empty(n, 3, dtype=torch.float64).pin_memory() for _ in range(2)]
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _width(case):
    return torch.float64 if case.get("precision") == "fp64" else torch.float32


def _kinetic(samples):
    """Kinetic samples (sample, replica, 5) by quantity."""
    return {"energy": samples[..., 0], "momentum": samples[..., 1:4], "count": samples[..., 4]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "replicas":
        b = state["batch"]
        samples = torch.empty(case["steps"] // SAMPLE_EVERY, b.R, 5, dtype=torch.float64, device="cuda")
        for s in range(samples.shape[0]):
            b.run(SAMPLE_EVERY)
            b.kinetic_device(samples[s].data_ptr())
        return _kinetic(samples.float())
    if kind == "gradient":
        ad = state["adjoint"]
        loss = ad.forward(GRADIENT_ZETA, state["pos"], state["vel"])
        dzeta, dpos = ad.backward()
        width = np.float64 if case["precision"] == "fp64" else np.float32
        return {"loss": width(loss), "dzeta": width(dzeta), "dpos": dpos.astype(width)}
    sim, width = state["sim"], _width(case)
    io = case.get("io", "device")
    if io == "host":
        for _ in range(case["cycles"]):
            sim.set_particles_async(*state["up"])
            sim.run_cycles(1)
            sim.particles_async(*state["down"])
            obs = sim.observables_async()
            sim.synchronize()
        o = lbmd.observables_dict(obs)
        kinetic = [o["kT_particles"], o["mass"], *o["p_particles"]]
        return {"pos": state["down"][0].to(width), "vel": state["down"][1].to(width),
                "observables": torch.tensor(kinetic, dtype=width)}
    sim.run_cycles(case["cycles"])
    pos = torch.empty(state["n"], 3, dtype=torch.float64, device="cuda")
    vel = torch.empty_like(pos)
    sim.particles_device(pos, vel)
    out = {"pos": pos.to(width), "vel": vel.to(width)}
    if io == "field":
        out["field"] = torch.from_numpy(sim.node_field()).to(width)
    return out


def _boxes(case):
    """(nodes, particles, LB steps, MD steps, bytes of a stored population) of
    every box of a case, boxes alike counted together."""
    kind = case["kind"]
    if kind == "replicas":
        c = inputs.replica_configs(case["replicas"], 1, edges=[e for e in (12, 16, 24, 32) if e <= case["largest"]],
                                   max_particles=case["most"])
        return [(int(np.prod(d)), int(n), case["steps"] // int(m), case["steps"], 4)
                for d, n, m in zip(c["dims"], c["n_particles"], c["n_sub"])]
    md = case["m"] * case["cycles"]
    if kind == "gradient":
        size = 8 if case["precision"] == "fp64" else 4
        # forward, then the adjoint of each step (the states kept meanwhile
        # are written once and read once more)
        return [(case["edge"] ** 3, case["n"], 2 * case["cycles"], 2 * md, size)]
    if kind == "kg":
        return [(case["box"] ** 3, case["chains"] * case["beads"], case["cycles"], md, 4)]
    size = {"fp64": 8, "fp32": 4}.get(case["precision"], 2)
    return [(case["nx"] * case["ny"] * case["nz"], case["n"], case["cycles"], md, size)]


def work(case):
    """An LB step reads and writes the 19 populations of every node; an MD
    step reads and writes a particle's position and velocity (6 values) and
    reads and updates the momentum of the nodes around it (at most 8 per
    particle, each node of the box at most once)."""
    total = {"bytes": 0.0, "flops": 0.0}
    for N, n, lb, md, size in _boxes(case):
        real = 8 if size == 8 else 4
        touched = N * (1.0 - math.exp(-8.0 * n / N))
        total["bytes"] += lb * 2 * 19 * size * N + md * real * (12 * n + 8 * touched)
        total["flops"] += lb * 250.0 * N + md * 250.0 * n
    if case.get("io") == "field":
        total["bytes"] += 32.0 * case["nx"] * case["ny"] * case["nz"]
    if case.get("io") == "host":
        total["bytes"] += 96.0 * case["n"] * case["cycles"]
    return total


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
               (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
               (0, 1, -1), (0, -1, 1)])
_C2 = (_C ** 2).sum(1)
_W = np.where(_C2 == 0, 1 / 3, np.where(_C2 == 1, 1 / 18, 1 / 36))


def _modes():
    x, y, z = _C.T
    c2 = _C2
    return np.array([np.ones(19), x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, x * z, y * z,
                     (3 * c2 - 5) * x, (3 * c2 - 5) * y, (3 * c2 - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y,
                     (x * x - y * y) * z, 3 * c2 * c2 - 6 * c2 + 1, (2 * c2 - 3) * (3 * x * x - c2),
                     (2 * c2 - 3) * (y * y - z * z)], dtype=np.float64)


_E = _modes()
_B = (_E * _E * _W).sum(1)  # squared norms


def _mul32(a, b):
    """High and low 32 bits of the product of a constant and 32-bit words held in int64."""
    p1, p2 = a * (b & 0xFFFF), a * (b >> 16)
    return (p2 + (p1 >> 16)) >> 16, (p1 + ((p2 & 0xFFFF) << 16)) & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10; counters and keys are int64 tensors or numbers."""
    zero = torch.zeros_like(c0)
    c1, c2, c3, k0, k1 = (zero + v for v in (c1, c2, c3, k0, k1))
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c0)
        h1, l1 = _mul32(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _normal_pair(w1, w2):
    u1, u2 = ((w1 >> 8).double() + 0.5) / 2 ** 24, ((w2 >> 8).double() + 0.5) / 2 ** 24
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


class _Exact:
    """Periodic boxes side by side, each with its particles, in 64 bits.
    Nothing is changed in place, so that autograd can follow every step."""

    def __init__(self, dims, n_sub, variant, zeta, seeds, kT, nu=1.0 / 6.0, force=(0.0, 0.0, 0.0), gauss=False,
                 half_step=False):
        dev = self.dev = "cuda"
        self.R, self.kT, self.gauss, self.half_step = len(dims), kT, gauss, half_step
        self.dims = torch.as_tensor(np.asarray(dims), dtype=torch.int64, device=dev)
        sizes = np.prod(np.asarray(dims, dtype=np.int64), axis=1)
        self.first = torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)[:-1]]), device=dev)
        self.N = int(sizes.sum())
        self.n_sub, self.variant = [int(v) for v in n_sub], list(variant)
        self.seeds = [int(s) for s in seeds]
        self.zeta = torch.as_tensor(zeta, dtype=torch.float64, device=dev)
        self.force = torch.as_tensor(force, dtype=torch.float64, device=dev)
        self.gs = (6 * nu - 1) / (6 * nu + 1)
        self.gamma = torch.zeros(19, dtype=torch.float64, device=dev)
        self.gamma[5:10] = self.gs
        self.E = torch.as_tensor(_E, device=dev)
        self.back = torch.as_tensor((_W[:, None] * _E.T) / _B, device=dev)  # modes -> populations
        self.amp = torch.as_tensor(np.sqrt(3 * kT * _B), device=dev) * torch.sqrt(1 - self.gamma ** 2)
        self.amp[:4] = 0
        self.f = torch.as_tensor(_W, device=dev)[:, None].repeat(1, self.N)
        self.lb, self.md = [0] * self.R, 0
        self.slices = [(int(a), int(a) + int(s)) for a, s in zip(self.first.tolist(), sizes)]
        self._moments()
        self.J = torch.zeros(3, self.N, dtype=torch.float64, device=dev)
        self.bonds = self.lj = None
        self._tables = {}

    def _moments(self):
        c = torch.as_tensor(_C.T.astype(np.float64), device=self.dev)
        self.rho, self.j = self.f.sum(0), c @ self.f

    def add(self, box, pos, vel):
        """Particles: their boxes, positions and velocities (mass 1); ids count from 0 in every box."""
        self.box = torch.as_tensor(box, dtype=torch.int64, device=self.dev)
        counts = np.bincount(np.asarray(box), minlength=self.R)
        self.id = torch.as_tensor(np.concatenate([np.arange(k) for k in counts]), dtype=torch.int64, device=self.dev)
        self.pos = torch.as_tensor(pos, device=self.dev)
        self.vel = torch.as_tensor(vel, device=self.dev)
        pick = lambda v, t: torch.as_tensor(v, dtype=t, device=self.dev)[self.box]  # noqa: E731
        self.p_dt = 1.0 / pick(self.n_sub, torch.float64)
        self.p_zeta = self.zeta if self.zeta.dim() == 0 else self.zeta[self.box]
        self.k0 = pick([s & 0xFFFFFFFF for s in self.seeds], torch.int64)
        self.k1 = pick([s >> 32 for s in self.seeds], torch.int64)
        self.seen = pick([1.0 if v == "B" else 0.0 for v in self.variant], torch.float64)
        self.F = torch.zeros_like(self.pos)
        self.Fc = self._conservative(self.pos)

    def _conservative(self, x):
        if self.bonds is None and self.lj is None:
            return torch.zeros_like(x)
        L = self.dims[0].double()
        F = torch.zeros_like(x)
        if self.bonds is not None:
            (i, k), kind, strength, r0 = self.bonds
            d = x[k] - x[i]
            d = d - L * torch.round(d / L)
            r2 = (d * d).sum(1, keepdim=True)
            r = torch.sqrt(r2)
            g = strength / (1 - r2 / r0 ** 2) if kind == "fene" else strength * (r - r0) / r
            F = F.index_add(0, i, g * d).index_add(0, k, -g * d)
        if self.lj is not None:
            eps, sigma, rc = self.lj
            for s in range(0, x.shape[0], 1024):
                d = x[None] - x[s:s + 1024, None]
                d = d - L * torch.round(d / L)
                r2 = (d * d).sum(2)
                near = (r2 < rc * rc) & (r2 > 0)
                r2 = torch.where(near, r2, torch.ones_like(r2))
                t = (sigma ** 2 / r2) ** 3
                g = torch.where(near, -24 * eps * (2 * t * t - t) / r2, torch.zeros_like(r2))
                F = F.index_add(0, torch.arange(s, s + d.shape[0], device=x.device), (g[:, :, None] * d).sum(1))
        return F

    def _corners(self, x):
        """Nodes and weights of the 8 corners of every particle's cell."""
        dims, first = self.dims[self.box], self.first[self.box]
        base = torch.floor(x.detach())
        frac = x - base
        base = base.long()
        nodes, weights = [], []
        for o in range(8):
            off = torch.tensor([o & 1, (o >> 1) & 1, o >> 2], device=self.dev)
            c = torch.remainder(base + off, dims)
            nodes.append(first + c[:, 0] + dims[:, 0] * (c[:, 1] + dims[:, 1] * c[:, 2]))
            weights.append(torch.where(off == 1, frac, 1 - frac).prod(1))
        return nodes, weights

    def _force(self, x, v):
        """Coupling force at positions x for velocities v, and where its transfer goes."""
        nodes, weights = self._corners(x)
        u = 0
        for k, w in zip(nodes, weights):
            u = u + (w / self.rho[k])[:, None] * (self.j[:, k] + self.seen * self.J[:, k]).T
        zeta = self.p_zeta if self.p_zeta.dim() == 0 else self.p_zeta[:, None]
        F = -zeta * (v - u)
        if self.kT > 0:
            r = _philox(self.id, self.md, 1, 0, self.k0, self.k1)
            if self.gauss:
                xi = torch.stack(_normal_pair(r[0], r[1]) + _normal_pair(r[2], r[3])[:1], 1)
            else:
                xi = torch.stack([math.sqrt(12.0) * ((w.double() + 0.5) / 2 ** 32 - 0.5) for w in r[:3]], 1)
            F = F + torch.sqrt(2 * zeta * self.kT / self.p_dt[:, None]) * xi
        return F, nodes, weights

    def md_step(self):
        dt = self.p_dt[:, None]
        h = 0.5 * dt
        x, v = self.pos, self.vel
        if self.half_step:
            v = v + h * (self.F + self.Fc)
            x = x + dt * v
            F, nodes, weights = self._force(x, v)
        else:
            F, nodes, weights = self._force(x, v)
            v = v + h * (F + self.Fc)
            x = x + dt * v
        self.Fc = self._conservative(x)
        self.vel = v + h * (F + self.Fc)
        L = self.dims[self.box].double()
        self.pos = x - L * torch.floor(x.detach() / L)
        self.F = F
        dP = (dt * F).T
        J = self.J
        for k, w in zip(nodes, weights):
            J = J.index_add(1, k, -w * dP)
        self.J = J
        self.md += 1
        if self.variant[0] == "C":
            self._forcing_update()

    def _stress(self, u, F):
        """The forcing part of the stress modes, u F + F u, in the mode basis (without its prefactor)."""
        uF = (u * F).sum(0)
        return torch.stack([uF, 3 * u[0] * F[0] - uF, u[1] * F[1] - u[2] * F[2], 0.5 * (u[0] * F[1] + u[1] * F[0]),
                            0.5 * (u[0] * F[2] + u[2] * F[0]), 0.5 * (u[1] * F[2] + u[2] * F[1])])

    def _forcing_update(self):
        F = self.J
        u = (self.j + 0.5 * F) / self.rho
        dm = torch.cat([torch.zeros_like(F[:1]), F, (1 + self.gamma[4:10, None]) * self._stress(u, F),
                        torch.zeros(9, self.N, dtype=torch.float64, device=self.dev)])
        self.f = self.f + self.back @ dm
        self._moments()
        self.J = torch.zeros_like(F)

    def _collide(self, f, rho, j, F, node, step, k0, k1):
        u = (j + 0.5 * F) / rho
        m = self.E @ f
        uu = (u * u).sum(0)
        zero = torch.zeros_like(rho)
        eq = torch.stack([rho, j[0], j[1], j[2], rho * uu, rho * (3 * u[0] ** 2 - uu), rho * (u[1] ** 2 - u[2] ** 2),
                          rho * u[0] * u[1], rho * u[0] * u[2], rho * u[1] * u[2]] + 9 * [zero])
        m = eq + self.gamma[:, None] * (m - eq)
        add = torch.cat([F, (1 + self.gamma[4:10, None]) * self._stress(u, F)])
        m = torch.cat([m[:1], m[1:10] + add, m[10:]])
        if self.kT > 0:
            xi = []
            for q in range(4 if self.gauss else 2):
                r = _philox(node, step, 0, q, k0, k1)
                if self.gauss:
                    xi += _normal_pair(r[0], r[1]) + _normal_pair(r[2], r[3])
                else:
                    for w in r:
                        xi += [math.sqrt(12.0) * ((b.double() + 0.5) / 2 ** 16 - 0.5) for b in (w & 0xFFFF, w >> 16)]
            m = torch.cat([m[:4], m[4:] + self.amp[4:, None] * torch.sqrt(rho) * torch.stack(xi[:15])])
        return self.back @ m

    def _neighbours(self, due):
        """The nodes of the boxes `due`, their boxes and numbers within them, and, for every velocity,
        the place in this list that a population streams from."""
        if due not in self._tables:
            node, box, source, at = [], [], [[] for _ in range(19)], 0
            for r in due:
                a, b = self.slices[r]
                nx, ny, nz = self.dims[r].tolist()
                local = torch.arange(b - a, device=self.dev).view(nz, ny, nx)
                node.append(local.reshape(-1))
                box.append(torch.full((b - a,), r, device=self.dev))
                for i in range(19):
                    shift = tuple(int(v) for v in _C[i, ::-1])
                    source[i].append(at + torch.roll(local, shift, (0, 1, 2)).reshape(-1))
                at += b - a
            node, box = torch.cat(node), torch.cat(box)
            self._tables[due] = (self.first[box] + node, box, node, [torch.cat(v) for v in source])
        return self._tables[due]

    def lb_step(self, due):
        nodes, box, node, source = self._neighbours(due)
        whole = len(due) == self.R
        pick = (lambda v: v) if whole else (lambda v: v[..., nodes])  # noqa: E731
        f, rho, j, J = pick(self.f), pick(self.rho), pick(self.j), pick(self.J)
        F = (torch.zeros_like(J) if self.variant[0] == "C" else J) + self.force[:, None]
        per_box = lambda v: torch.as_tensor(v, dtype=torch.int64, device=self.dev)[box]  # noqa: E731
        step = per_box(self.lb)
        k0, k1 = per_box([s & 0xFFFFFFFF for s in self.seeds]), per_box([s >> 32 for s in self.seeds])
        out, part = [], 1 << 21  # in parts, for the temporaries' sake
        for s in range(0, f.shape[1], part):
            c = slice(s, s + part)
            out.append(self._collide(f[:, c], rho[c], j[:, c], F[:, c], node[c], step[c], k0[c], k1[c]))
        g = torch.cat(out, 1)
        del out
        g = torch.stack([g[i][source[i]] for i in range(19)])
        if whole:
            self.f, self.J = g, torch.zeros_like(self.J)
            self._moments()
        else:
            c = torch.as_tensor(_C.T.astype(np.float64), device=self.dev)
            self.f[:, nodes], self.J[:, nodes], self.rho[nodes], self.j[:, nodes] = g, 0.0, g.sum(0), c @ g
        for r in due:
            self.lb[r] += 1

    def advance(self, steps):
        for _ in range(steps):
            self.md_step()
            due = tuple(r for r in range(self.R) if self.md % self.n_sub[r] == 0)
            if due:
                self.lb_step(due)


def _exact_gradient(case, seed):
    shape, pos, vel = _gradient(case, seed)
    zeta = torch.tensor(GRADIENT_ZETA, dtype=torch.float64, device="cuda", requires_grad=True)
    x0 = torch.as_tensor(pos, device="cuda").requires_grad_(True)
    e = _Exact([shape], [case["m"]], "B", 0.0, [seed], KT, force=GRADIENT_FORCE)
    e.zeta = zeta
    e.add(np.zeros(case["n"], dtype=np.int64), pos, vel)
    e.pos = x0
    loss = 0
    for _ in range(case["m"] * case["cycles"]):
        e.advance(1)
        loss = loss + e.F[:, 0].mean()
    loss = loss / (case["m"] * case["cycles"])
    dzeta, dpos = torch.autograd.grad(loss, (zeta, x0))
    return {"loss": loss.detach(), "dzeta": dzeta, "dpos": dpos}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if kind == "replicas":
            c = _replicas(case, seed)
            e = _Exact(c["dims"], c["n_sub"], c["variant"], c["zeta"], c["seed"], KT)
            e.add(np.repeat(np.arange(case["replicas"]), c["n_particles"]), np.concatenate(c["pos"]),
                  np.concatenate(c["vel"]))
            samples = []
            for _ in range(case["steps"] // SAMPLE_EVERY):
                e.advance(SAMPLE_EVERY)
                row = torch.cat([(e.vel ** 2).sum(1, keepdim=True), e.vel, torch.ones_like(e.vel[:, :1])], 1)
                samples.append(torch.zeros(case["replicas"], 5, dtype=torch.float64, device="cuda")
                               .index_add(0, e.box, row))
            return _kinetic(torch.stack(samples))
        if kind == "kg":
            lp = lj_units.lattice_params(case["m"], case["dt"], case["zeta"])
            shape = (case["box"],) * 3
            pos, bonds = inputs.self_avoiding_chains(case["chains"], case["beads"], shape, seed)
            vel = inputs.maxwell_velocities(pos.shape[0], lp["kT"], seed)
            e = _Exact([shape], [case["m"]], case["variant"], lp["zeta"], [seed], lp["kT"], nu=lp["nu"],
                       half_step=case["integrator"] == "half_step")
            e.bonds = (torch.as_tensor(bonds.T.copy(), device="cuda"), "fene", lp["fene_k"], lp["fene_R0"])
            e.lj = (lp["lj_eps"], lp["lj_sigma"], lp["lj_rc"])
        else:
            pos, vel, bonds = _particles(case, seed)
            e = _Exact([(case["nx"], case["ny"], case["nz"])], [case["m"]], case["variant"], case["zeta"], [seed], KT,
                       force=(case["force"], 0.0, 0.0), gauss=case["noise"] == "gauss",
                       half_step=case["integrator"] == "half_step")
            if bonds is not None:
                e.bonds = (torch.as_tensor(bonds.T.copy(), device="cuda"), "harmonic", *SPRING)
        e.add(np.zeros(pos.shape[0], dtype=np.int64), pos, vel)
        if case.get("io") == "host":
            for _ in range(case["cycles"]):
                e.pos, e.vel = (torch.as_tensor(a, device="cuda") for a in (pos, vel))
                e.advance(case["m"])
            kT = (e.vel ** 2).sum() / (3 * case["n"])
            return {"pos": e.pos, "vel": e.vel,
                    "observables": torch.cat([torch.stack([kT, e.rho.sum()]), e.vel.sum(0)])}
        e.advance(case["m"] * case["cycles"])
        out = {"pos": e.pos, "vel": e.vel}
        if case.get("io") == "field":
            out["field"] = torch.cat([e.rho[None], e.j]).T.contiguous()
        return out
