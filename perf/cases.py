"""Performance cases: what a user of this library has it do, through its public entry points.

A case names a body (its grid or cloud, material and loads), the form of the computation (FP64 or
mixed, linearized or nonlinear bonds, influence function, solver) and the number of steps between two
reads of the state.  `prepare` builds the simulation and draws the initial displacement and velocity
from the seed; one `run` advances it by the steps of one read interval and reads u, v and theta (and
the damage, where a program that watches a crack does), as a program that follows the run does.

`exact` restates the same steps in plain torch in 64 bits, direction by direction over the grid.

The steps of the mixed form carry about single precision (FP32 bond arithmetic), so their programs
keep the frames they read as float32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2309_11273_gb300 import PD_FP64, PD_MIXED, BatchSimulation, Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W


def listed():
    return [
        # The paper's smallest plates (Section 4.1's convergence studies): 40 x 40 particles in free
        # vibration, read every 100 steps.  One step is a few microseconds: launches and latency.
        dict(name="plate_small_fp64", kind="plate", nx=40, ny=40, nz=1, ratio=3.015, form="fp64", steps=100),
        # A plate with an edge crack under traction (Section 4.2), the working size of 2D fracture
        # studies, followed with the damage field.
        dict(name="cracked_plate_fp64", kind="cracked", nx=400, ny=160, nz=1, ratio=3.015, form="fp64", steps=100),
        # Kalthoff-Winkler impact (Section 4.3) at the paper's node count, FP32 bonds.
        dict(name="impact_plate_mixed", kind="impact", nx=402, ny=201, nz=1, ratio=3.015, form="mixed", steps=100),
        # A sweep over many uneven plates (sizes, materials, horizons) stepped in one context.
        dict(name="plate_batch_mixed", kind="batch", nx=200, ny=200, nz=128, ratio=0.0, form="mixed", steps=50),
        # The notched 3D block under torsion (Section 4.4 in shape), one million particles: the FP64
        # form, the mixed form, and odd sizes in the nonlinear forms.
        dict(name="block_fp64", kind="block", nx=200, ny=100, nz=50, ratio=3.015, form="fp64", steps=20),
        dict(name="block_mixed", kind="block", nx=200, ny=100, nz=50, ratio=3.015, form="mixed", steps=100),
        dict(name="block_large_mixed", kind="block", nx=301, ny=153, nz=75, ratio=3.015, form="mixed", steps=50),
        dict(name="block_nonlinear_fp64", kind="block", nx=101, ny=50, nz=49, ratio=3.015, form="fp64_nl", steps=20),
        dict(name="block_nonlinear_mixed", kind="block", nx=157, ny=83, nz=41, ratio=3.015, form="mixed_nl", steps=50),
        # Quasi-static loading of a small 3D block by adaptive dynamic relaxation (Section 4.4's solver).
        dict(name="relaxation_fp64", kind="static", nx=60, ny=30, nz=25, ratio=3.015, form="adr", steps=50),
        # An unstructured body: a scattered 3D cloud with uneven volumes (no lattice), mixed form.
        dict(name="cloud_mixed", kind="cloud", nx=64, ny=48, nz=40, ratio=3.015, form="mixed", steps=50),
        # Coupling to another solver: the state goes out to the host and back in every step (pinned
        # buffers), as the end-to-end measurement of the benchmark does.
        dict(name="exchange_fp64", kind="exchange", nx=100, ny=100, nz=50, ratio=3.015, form="fp64", steps=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plate", "cracked", "cracked", "impact", "batch", "block", "block", "block", "static", "cloud",
                       "exchange"])
    ratio = rng.choice([3.015, 3.015, 4.015])
    steps = rng.choice([20, 25, 50, 64, 100])
    if kind in ("plate", "cracked", "impact"):
        nx, ny, nz = _log_int(rng, 30, 500), _log_int(rng, 30, 240), 1
        form = rng.choice(["fp64", "fp64", "mixed", "mixed_lo", "fp64_winv", "mixed_winv", "fp64_nl", "mixed_nl"])
        ny += ny % 2  # the edge crack runs between two rows
    elif kind == "batch":
        nx = _log_int(rng, 40, 200)
        ny, nz, ratio = nx, _log_int(rng, 4, 128), 0.0
        form = rng.choice(["fp64", "mixed", "mixed_nl"])
    elif kind == "cloud":
        nx, ny, nz = _log_int(rng, 12, 64), _log_int(rng, 12, 48), _log_int(rng, 12, 40)
        form = rng.choice(["fp64", "mixed", "mixed_nl"])
        ratio, steps = 3.015, min(steps, 50)
    elif kind == "static":
        nx, ny, nz = _log_int(rng, 12, 100), _log_int(rng, 12, 50), _log_int(rng, 12, 40)
        form, ratio, steps = "adr", 3.015, min(steps, 25)
    elif kind == "exchange":
        nx, ny, nz = _log_int(rng, 20, 120), _log_int(rng, 20, 100), _log_int(rng, 12, 50)
        form, ratio, steps = rng.choice(["fp64", "mixed"]), 3.015, 1
    else:
        nx, ny, nz = _log_int(rng, 24, 200), _log_int(rng, 16, 100), _log_int(rng, 12, 50)
        form = rng.choice(["fp64", "mixed", "mixed", "mixed_lo", "mixed_winv", "fp64_nl", "mixed_nl"])
        if form == "fp64_nl":
            nx, ny, nz, ratio = min(nx, 100), min(ny, 50), min(nz, 48), 3.015
        if ratio > 4:
            nx, ny, nz = min(nx, 120), min(ny, 60), min(nz, 40)
    if form.startswith("fp64") and nz > 1 and kind != "batch":
        steps = min(steps, 20)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, ratio=ratio, form=form, steps=steps)


# ------------------------------------------------------------------------------------- workloads
def _smooth(rng, w, amp, modes=4):
    """A smooth random vector field of rms amplitude amp: a sum of plane waves of 1 to 3 periods
    over the body."""
    X = [w.x, w.y] if w.z is None else [w.x, w.y, w.z]
    X = [x / (x.max() + w.dx) for x in X]
    u = np.zeros((w.dim, w.n))
    for _ in range(modes):
        k = rng.uniform(-3.0, 3.0, size=w.dim)
        phase = rng.uniform(0.0, 2.0 * np.pi)
        s = np.sin(sum(2.0 * np.pi * k[c] * X[c] for c in range(w.dim)) + phase)
        u += rng.normal(size=(w.dim, 1)) * s[None, :]
    return amp * u / np.sqrt(modes / 2.0)


def _cloud(case, rng):
    """A jittered 3D grid with uneven volumes; no load, no failure."""
    dx = 1e-3
    x, y, z = W.grid_3d(case["nx"], case["ny"], case["nz"], dx)
    x, y, z = (a + rng.uniform(-0.2, 0.2, a.size) * dx for a in (x, y, z))
    return W.Workload("cloud", W.MODEL_3D, dx=dx, delta=case["ratio"] * dx, dt=2e-7, nsteps=1000, x=x, y=y, z=z,
                      vol=dx ** 3 * rng.uniform(0.8, 1.2, x.size), **W.CONCRETE)


def _workload(case, seed):
    """The body of a case with its loads, and the random initial state of the seed."""
    rng = np.random.default_rng(seed)
    kind, nx, ny, nz, ratio = case["kind"], case["nx"], case["ny"], case["nz"], case["ratio"]
    # the time steps are 0.8 of the stable one for w = 1 at horizon 3.015 dx; a larger horizon allows more,
    # w = delta / |xi|, which weighs the short bonds, less
    slow = 0.7 if case["form"].endswith("_winv") else 1.0
    if kind == "plate":
        return W.plate_vibration(nx=nx, ny=ny, ratio=ratio, seed=seed, dt=2.6954e-7 * slow)
    if kind == "cracked":
        w = W.cracked_plate(nx=nx, ny=ny, ratio=ratio, crack_cells=float(nx // 2) + 0.125, dt=6.7385e-8 * slow)
        # pulled to about half of the critical stretch across the crack, over a random smooth field
        s0 = _critical_stretch(w)
        w.u0 = _smooth(rng, w, 0.01 * s0 * w.y.max())
        w.u0[1] += 0.4 * s0 * (w.y - 0.5 * w.y.max())
        return w
    if kind == "impact":
        gap = 2 * max(2, ny // 4)
        w = W.kalthoff(nx=nx, ny=ny, ratio=ratio, gap_cells=gap, notch_cells=float(nx // 4) + 0.125, dt=2e-8 * slow)
        w.u0 = _smooth(rng, w, 1e-8)
        return w
    if kind == "static":
        x, y, z = W.grid_3d(nx, ny, nz, 1e-3)
        flag = np.where(np.arange(x.size) % nx < 3, W.FIXED, W.FREE).astype(np.uint8)
        w = W.Workload("static", W.MODEL_3D, dx=1e-3, delta=ratio * 1e-3, dt=3.79e-7, nsteps=1000, x=x, y=y, z=z,
                       vol=np.full(x.size, 1e-9), flag=flag, **W.CONCRETE)
        # its own weight, of a random density: where the velocities change sign the solver's damping, a
        # Rayleigh quotient with the velocity in its denominator, would amplify any rounding
        w.b = np.zeros((3, x.size))
        w.b[2] = -rng.uniform(1e6, 4e6)
        return w
    if kind == "cloud":
        w = _cloud(case, rng)
        w.u0 = _smooth(rng, w, 1e-6)
        return w
    # block and exchange: a run of 20,000 steps of the clamped, twisted, notched block
    w = W.notched_block(nx=nx, ny=ny, nz=nz, ratio=ratio, nsteps=20000, dt=3.79e-7 * slow)
    w.u0 = _smooth(rng, w, 4e-7) * np.sin(np.pi * w.x / w.x.max())[None, :]
    w.u0[:, w.flag != W.FREE] = 0.0
    return w


def _batch(case, seed):
    bw = W.plate_batch(nplates=case["nz"], side_lo=max(16, case["nx"] // 10), side_hi=case["nx"])
    rng = np.random.default_rng(seed)
    for w in bw.bodies:
        w.u0 = _smooth(rng, w, 1e-7, modes=2)
    return bw


# --------------------------------------------------------------------------------------- the runs
class _State:
    pass


def prepare(case, seed):
    form = case["form"]
    kw = dict(precision=PD_MIXED if form.startswith("mixed") else PD_FP64,
              kinematics=B.PD_NONLINEAR if form.endswith("_nl") else B.PD_LINEARIZED,
              influence=B.PD_W_INV if form.endswith("_winv") else B.PD_W_ONE)
    s = _State()
    s.steps = case["steps"]
    s.single = form.startswith("mixed")
    s.damage = case["kind"] == "cracked"
    s.io = None
    if case["kind"] == "batch":
        s.sim = BatchSimulation(_batch(case, seed), **kw)
        return s
    w = _workload(case, seed)
    s.sim = Simulation(w, shadow_lo=1 if form == "mixed_lo" else None, **kw)
    if form == "adr":
        s.sim.set_option(B.PD_OPT_SOLVER, B.PD_SOLVER_ADR)
    if case["kind"] == "exchange":
        s.io = [torch.zeros((w.dim, w.n), dtype=torch.float64).pin_memory().numpy() for _ in range(2)]
        s.io[0][:] = w.initial_u()
        s.io[1][:] = w.initial_v()
    return s


def run(s):
    sim = s.sim
    if s.io is not None:
        u, v = s.io
        sim.set_state(u, v)
        sim.step(s.steps)
        B.pd_get_state(sim.h, sim.dim, sim.n, u=u, v=v, theta=False)
        return _frame(s, {"u": u, "v": v})
    sim.step(s.steps)
    u, v, theta = sim.state()
    out = {"u": u, "v": v, "theta": theta}
    if s.damage:
        out["phi"] = sim.damage()
    return _frame(s, out)


def _frame(s, out):
    if not s.single:
        return out
    return {k: torch.from_numpy(a).to(torch.float32) for k, a in out.items()}


# --------------------------------------------------------------------- sizes, as one pass needs them
def _counts(case):
    """(particles, directed bonds, dimension); interior families times the particles."""
    d = 2 if case["kind"] == "batch" or case["nz"] == 1 else 3
    fam = {(2, False): 28.0, (2, True): 48.0, (3, False): 122.0, (3, True): 256.0}
    if case["kind"] == "batch":
        n = case["nz"] * (0.55 * case["nx"]) ** 2
        return n, n * 38.0 * 0.95, d
    n = float(case["nx"] * case["ny"] * case["nz"])
    sides = [case["nx"], case["ny"]] + ([case["nz"]] if d == 3 else [])
    return n, n * fam[(d, case["ratio"] > 4)] * float(np.prod([1.0 - 1.2 / s for s in sides])), d


def work(case):
    """Per step the two passes over the bonds: the neighbour index (4 bytes), the status bit, and
    per particle x, u, theta, v and the per-particle constants; once per pass the state read.  Flops:
    the difference, dot product, sums and force of each bond (an FMA counts two); the nonlinear
    forms add the root, the division and the deformed direction."""
    n, nb, d = _counts(case)
    word = 4 if case["form"].startswith("mixed") else 8
    per_particle = word * (2 * d + 2 * d + 2) + 8 * 4 * d + 16
    step_bytes = 8.4 * nb + per_particle * n
    flops = (36.0 if case["form"].endswith("_nl") else 19.0) * nb
    io = n * 8 * (2 * d + (0 if case["kind"] == "exchange" else 1))
    if case["kind"] == "exchange":
        io += n * 8 * 2 * d
    return {"bytes": case["steps"] * step_bytes + io, "flops": case["steps"] * flops}


# ----------------------------------------------------------------- the same steps, plainly in 64 bits
def _constants(w):
    """A, K, G of Eqs 1.8, 1.15, 1.16."""
    E, nu = w.E, w.nu
    kappa, mu = E / (3 * (1 - 2 * nu)), E / (2 * (1 + nu))
    if w.model == W.MODEL_3D:
        return 3.0, 3 * kappa, 15 * mu
    if w.model == W.MODEL_PLANE_STRESS:
        return (2 * (1 - 2 * nu) / (1 - nu),
                2 * kappa * (1 - 2 * nu) / (1 - nu) - 2 / 3 * mu * (1 + nu) * (1 - 3 * nu) / ((1 - nu) * (1 - 2 * nu)),
                8 * mu)
    return 2.0, 2 * kappa - 2 / 3 * mu, 8 * mu


def _critical_stretch(w):
    """s_c of Eqs 1.26-1.29."""
    if not w.Gc:
        return 0.0
    kappa, mu = w.E / (3 * (1 - 2 * w.nu)), w.E / (2 * (1 + w.nu))
    if w.model == W.MODEL_3D:
        return math.sqrt(w.Gc / ((9 * kappa - 15 * mu) * 125 * w.delta / 1848 + 15 * mu * 5 * w.delta / 24))
    A, _, _ = _constants(w)
    kp = kappa + mu / 9 * (((1 + w.nu) / (1 - 2 * w.nu)) ** 2 if w.model == W.MODEL_PLANE_STRESS else 1.0)
    beta, betap = 1087 * w.delta / (1250 * math.pi ** 2), 4 * w.delta / (5 * math.pi)
    return math.sqrt(w.Gc / (A * A * (kp - 8 * mu / 9) * beta + 8 * mu * betap))


def _cut(a, b, crack, d):
    """Bonds a-b crossing the crack: ends strictly on opposite sides, crossing point on it."""
    p = torch.tensor(crack, dtype=torch.float64, device=a.device).reshape(3, 3)
    p0 = p[0, :d, None]
    e1 = p[1, :d, None] - p0
    if d == 2:
        normal = torch.stack([-e1[1], e1[0]])
    else:
        e2 = p[2, :d, None] - p0
        normal = torch.linalg.cross(e1[:, 0], e2[:, 0])[:, None]
    sa, sb = (normal * (a - p0)).sum(0), (normal * (b - p0)).sum(0)
    opposite = ((sa > 0) & (sb < 0)) | ((sa < 0) & (sb > 0))
    r = a + (sa / (sa - sb)) * (b - a) - p0
    if d == 2:
        lam = (r * e1).sum(0) / (e1 * e1).sum()
        return opposite & (lam >= 0) & (lam <= 1)
    g11, g12, g22 = (e1 * e1).sum(), (e1 * e2).sum(), (e2 * e2).sum()
    r1, r2 = (r * e1).sum(0), (r * e2).sum(0)
    det = g11 * g22 - g12 * g12
    al, be = (r1 * g22 - r2 * g12) / det, (g11 * r2 - g12 * r1) / det
    return opposite & (al >= 0) & (al <= 1) & (be >= 0) & (be <= 1)


class _Exact:
    """Bodies given on (jittered) grids, one direction of the grid at a time over all particles."""

    def __init__(self, bodies, shapes, jitter, kin, winv):
        dev = self.dev = torch.device("cuda")

        def per(vals):
            return torch.cat([torch.full((w.n,), float(v), dtype=torch.float64) for w, v in zip(bodies, vals)]).to(dev)

        def cat(arrs):
            return torch.from_numpy(np.concatenate(arrs, axis=-1)).to(dev)

        w0 = bodies[0]
        d = self.d = w0.dim
        self.kin = kin
        self.X = cat([np.stack([w.x, w.y] if d == 2 else [w.x, w.y, w.z]) for w in bodies])
        self.V = cat([w.vol for w in bodies])
        consts = [_constants(w) for w in bodies]
        self.A, self.K, self.G = (per([c[t] for c in consts]) for t in range(3))
        self.s0 = per([_critical_stretch(w) for w in bodies])
        self.dt, self.rho, delta = per([w.dt for w in bodies]), per([w.rho for w in bodies]), per([w.delta for w in bodies])
        self.u, self.v = cat([w.initial_u() for w in bodies]).clone(), cat([w.initial_v() for w in bodies]).clone()
        self.b = cat([w.b for w in bodies]) if w0.b is not None else torch.zeros_like(self.u)
        n = self.V.numel()
        ids = torch.arange(n, device=dev)
        off = per(np.concatenate([[0], np.cumsum([w.n for w in bodies])])[:-1]).long()
        size = [per([s[t] for s in shapes]).long() for t in range(3)]
        loc = ids - off
        g = [loc % size[0], (loc // size[0]) % size[1], loc // (size[0] * size[1])]
        R = int(math.ceil(max(w.delta / w.dx for w in bodies) + 2 * jitter)) if jitter else \
            int(math.floor(max(w.delta / w.dx for w in bodies)))
        reach = max(w.delta / w.dx for w in bodies) + 2 * jitter * math.sqrt(d)
        self.bonds = []  # (particles i, neighbours j, intact) of each direction that has bonds
        for oz in range(-R if d == 3 else 0, (R if d == 3 else 0) + 1):
            for oy in range(-R, R + 1):
                for ox in range(-R, R + 1):
                    if (ox, oy, oz) == (0, 0, 0) or ox * ox + oy * oy + oz * oz > reach * reach:
                        continue
                    ok = torch.ones(n, dtype=torch.bool, device=dev)
                    for t, o in enumerate((ox, oy, oz)):
                        ok &= (g[t] + o >= 0) & (g[t] + o < size[t])
                    i = ids[ok]
                    j = i + ox + oy * size[0][i] + oz * size[0][i] * size[1][i]
                    xi = self.X[:, j] - self.X[:, i]
                    keep = (xi * xi).sum(0) <= delta[i] ** 2
                    for c in w0.cracks if len(bodies) == 1 else []:
                        keep &= ~_cut(self.X[:, i], self.X[:, j], c, d)
                    i, j = i[keep], j[keep]
                    if i.numel():
                        self.bonds.append([i, j, torch.ones(i.numel(), dtype=torch.bool, device=dev)])
        self.delta, self.winv = delta, winv
        self.m, self.den = torch.zeros_like(self.V), torch.zeros_like(self.V)
        for i, j, _ in self.bonds:
            xi = self.X[:, j] - self.X[:, i]
            q = (xi * xi).sum(0)
            wt = self._w(i, q)
            self.m[i] += wt * q * self.V[j]
            self.den[i] += wt * self.V[j]
        self.mi = torch.where(self.m > 0, 1.0 / self.m, torch.zeros_like(self.m))
        self.n, self.t, self.theta = n, 0, None
        self.fixed = self.moved = None
        if len(bodies) == 1 and w0.flag is not None:
            flag = torch.from_numpy(w0.flag).to(dev)
            self.fixed, self.moved = flag == W.FIXED, flag == W.PRESCRIBED
            if w0.vp is not None:
                self.motion = torch.from_numpy(w0.vp).to(dev)
            else:
                a = torch.from_numpy(w0.axis_dir if w0.axis_dir is not None else np.zeros(3)).to(dev)
                c = torch.from_numpy(w0.axis_point if w0.axis_point is not None else np.zeros(3)).to(dev)
                r = self.X - c[:d, None]
                self.motion = w0.rotation_rate(_critical_stretch(w0)) * torch.linalg.cross(
                    a[:, None].expand_as(r).contiguous(), r, dim=0) if d == 3 else torch.zeros_like(self.u)
            self._constrain()

    def _w(self, i, q):
        return self.delta[i] / q.sqrt() if self.winv else torch.ones_like(q)

    def _constrain(self):
        if self.fixed is None:
            return
        self.u[:, self.fixed] = 0.0
        self.v[:, self.fixed] = 0.0
        time = self.t * self.dt[0]
        self.u[:, self.moved] = time * self.motion[:, self.moved]
        self.v[:, self.moved] = self.motion[:, self.moved]

    def _bond(self, i, j):
        """xi, |xi|, e and the direction of the force."""
        xi = self.X[:, j] - self.X[:, i]
        eta = self.u[:, j] - self.u[:, i]
        x = (xi * xi).sum(0).sqrt()
        if not self.kin:
            return x, (xi * eta).sum(0) / x, xi / x
        Y = xi + eta
        y = (Y * Y).sum(0).sqrt()
        return x, ((2 * xi + eta) * eta).sum(0) / (y + x), Y / y

    def check(self):
        if bool((self.s0 > 0).any()):
            for rec in self.bonds:
                i, j, intact = rec
                x, e, _ = self._bond(i, j)
                s0 = self.s0[i]
                rec[2] = intact & ~((s0 > 0) & (e / x >= s0))

    def force(self):
        th = torch.zeros_like(self.V)
        for i, j, intact in self.bonds:
            x, e, _ = self._bond(i, j)
            th[i] += torch.where(intact, self._w(i, x * x) * x * e * self.V[j], torch.zeros_like(e))
        self.theta = th = self.A * self.mi * th
        f = torch.zeros_like(self.u)
        p, g = (self.K - self.G / 3) * th * self.mi, self.G * self.mi
        for i, j, intact in self.bonds:
            x, e, M = self._bond(i, j)
            c = torch.where(intact, self._w(i, x * x) * ((p[i] + p[j]) * x + (g[i] + g[j]) * e) * self.V[j],
                            torch.zeros_like(e))
            f[:, i] += c * M
        return f

    def step(self):
        f = self.force()
        self.t += 1
        self.v = self.v + self.dt * ((f + self.b) / self.rho)
        self.u = self.u + self.dt * self.v
        self._constrain()
        self.check()

    def density(self):
        """The fictitious density of the relaxation solver: a quarter of a bound of the absolute row
        sums of the force-density stiffness."""
        alpha, rg, rt = (torch.zeros_like(self.V) for _ in range(3))
        for i, j, _ in self.bonds:
            xi = self.X[:, j] - self.X[:, i]
            alpha[i] += xi.abs().sum(0) * self.V[j]
        alpha = self.A * self.mi * alpha
        for i, j, _ in self.bonds:
            xi = self.X[:, j] - self.X[:, i]
            x = (xi * xi).sum(0).sqrt()
            rg[i] += (self.mi[i] + self.mi[j]) * self.V[j] * xi.abs().sum(0) / x
            rt[i] += x * self.V[j] * (alpha[i] * self.mi[i] + alpha[j] * self.mi[j])
        return 0.25 * (2 * self.G * rg + 2 * (self.K - self.G / 3).abs() * rt)

    def relax(self, lam, last):
        g = self.force() + self.b
        free = ~self.fixed if self.fixed is not None else torch.ones(self.n, dtype=torch.bool, device=self.dev)
        if last is None:
            v = g / (2 * lam)
        else:
            k = torch.where(self.v != 0, -(g - last) / (lam * self.v), torch.zeros_like(g))
            num, den = float((self.u * k * self.u)[:, free].sum()), float((self.u * self.u)[:, free].sum())
            c = 2 * math.sqrt(num / den) if num > 0 and den > 0 else 0.0
            v = ((2 - c) * self.v + 2 * g / lam) / (2 + c)
        self.t += 1
        self.v = v
        self.u = self.u + v
        self._constrain()
        return g


def exact(case, seed):
    n, nb, _ = _counts(case)
    if nb * case["steps"] > 1.3e10 or not torch.cuda.is_available():
        return None  # over about 20 seconds
    nl, winv = case["form"].endswith("_nl"), case["form"].endswith("_winv")
    if case["kind"] == "batch":
        bodies = _batch(case, seed).bodies
        shapes = [(int(round(w.x.max() / w.dx + 0.5)), int(round(w.y.max() / w.dx + 0.5)), 1) for w in bodies]
    else:
        bodies, shapes = [_workload(case, seed)], [(case["nx"], case["ny"], case["nz"])]
    r = _Exact(bodies, shapes, 0.2 if case["kind"] == "cloud" else 0.0, nl, winv)
    if case["form"] == "adr":
        lam, last = r.density(), None
        for _ in range(case["steps"]):
            last = r.relax(lam, last)
    else:
        for _ in range(case["steps"]):
            r.step()
    out = {"u": r.u, "v": r.v}
    if case["kind"] != "exchange":
        out["theta"] = r.theta
    if case["kind"] == "cracked":
        num = torch.zeros_like(r.V)
        for i, j, intact in r.bonds:
            xi = r.X[:, j] - r.X[:, i]
            num[i] += torch.where(intact, r._w(i, (xi * xi).sum(0)) * r.V[j], torch.zeros_like(r.V[j]))
        out["phi"] = torch.where(r.den > 0, 1 - num / r.den, torch.zeros_like(num))
    return {k: a.cpu().numpy() for k, a in out.items()}
