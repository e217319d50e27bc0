"""Performance cases of the SPH engine: what a user's program has it do.

Three kinds of call, each through the package's public entry points:

- ``run``: one resident case (``Engine.create``), advanced by a chunk of steps
  (``Engine.step``) and read out as a frame (``Engine.get_state`` into the
  program's own page-locked buffers), the loop of every simulation;
- ``batch``: many uneven cases in one engine (``Engine.batch``), advanced
  together and all read out, the loop of a parameter study;
- ``serve``: a resident pool (``Engine.pool``) to which a server
  (``serve.Server``) admits requests of different sizes, steps them to their
  end times, reads their results and releases them.

The cases come from the package's seeded generators (``cases``), with the
tank, column and flume sizes of its tests and benchmark; only the particle
spacing sets the particle count.  Every fluid starts in motion: a seeded,
divergence-free stir and a disorder of 5 % of the spacing, so that the first
pass already crosses cells, rebuilds neighbour lists and has every term of the
interaction at work, as a flow has after its first instants.

A frame is positions, velocities, densities and pressures of all particles in
the caller's order, with the simulated time; positions are handed on in single
precision, as simulation frames are written.

``exact`` is the same computation in 64-bit PyTorch, from the equations of the
method (Wendland C2, weakly compressible; Symplectic and Verlet schemes,
density diffusion, artificial or laminar + SPS viscosity, dynamic and modified
dynamic boundaries).
"""
import math

import numpy as np
import torch

from paper_2104_00537_gb300 import cases as gen
from paper_2104_00537_gb300 import serve, sph

G = 9.81


def _run(name, shape, dp, **kw):
    c = dict(name=name, kind="run", shape=shape, dp=dp, steps=10, cell_mode=1, graph=True,
             pair_once=False, integrator=0, ddt_mode=1, visc_mode=0, boundary_mode=0)
    c.update(kw)
    return c


def listed():
    return [
        # a first try-out of a set-up at coarse resolution (6k particles): all
        # latency and launches; the engine as it is created, no options set
        _run("dam_break_6k", "dam_break", 0.04, cell_mode=0, graph=False),
        # the small validation dam break (28k particles), graph replay
        _run("dam_break_28k", "dam_break", 0.02),
        # a sloshing tank moved as a whole (imposed motion of every wall), of the
        # size in the middle of the served range
        _run("sloshing_167k", "sloshing", 0.0106),
        # the same kind of run with each pair evaluated once
        _run("dam_break_220k_once", "dam_break", 0.0083, pair_once=True),
        # the production dam break (1.48M particles): reproducible sums ...
        _run("dam_break_1.5M", "dam_break", 0.004),
        # ... and each pair once, the benchmark's mode
        _run("dam_break_1.5M_once", "dam_break", 0.004, pair_once=True),
        # a long wave flume with its piston: the largest run
        _run("flume_4M_once", "flume", 0.0163, steps=5, pair_once=True),
        # the Verlet scheme: one evaluation per step
        _run("verlet_410k", "dam_break", 0.0065, integrator=1),
        # laminar viscosity + SPS turbulence
        _run("sps_270k", "dam_break", 0.0077, visc_mode=1),
        # modified dynamic boundaries with the Fourtakas density diffusion
        _run("mdbc_190k", "dam_break", 0.0105, boundary_mode=1, ddt_mode=2),
        # a parameter study: uneven dam breaks in one engine
        dict(name="batch_12", kind="batch", cases=12, geometry=1, n_min=5000, n_max=120000,
             steps=10, cell_mode=1, pair_once=False),
        # a server's burst of requests of different sizes, to their end times
        dict(name="serve_8", kind="serve", requests=8, geometry=1, n_min=10000, n_max=60000,
             chunk=10, t_end=0.004, cell_mode=1, pair_once=False),
    ]


def draw(rng):
    """One more case: kinds and options as listed, spacings log-uniform over
    the listed range of particle counts."""
    def log_uniform(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    kind = rng.choice(["run"] * 6 + ["physics"] * 3 + ["batch", "serve"])
    if kind in ("run", "physics"):
        shape = rng.choice(["dam_break", "sloshing", "flume"])
        # the finest drawn spacing of a shape gives at most the particles of
        # the largest listed case; the costlier physics starts coarser
        fine = {"dam_break": 0.004, "sloshing": 0.0045, "flume": 0.018}[shape]
        coarse = {"dam_break": 0.04, "sloshing": 0.03, "flume": 0.06}[shape]
        if kind == "physics":
            fine *= 1.6
        dp = round(log_uniform(fine, coarse), 5)
        c = _run("", shape, dp, steps=5 if shape == "flume" else 10,
                 pair_once=rng.random() < 0.5, graph=rng.random() < 0.75,
                 cell_mode=1 if rng.random() < 0.8 else 0)
        if kind == "physics":
            which = rng.choice(["verlet", "sps", "mdbc", "fourtakas"])
            if which == "verlet":
                c["integrator"] = 1
            elif which == "sps":
                c["visc_mode"] = 1
            elif which == "mdbc":
                c["boundary_mode"] = 1
                c["shape"] = "dam_break"
                c["dp"] = round(log_uniform(0.0075, 0.03), 5)
                c["steps"] = 10
            if which in ("mdbc", "fourtakas"):
                c["ddt_mode"] = 2
            c["pair_once"] = which == "verlet" and c["pair_once"]
    elif kind == "batch":
        c = dict(kind="batch", cases=rng.randint(4, 12), geometry=rng.randint(2, 9999),
                 n_min=5000, n_max=int(log_uniform(12000, 120000)), steps=10, cell_mode=1,
                 pair_once=rng.random() < 0.5)
    else:
        c = dict(kind="serve", requests=rng.randint(3, 8), geometry=rng.randint(2, 9999),
                 n_min=10000, n_max=int(log_uniform(20000, 60000)), chunk=10,
                 t_end=round(rng.uniform(0.002, 0.004), 4), cell_mode=1,
                 pair_once=rng.random() < 0.5)
    c.pop("name", None)
    return c


# ---- inputs -------------------------------------------------------------------

def _stir(c, seed):
    """Seeded motion and disorder of the case's fluid: rolls in the x-z plane
    (the curl of a stream function that vanishes on the walls, the bottom and
    the still surface, varied along y: divergence-free), and 5 % of the
    spacing of position noise."""
    f = c.ptype == 0
    rng = np.random.default_rng([seed, 77])
    p = c.pos[f]
    lo, hi = p.min(0), p.max(0)
    L = hi - lo
    X = (p - lo) / L
    speed = 0.25 * math.sqrt(G * L[2])
    v = np.zeros_like(p)
    for kx in (1, 2, 3):
        a = speed * rng.uniform(-1.0, 1.0) / kx
        ay, py = rng.uniform(0.0, 0.5), rng.uniform(0.0, 2.0 * math.pi)
        w = a * (1.0 + ay * np.sin(2.0 * math.pi * X[:, 1] + py))
        sx, cx = np.sin(kx * math.pi * X[:, 0]), np.cos(kx * math.pi * X[:, 0])
        sz, cz = np.sin(math.pi * X[:, 2]), np.cos(math.pi * X[:, 2])
        # psi = sin(kx pi X) sin(pi Z): (vx, vz) = (-dpsi/dz, dpsi/dx)
        q = L[2] / L[0] * kx
        s = 1.0 / max(1.0, q)
        v[:, 0] -= w * s * sx * cz
        v[:, 2] += w * s * q * cx * sz
    c.vel[f] += v.astype(np.float32)
    c.pos[f] += (0.05 * c.params["dp"]) * rng.uniform(-1.0, 1.0, p.shape)
    return c


def _physics(case):
    return {k: case[k] for k in ("cell_mode", "ddt_mode", "visc_mode", "boundary_mode",
                                 "integrator") if k in case}


def _inputs(case, seed):
    """The package's cases (host arrays) of one performance case."""
    kw = _physics(case)
    if case["kind"] == "run":
        dp = case["dp"]
        if case["shape"] == "dam_break":
            c = gen.dam_break(dp, seed=seed, **kw)
        elif case["shape"] == "flume":
            c = gen.wave_flume(dp, seed=seed, **kw)
        else:
            depth = 0.3
            c = gen.sloshing_tank(int(0.5 * depth / dp ** 3), depth, 0.03, 1.0, seed=seed, **kw)
        return [_stir(c, seed)]
    if case["kind"] == "batch":
        cs = gen.batch_dam_breaks(case["cases"], seed=case["geometry"], n_min=case["n_min"],
                                  n_max=case["n_max"], **kw)
    else:  # sizes, fill depths and excitations by "geometry", the flow by the seed
        u = np.random.default_rng([case["geometry"], 78]).uniform(size=(case["requests"], 4))
        cs = []
        for i in range(case["requests"]):
            n = case["n_min"] * (case["n_max"] / case["n_min"]) ** u[i, 0]
            cs.append(gen.sloshing_tank(int(n), 0.2 + 0.2 * u[i, 1], 0.01 + 0.04 * u[i, 2],
                                        0.5 + u[i, 3], seed=seed + 1 + i, **kw))
    return [_stir(c, seed + i) for i, c in enumerate(cs)]


def prepare(case, seed):
    cs = _inputs(case, seed)
    if case["kind"] == "serve":
        n = sum(c.n for c in cs)
        cells = 0
        for c in cs:
            p = c.params
            m = p["cell_mode"] + 1
            cs_ = 2.0 * p["h"] / m
            cells += math.prod(2 * m + 1 + int((b - a) / cs_)
                               for a, b in zip(p["domain_min"], p["domain_max"]))
        # room for a burst while the last one's particles are still in place
        pool = sph.Engine.pool(2 * n, 2 * cells, len(cs))
        pool.set_options(use_graph=1, pair_once=int(case["pair_once"]))
        return dict(case=case, pool=pool, cases=cs)
    if case["kind"] == "batch":
        eng = sph.Engine.batch(cs)
        eng.set_options(use_graph=1, pair_once=int(case["pair_once"]))
    else:
        eng = sph.Engine.create(cs[0])
        if case["graph"] or case["pair_once"]:
            eng.set_options(use_graph=int(case["graph"]), pair_once=int(case["pair_once"]))
    return dict(case=case, engine=eng, frames=[sph.state_buffers(c.n, pinned=True) for c in cs])


def _frame(s):
    """A frame as it is written: positions in single precision."""
    return dict(pos=torch.from_numpy(s["pos"]).float(), vel=s["vel"], rho=s["rho"],
                press=s["press"], t=np.float32(s["t"]))


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        reqs = [serve.Request(i, 0.0, c, case["t_end"]) for i, c in enumerate(state["cases"])]
        server = serve.Server(state["pool"], chunk=case["chunk"], keep_results=True)
        return [_frame(r.result) for r in server.run(reqs)]
    eng = state["engine"]
    eng.step(case["steps"])
    return [_frame(eng.get_state(i, out=f)) for i, f in enumerate(state["frames"])]


# ---- what a pass cannot do without ------------------------------------------------

def _sizes(case):
    """(fluid particles, all particles) of a performance case, about."""
    if case["kind"] == "run":
        dp = case["dp"]
        layers = 4 if case["boundary_mode"] == 1 else 2
        if case["shape"] == "dam_break":
            fl, walls = 0.4 ** 3, 1.6 * 0.67 + 2 * 0.6 * (1.6 + 0.67)
        elif case["shape"] == "flume":
            fl, walls = 25.0 * 1.0 * 0.6, 25.0 + 2 * 1.2 * 25.0 + 2 * 1.2
        else:
            fl, walls = 1.0 * 0.5 * 0.3, 0.5 + 2 * 0.6 * 1.5
        return fl / dp ** 3, fl / dp ** 3 + layers * walls / dp ** 2
    a, b = case["n_min"], case["n_max"]
    one = (b - a) / math.log(b / a)
    k = case["cases"] if case["kind"] == "batch" else case["requests"]
    return k * one, 2.0 * k * one


def work(case):
    """Flops: each unordered pair inside the support once per evaluation (56
    operations for two fluid particles: kernel, pressure, viscosity,
    continuity, density diffusion; SPS adds 108), about 85 per fluid particle.
    Bytes: each particle's 40 bytes of state in once, its 48 bytes of frame
    out once."""
    nf, n = _sizes(case)
    if case["kind"] == "serve":
        steps = case["t_end"] / 1.6e-4
    else:
        steps = case["steps"]
    evals = steps * (1 if case.get("integrator") == 1 else 2)
    per_pair = 56 + (108 if case.get("visc_mode") == 1 else 0)
    return {"bytes": 88.0 * n, "flops": 85.0 * nf * per_pair * evals}


# ---- the same in 64 bits ----------------------------------------------------------

CHUNK = 1 << 23  # pairs worked on at a time


class _Slow(Exception):
    """A case whose 64-bit computation would take too long."""


def _near(q, p, R):
    """All (i, j) with |q_i - p_j| < R, as two int32 tensors."""
    lo = torch.minimum(q.min(0).values, p.min(0).values) - 2.0 * R
    hi = torch.maximum(q.max(0).values, p.max(0).values) + 2.0 * R
    nc = ((hi - lo) / R).floor().long() + 1
    cq, cp = ((q - lo) / R).floor().long(), ((p - lo) / R).floor().long()
    key = (cp[:, 2] * nc[1] + cp[:, 1]) * nc[0] + cp[:, 0]
    order = key.argsort(stable=True)
    start = torch.zeros(int(nc.prod()) + 1, dtype=torch.long, device=q.device)
    start[1:] = torch.bincount(key, minlength=int(nc.prod())).cumsum(0)
    ps = p[order]
    base = (cq[:, 2] * nc[1] + cq[:, 1]) * nc[0] + cq[:, 0]
    rows = torch.tensor([int(dz) * int(nc[1] * nc[0]) + int(dy) * int(nc[0])
                         for dz in (-1, 0, 1) for dy in (-1, 0, 1)], device=q.device)
    out_i, out_j = [], []
    step = max(1, 1 << 17)
    for a in range(0, len(q), step):
        b = min(len(q), a + step)
        c = base[a:b, None] + rows[None, :]
        s, e = start[c - 1].reshape(-1), start[c + 2].reshape(-1)
        cnt = e - s
        total = int(cnt.sum())
        if not total:
            continue
        idx = torch.repeat_interleave(torch.arange(len(cnt), device=q.device), cnt)
        j = torch.arange(total, device=q.device) - (cnt.cumsum(0) - cnt)[idx] + s[idx]
        i = a + idx // len(rows)
        ok = ((q[i] - ps[j]) ** 2).sum(1) < R * R
        out_i.append(i[ok].int())
        out_j.append(order[j[ok]].int())
    none = torch.zeros(0, dtype=torch.int32, device=q.device)
    return (torch.cat(out_i), torch.cat(out_j)) if out_i else (none, none)


class _Exact:
    """One case advanced in 64 bits from its initial arrays."""

    def __init__(self, c, dev):
        p = c.params
        def t(x):
            return torch.as_tensor(np.array(x, np.float64), device=dev)
        self.p = p
        self.pos, self.vel, self.rho = t(c.pos), t(c.vel), t(c.rho)
        # velocities and densities enter as single precision numbers
        self.vel, self.rho = self.vel.float().double(), self.rho.float().double()
        self.fluid = torch.as_tensor(c.ptype == 0, device=dev)
        self.group = torch.as_tensor(c.group.astype(np.int64), device=dev)
        self.motions = c.motions
        self.ghost = t(c.ghost).float().double() if p["boundary_mode"] == 1 else None
        self.g = t(p["gravity"])
        self.t, self.step_no = 0.0, 0
        self.vp, self.rp = self.vel.clone(), self.rho.clone()
        self.h, self.m = p["h"], p["rho0"] * p["dp"] ** 3
        self.B = p["cs0"] ** 2 * p["rho0"] / p["gamma"]
        self.aD = 21.0 / (16.0 * math.pi * self.h ** 3)
        self.built = None  # positions at the pair list's build

    def tait(self, rho):
        return self.B * torch.expm1(self.p["gamma"] * torch.log(rho / self.p["rho0"]))

    def grad(self, r2):
        """F of grad_a W_ab = F r_ab, zero outside the support."""
        t = 1.0 - torch.sqrt(r2) / (2.0 * self.h)
        return torch.where(t > 0, -5.0 * self.aD / self.h ** 2 * t ** 3, torch.zeros_like(t))

    def lists(self):
        """Unordered pairs with a fluid particle (and the fluid around every
        ghost node) within 2h and a margin, kept while nothing moved out of it."""
        margin = 0.08 * self.h
        if self.built is not None and \
                float(((self.pos - self.built) ** 2).sum(1).max()) < (0.45 * margin) ** 2:
            return
        self.built = self.pos.clone()
        R = 2.0 * self.h + margin
        i, j = _near(self.pos, self.pos, R)
        ok = (i < j) & (self.fluid[i] | self.fluid[j])
        self.pairs = i[ok], j[ok]
        if self.ghost is not None:
            fl, bo = self.fluid.nonzero()[:, 0], (~self.fluid).nonzero()[:, 0]
            i, j = _near(self.pos[bo] + self.ghost[bo], self.pos[fl], R)
            self.near_ghost = bo, i, fl[j]

    def chunks(self, i, j):
        for k in range(0, len(i), CHUNK):
            yield i[k:k + CHUNK].long(), j[k:k + CHUNK].long()

    def stress(self):
        """tau / rho of the SPS model, six components per particle."""
        n = len(self.rho)
        grad = torch.zeros(n, 9, dtype=torch.float64, device=self.pos.device)
        for a, b in self.chunks(*self.pairs):
            r = self.pos[a] - self.pos[b]
            F = self.grad((r * r).sum(1))
            dv = self.vel[b] - self.vel[a]
            outer = (dv[:, :, None] * r[:, None, :]).reshape(-1, 9) * F[:, None]
            # the same product for b: both differences change sign
            grad.index_add_(0, a, outer * (self.m / self.rho[b])[:, None])
            grad.index_add_(0, b, outer * (self.m / self.rho[a])[:, None])
        D = grad.reshape(n, 3, 3)
        S = 0.5 * (D + D.transpose(1, 2))
        mag = 0.5 * torch.sqrt(2.0 * (S * S).sum((1, 2)))
        dp = self.p["dp"]
        nu = (0.12 * dp) ** 2 * mag
        tr = S.diagonal(dim1=1, dim2=2).sum(1)
        eye = torch.eye(3, dtype=torch.float64, device=S.device)
        tau = 2.0 * nu[:, None, None] * (S - tr[:, None, None] / 3.0 * eye) - \
            (2.0 / 3.0 * 0.0066 * dp ** 2 * mag ** 2)[:, None, None] * eye
        return torch.where(self.fluid[:, None, None], tau, torch.zeros_like(tau))

    def rho_hydro(self, r):
        x = -self.p["rho0"] / self.B * (r * self.g).sum(1)
        return self.p["rho0"] * torch.expm1(torch.log1p(x) / self.p["gamma"])

    def evaluate(self):
        """dv/dt, drho/dt and the largest mu of the current state."""
        p, n = self.p, len(self.rho)
        self.lists()
        if self.ghost is not None:
            self.walls()
        P = self.tait(self.rho)
        acc = torch.zeros(n, 3, dtype=torch.float64, device=self.pos.device)
        drho = torch.zeros(n, dtype=torch.float64, device=self.pos.device)
        tau = self.stress() if p["visc_mode"] == 1 else None
        mu_max = 0.0
        for a, b in self.chunks(*self.pairs):
            fa, fb = self.fluid[a], self.fluid[b]
            ra, rb = self.rho[a], self.rho[b]
            r, v = self.pos[a] - self.pos[b], self.vel[a] - self.vel[b]
            r2 = (r * r).sum(1)
            F = self.grad(r2)
            vr = (v * r).sum(1)
            ca, cb = ra * self.m / rb * F * vr, rb * self.m / ra * F * vr
            if p["boundary_mode"] == 1:
                ca, cb = ca * fa, cb * fb
            if p["ddt_mode"]:
                k = -2.0 * p["delta"] * self.h * p["cs0"] * F * (fa & fb)
                da, db = rb - ra, ra - rb
                if p["ddt_mode"] == 2:
                    da, db = da - self.rho_hydro(r), db - self.rho_hydro(-r)
                ca, cb = ca + k * da * self.m / rb, cb + k * db * self.m / ra
            drho.index_add_(0, a, ca)
            drho.index_add_(0, b, cb)
            s = self.m * (P[a] + P[b]) / (ra * rb)
            mu = self.h * vr / (r2 + p["eta2"])
            if p["visc_mode"] == 0:
                s = s - self.m * p["alpha"] * p["cs0"] * mu.clamp(max=0.0) / (0.5 * (ra + rb))
            f = -(s * F)[:, None] * r
            if tau is not None:
                f = f + (self.m * 4.0 * p["nu0"] * F * r2 /
                         ((ra + rb) * (r2 + p["eta2"])))[:, None] * v
                T = (ra[:, None, None] * tau[a] + rb[:, None, None] * tau[b]) / \
                    (ra * rb)[:, None, None]
                f = f + (self.m * F)[:, None] * (T @ r[:, :, None])[:, :, 0]
            acc.index_add_(0, a, f * fa[:, None])
            acc.index_add_(0, b, -f * fb[:, None])
            inside = r2 < 4.0 * self.h ** 2
            mu_max = max(mu_max, float((mu.abs() * inside).max()))
        acc += self.g * self.fluid[:, None]
        return acc, drho, mu_max

    def walls(self):
        """Densities of the boundary particles from their ghost nodes."""
        bo, i, fl = self.near_ghost
        nb = len(bo)
        M = torch.zeros(nb, 16, dtype=torch.float64, device=self.pos.device)
        rhs = torch.zeros(nb, 4, dtype=torch.float64, device=self.pos.device)
        xg = self.pos[bo] + self.ghost[bo]
        for a, b in self.chunks(i, fl):
            d = xg[a] - self.pos[b]
            r2 = (d * d).sum(1)
            t = (1.0 - torch.sqrt(r2) / (2.0 * self.h)).clamp(min=0.0)
            W = self.aD * t ** 4 * (5.0 - 4.0 * t)
            row = torch.cat([W[:, None], self.grad(r2)[:, None] * d], 1)
            e = torch.cat([torch.ones_like(W)[:, None], -d], 1)
            V = self.m / self.rho[b]
            M.index_add_(0, a, ((V[:, None] * row)[:, :, None] * e[:, None, :]).reshape(-1, 16))
            rhs.index_add_(0, a, self.m * row)
        M = M.reshape(nb, 4, 4)
        rho0 = self.p["rho0"]
        none = M[:, 0, 0] <= 0.0
        shepard = rhs[:, 0] / torch.where(none, torch.ones_like(rhs[:, 0]), M[:, 0, 0])
        use = torch.linalg.det(M).abs() >= 1e-3
        eye = torch.eye(4, dtype=torch.float64, device=M.device)
        x = torch.linalg.solve(torch.where(use[:, None, None], M, eye), rhs)
        full = x[:, 0] - (self.ghost[bo] * x[:, 1:]).sum(1)
        use &= (full > 0.0) & (full < 1e30)
        self.rho[bo] = torch.where(none, torch.full_like(full, rho0),
                                   torch.where(use, full, shepard))

    def move_walls(self, t0, t1, pos, vel):
        """Imposed motion from t0 to t1 of the moving groups."""
        for k, mo in enumerate(self.motions):
            ph, om = mo.get("phase", 0.0), mo["omega"]
            axis = torch.tensor(mo["axis"], dtype=torch.float64, device=pos.device)
            sel = self.group == k
            d = mo["amp"] * (math.sin(om * t1 + ph) - math.sin(om * t0 + ph))
            pos[sel] += d * axis
            vel[sel] = mo["amp"] * om * math.cos(om * t1 + ph) * axis

    def time_step(self, acc, mu):
        f = float(acc[self.fluid].norm(dim=1).max())
        return self.p["cfl"] * min(math.sqrt(self.h / f) if f > 0 else math.inf,
                                   self.h / (self.p["cs0"] + mu))

    def clamp(self, rho):
        if not self.p["clamp_boundary_rho"]:
            return rho
        return torch.where(self.fluid, rho, rho.clamp(min=self.p["rho0"]))

    def step(self):
        fl = self.fluid[:, None]
        acc, drho, mu = self.evaluate()
        dt = self.time_step(acc, mu)
        p0, v0, r0 = self.pos, self.vel, self.rho
        if self.p["integrator"] == 1:
            first = self.step_no % self.p["verlet_steps"] == 0
            k = dt if first else 2.0 * dt
            vb, rb = (v0, r0) if first else (self.vp, self.rp)
            self.pos = p0 + fl * (dt * v0 + 0.5 * dt * dt * acc)
            self.vel = torch.where(fl, vb + k * acc, v0)
            self.rho = self.clamp(rb + k * drho)
            self.move_walls(self.t, self.t + dt, self.pos, self.vel)
            self.vp, self.rp = v0, r0
        else:
            self.pos = p0 + fl * (0.5 * dt * v0)
            self.vel = torch.where(fl, v0 + 0.5 * dt * acc, v0)
            self.rho = self.clamp(r0 + 0.5 * dt * drho)
            self.move_walls(self.t, self.t + 0.5 * dt, self.pos, self.vel)
            acc, drho, _ = self.evaluate()
            eps = -(drho / self.rho) * dt
            self.rho = self.clamp(r0 * (2.0 - eps) / (2.0 + eps))
            self.vel = torch.where(fl, v0 + dt * acc, v0)
            self.pos = p0 + fl * (0.5 * dt * (self.vel + v0))
            self.move_walls(self.t, self.t + dt, self.pos, self.vel)
        self.t += dt
        self.step_no += 1
        lo = torch.tensor(self.p["domain_min"], dtype=torch.float64, device=self.pos.device)
        hi = torch.tensor(self.p["domain_max"], dtype=torch.float64, device=self.pos.device)
        if not bool(((self.pos >= lo) & (self.pos < hi)).all()):
            raise _Slow  # a particle left the domain: frozen there, not followed here

    def frame(self):
        return dict(pos=self.pos, vel=self.vel, rho=self.rho, press=self.tait(self.rho),
                    t=torch.tensor(self.t, dtype=torch.float64))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    out = []
    try:
        for c in _inputs(case, seed):
            x = _Exact(c, dev)
            if case["kind"] == "serve":
                while x.t < case["t_end"]:
                    x.step()
            else:
                for _ in range(case["steps"]):
                    x.step()
            out.append(x.frame())
            del x
    except _Slow:
        return None
    return out
