"""Performance cases: the work a user of this framework has it do.

Each case is one piece of a user's loop through the public binding
(`paper_2106_08950_gb300.dilbm`): advance a lattice (or a batch, or a served
set of jobs) by some steps and take the results that such a loop takes: the
forces, the particles' state and the macroscopic fields.  Sizes come from the
repository's workloads, tests and benchmark.

Kinds:

* ``channel``    -- fixed discs between a velocity inlet and a density outlet;
* ``box``        -- discs settling in a closed box (four walls);
* ``suspension`` -- free discs in a fully periodic box;
* ``frame``      -- one neutrally buoyant disc in a pressure-driven channel,
                    the frame following the disc;
* ``batch``      -- many uneven lattices advanced together;
* ``serve``      -- jobs of mixed sizes through the continuous-batching server;
* ``coupled``    -- a host-coupled particle loop: upload, one step, read back;
* ``checkpoint`` -- populations to the host and back.

``exact`` is the method in 64 bits with plain torch.
"""
import ctypes as C
import math
import random

import numpy as np
import torch

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

STORED_BYTES = {"fp32": 4, "fp16": 2, "bf16": 2, "auto": 4}
FLOPS_PER_NODE = 200            # moments, equilibrium and relaxation of nine populations


def _case(name, kind, **kw):
    c = {"kind": kind, "storage": "fp32", "method": "di", "steps": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest lattice: a drag sample of the 200 x 100 cylinder channel every 100 steps
        _case("cylinder 200x100", "channel", nx=200, ny=100, discs=1, steps=100),
        # a lattice that fits the L2: the settling disc's trajectory, sampled every 100 steps
        _case("settling 400x2000", "box", nx=400, ny=2000, discs=1, steps=100),
        # a served job's size run alone, ragged (nx = 1 mod 128) and in FP16
        _case("channel 1793x179 fp16", "channel", nx=1793, ny=179, discs=12, storage="fp16", steps=100),
        # the 512 x 512 copy of the suspension, as the parity and down-scaled runs use it
        _case("suspension 512 fp32", "suspension", nx=512, ny=512, discs=32, steps=100),
        # the headline workload in its two storages
        _case("suspension 4096 fp32", "suspension", nx=4096, ny=4096, discs=2048, steps=20),
        _case("suspension 4096 fp16", "suspension", nx=4096, ny=4096, discs=2048, storage="fp16", steps=20),
        # the comparison method on the headline workload
        _case("ps suspension 4096", "suspension", nx=4096, ny=4096, discs=2048, method="ps", steps=20),
        # the moving frame (Sec. 3.5): a sample of the migrating disc every 100 steps
        _case("moving frame 501x101", "frame", nx=501, ny=101, discs=1, steps=100),
        # 64 uneven lattices in one launch per step
        _case("batch of 64", "batch", lattices=64, layout=4, steps=20),
        # a served set of jobs that join and leave, storage chosen by the server
        _case("served 16 jobs", "serve", jobs=16, layout=5, storage="auto", max_jobs=8, min_steps=200, max_steps=1000),
        # the smallest call: one step between two host reads of a coupled particle code
        _case("coupled step 512", "coupled", nx=512, ny=512, discs=32),
        # checkpoint and resume
        _case("checkpoint 1024", "checkpoint", nx=1024, ny=1024, discs=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps_for(rng, nodes):
    """Steps between two samples: up to 100, fewer on large lattices."""
    most = max(5, min(100, int(2e8 // nodes)))
    return _log_int(rng, max(5, most // 4), most)


def draw(rng):
    kind = rng.choice(["channel", "box", "suspension", "suspension", "suspension", "frame", "batch", "serve",
                       "coupled", "checkpoint"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind in ("channel", "box"):
        nx, ny = _log_int(rng, 128, 2048), _log_int(rng, 128, 2048)
        discs = min(_log_int(rng, 1, 32), max(1, nx * ny // 6000))
        return _case(None, kind, nx=nx, ny=ny, discs=discs, storage=storage, steps=_steps_for(rng, nx * ny))
    if kind == "suspension":
        nx, ny = _log_int(rng, 256, 4096), _log_int(rng, 256, 4096)
        # the benchmark's disc density, half of it, or a plain periodic flow
        discs = int(nx * ny / 8192 * rng.choice([1.0, 1.0, 0.5, 0.0]))
        method = "ps" if discs and rng.random() < 0.25 else "di"
        return _case(None, kind, nx=nx, ny=ny, discs=discs, storage=storage, method=method,
                     steps=_steps_for(rng, nx * ny))
    if kind == "frame":
        return _case(None, kind, nx=rng.randrange(301, 1002, 4), ny=rng.randrange(101, 202), discs=1,
                     storage=storage, steps=rng.randrange(30, 101))
    if kind == "batch":
        return _case(None, kind, lattices=rng.randrange(8, 49), layout=rng.randrange(1 << 20), storage=storage,
                     steps=rng.randrange(7, 21))
    if kind == "serve":
        return _case(None, kind, jobs=rng.randrange(4, 13), layout=rng.randrange(1 << 20),
                     storage=rng.choice(["auto", "fp32", "fp16"]), max_jobs=rng.randrange(3, 9), min_steps=100,
                     max_steps=rng.randrange(200, 601))
    if kind == "coupled":
        nx, ny = _log_int(rng, 256, 4096), _log_int(rng, 256, 4096)
        return _case(None, kind, nx=nx, ny=ny, discs=max(1, nx * ny // 8192), storage=storage)
    nx, ny = _log_int(rng, 128, 1024), _log_int(rng, 128, 1024)
    return _case(None, "checkpoint", nx=nx, ny=ny, discs=max(1, nx * ny // 8192), storage=storage)


# ------------------------------------------------------------------ problems
def _discs(rng, nx, ny, count, rmin, rmax, periodic, margin=0.0):
    """Seeded discs without overlap."""
    return W._place_discs(rng, nx, ny, count, rmin, rmax, 4.0, periodic=periodic, margin=margin)


def _problem(case, seed):
    rng = np.random.default_rng(seed)
    kind, nx, ny, count = case["kind"], case["nx"], case["ny"], case["discs"]
    if kind == "channel":
        p = W.cylinder_drag(nx=nx, ny=ny, u=0.05 * rng.uniform(0.8, 1.0))
        if count == 1:
            p.particles = [W.Particle(nx / 4 + rng.uniform(-1, 1), ny / 2 + rng.uniform(-1, 1), 10.0, fixed=True)]
        else:
            p.particles = [W.Particle(x, y, r, fixed=True)
                           for x, y, r in _discs(rng, nx, ny, count, 5.0, 12.0, False, 6.0)]
        return p
    if kind == "box":
        p = W.sedimentation(nx=nx, ny=ny)
        if count == 1:
            p.particles = [W.Particle((nx - 1) / 2 + rng.uniform(-1, 1), (ny - 1) / 2 + rng.uniform(-1, 1), 12.0,
                                      uy=-0.01, rho_s=1.5)]
        else:
            p.particles = [W.Particle(x, y, r, uy=-0.01, rho_s=1.5)
                           for x, y, r in _discs(rng, nx, ny, count, 5.0, 15.0, False, 6.0)]
        return p
    if kind == "frame":
        # Sec. 3.5: a pressure-driven channel between resting walls
        rho_in = 1.0 + 3 * 0.00267 * (nx - 1) / 500.0
        return W.Problem(nx=nx, ny=ny, tau=0.9, eps=2.0, west=W.Side(W.PRESSURE, rho=rho_in),
                         east=W.Side(W.PRESSURE, rho=1.0), south=W.wall(), north=W.wall(), force_model=W.FORCE_MOMENTUM,
                         wan_turek=W.wan_turek_defaults(12.5, 1.5, 1.0, 1e-5),
                         particles=[W.Particle((nx - 1) / 2, ny / 4 + rng.uniform(0, 2), 12.5, ux=0.02, uy=0.001,
                                               rho_s=1.0)])
    # the periodic suspension, its discs in motion
    p = W.Problem(nx=nx, ny=ny, tau=0.8, eps=2.0, gravity=(0.0, -1e-6),
                  u0=(rng.uniform(-5e-3, 5e-3), rng.uniform(-5e-3, 5e-3)),
                  wan_turek=W.wan_turek_defaults(9.0, 1.2, 1.0, 1e-6),
                  method=W.METHOD_PS if case["method"] == "ps" else W.METHOD_DI)
    p.particles = [W.Particle(x, y, r, ux=rng.uniform(-0.01, 0.01), uy=rng.uniform(-0.01, 0.01),
                              omega=rng.uniform(-1e-3, 1e-3), rho_s=1.2)
                   for x, y, r in _discs(rng, nx, ny, count, 6.0, 12.0, True)]
    return p


def _layout(case):
    """The lattices of a batch or the jobs of a served set: (nx, ny, discs, steps) of each, by the case alone."""
    rng = random.Random(case["layout"])
    if case["kind"] == "batch":
        return [(_log_int(rng, 128, 1024), _log_int(rng, 128, 2048), rng.randint(1, 32), case["steps"])
                for _ in range(case["lattices"])]
    return [(_log_int(rng, 128, 2048), _log_int(rng, 128, 2048), rng.randint(1, 64),
             _log_int(rng, case["min_steps"], case["max_steps"])) for _ in range(case["jobs"])]


def _problems(case, seed):
    out = []
    for k, (nx, ny, discs, _) in enumerate(_layout(case)):
        rng = np.random.default_rng([seed, k])
        out.append(W.random_job(rng, nx_range=(nx, nx), ny_range=(ny, ny), p_range=(discs, discs)))
    return out


# ------------------------------------------------------------------ the cases' passes
class _State:
    pass


def _field_buffers(nx, ny):
    return [torch.empty(ny, nx, dtype=torch.float32, device="cuda") for _ in range(4)]


def prepare(case, seed):
    s = _State()
    s.case = dict(case)
    kind = case["kind"]
    s.stream = torch.cuda.Stream()
    handle = int(s.stream.cuda_stream)
    if kind == "serve":
        s.problems = _problems(case, seed)
        s.steps = [j[3] for j in _layout(case)]
        s.server = D.Server(case["storage"], max_jobs=case["max_jobs"])
        return s
    if kind == "batch":
        problems = _problems(case, seed)
        s.sims = [D.Simulation(p, storage=case["storage"], stream=handle) for p in problems]
        s.batch = D.Batch(s.sims)
        s.flat = torch.empty(4, sum(p.nodes for p in problems), dtype=torch.float32, device="cuda")
        s.views, at = [], 0
        for p in problems:
            s.views.append([s.flat[q, at:at + p.nodes] for q in range(4)])
            at += p.nodes
        return s
    prob = _problem(case, seed)
    s.sim = D.Simulation(prob, storage=case["storage"], stream=handle)
    if kind == "frame":
        s.sim.set_moving_frame(0)
    if kind == "coupled":
        # the coupled code's particles live in pinned memory and are read and written in place
        n = len(prob.particles)
        s.pinned = torch.empty(n * C.sizeof(D.Particle), dtype=torch.uint8).pin_memory()
        s.parts = (D.Particle * n).from_address(s.pinned.data_ptr())
        C.memmove(s.parts, D.make_particles(prob.particles), n * C.sizeof(D.Particle))
        s.force = np.zeros((n, 3))
        s.table = np.frombuffer(s.parts, dtype=np.dtype([(k, "f8") for k in ("x", "y", "r", "ux", "uy", "omega",
                                                                            "theta", "rho_s")] + [("fixed", "i4"), ("pad", "i4")]))
        return s
    if kind == "checkpoint":
        s.sim.step(10)
        s.sim.sync()
        return s
    s.fields = _field_buffers(prob.nx, prob.ny)
    return s


def _table(t):
    return np.stack([t[k] for k in ("x", "y", "r", "ux", "uy", "omega", "theta", "rho_s")], axis=1)


def run(s):
    kind = s.case["kind"]
    if kind == "serve":
        ids = [s.server.submit(p, n) for p, n in zip(s.problems, s.steps)]
        while True:
            st = s.server.progress()
            if st.running == 0 and st.queued == 0:
                break
        got = [s.server.result(j) for j in ids]
        return {"force": np.concatenate([g[0] for g in got]), "state": np.concatenate([g[1] for g in got])}
    if kind == "batch":
        s.batch.step(s.case["steps"])
        for sim, v in zip(s.sims, s.views):
            sim.fields_device(*v)
        got = [sim.forces() for sim in s.sims]
        return {"force": np.concatenate([g[0] for g in got]), "repulsion": np.concatenate([g[1] for g in got]),
                "state": np.concatenate([g[2] for g in got]), "fields": s.flat}
    if kind == "coupled":
        s.sim.set_particles_raw(s.parts)
        s.sim.step(1)
        D.check(s.sim.L.dilbm_forces(s.sim.h, s.force.ctypes.data, None, C.cast(s.parts, C.c_void_p)))
        return {"force": s.force, "state": _table(s.table)}
    if kind == "checkpoint":
        f = s.sim.populations()
        s.sim.set_populations(f)
        return {"populations": f}
    s.sim.step(s.case["steps"])
    s.sim.fields_device(*s.fields)
    out = {"fields": s.fields}
    if s.case["discs"]:
        out["force"], out["repulsion"], out["state"] = s.sim.forces()
    else:
        s.sim.sync()
    if kind == "frame":
        out["offset"] = s.sim.frame_offset()
    return out


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        updates = sum(nx * ny * n for nx, ny, _, n in _layout(case))
        nodes = sum(nx * ny for nx, ny, _, _ in _layout(case)) if kind == "batch" else 0
    else:
        nodes = case["nx"] * case["ny"]
        updates = nodes * case["steps"]
    e = STORED_BYTES[case["storage"]]
    if kind == "checkpoint":        # nine populations: stored values and their FP64 copies, there and back
        return {"bytes": 2.0 * 9 * nodes * (e + 8), "flops": 2.0 * 9 * nodes}
    if kind == "coupled":
        return {"bytes": 18.0 * e * nodes, "flops": float(FLOPS_PER_NODE * nodes)}
    # every step reads and writes nine populations; the fields read them once more and write four values
    return {"bytes": 18.0 * e * updates + (9.0 * e + 16.0) * nodes, "flops": float(FLOPS_PER_NODE * (updates + nodes))}


# ------------------------------------------------------------------ the method in 64 bits
_CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_WT = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


def _equilibrium(rho, ux, uy):
    uu = 1.5 * (ux * ux + uy * uy)
    out = []
    for cx, cy, w in zip(_CX, _CY, _WT):
        cu = 3.0 * (cx * ux + cy * uy)
        out.append(w * rho * (1.0 + cu + 0.5 * cu * cu - uu))
    return torch.stack(out)


def _quadrant(x, y, r):
    """Area of the disc of radius r about the origin with X <= x and Y <= y."""
    x, y = torch.clamp(x, min=-r, max=r), torch.clamp(y, min=-r, max=r)

    def beyond(t):                               # the part farther out than t >= 0 along one axis
        return r * r * torch.acos(t / r) - t * torch.sqrt(torch.clamp(r * r - t * t, min=0.0))
    inside = x * x + y * y < r * r
    cut = (r * r * (math.pi / 2 + torch.asin(x / r) + torch.asin(y / r))
           + x * torch.sqrt(torch.clamp(r * r - x * x, min=0.0))
           + y * torch.sqrt(torch.clamp(r * r - y * y, min=0.0))) / 2 + x * y
    ax, ay = beyond(torch.abs(x)), beyond(torch.abs(y))
    out = torch.where((x >= 0) & (y >= 0), math.pi * r * r - ax - ay,
                      torch.where((x < 0) & (y < 0), torch.zeros_like(x), torch.where(x < 0, ax, ay)))
    return torch.where(inside, cut, out)


class _Exact:
    """One lattice in FP64: the procedure of Sec. 2.3, with the smooth fraction kept up to four widths."""

    def __init__(self, p, frame=False):
        self.p = p
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.ps = p.method == W.METHOD_PS
        self.px, self.py = p.west.kind == W.PERIODIC, p.south.kind == W.PERIODIC
        self.w = 1.0 / p.tau
        self.kf = 1.0 if self.ps else 1.0 - 0.5 / p.tau
        self.kforce = self.kf if p.force_model == W.FORCE_EQ18 else 1.0
        self.cut = 0.70711 if self.ps else 4.0 * p.eps
        one = torch.ones(p.ny, p.nx, dtype=torch.float64, device=self.dev)
        self.f = _equilibrium(p.rho_init * one, p.u0[0] * one, p.u0[1] * one)
        self.n = len(p.particles)
        g = [[q.x, q.y, q.r, q.ux, q.uy, q.omega, q.theta, q.rho_s, float(q.fixed)] for q in p.particles]
        t = torch.tensor(g, dtype=torch.float64, device=self.dev).reshape(self.n, 9)
        self.x, self.y, self.r, self.ux, self.uy, self.om, self.th, self.rs, self.fx = (t[:, k].clone() for k in range(9))
        self.F = torch.zeros(self.n, 3, dtype=torch.float64, device=self.dev)
        self.Fc = torch.zeros(self.n, 2, dtype=torch.float64, device=self.dev)
        self.x_ref = self.x[0].clone() if frame else None
        self.offset = 0

    def pulled(self):
        f = torch.stack([torch.roll(self.f[i], (_CY[i], _CX[i]), (0, 1)) for i in range(9)])
        p = self.p
        if not self.px:
            ys = slice(None) if self.py else slice(1, p.ny - 1)
            f[:, ys, 0] = self.edge(f[:, ys, 1], p.west)
            f[:, ys, -1] = self.edge(f[:, ys, -2], p.east)
        if not self.py:
            xs = torch.arange(p.nx, device=self.dev)
            if not self.px:
                xs = torch.clamp(xs, 1, p.nx - 2)
            f[:, 0] = self.edge(f[:, 1][:, xs], p.south)
            f[:, -1] = self.edge(f[:, -2][:, xs], p.north)
        return f

    @staticmethod
    def moments(f):
        rho = f.sum(0)
        return rho, (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho, (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho

    def edge(self, fn, side):
        rho, ux, uy = self.moments(fn)
        if side.kind == W.VELOCITY:
            b = _equilibrium(rho, torch.full_like(ux, side.ux), torch.full_like(uy, side.uy))
        else:
            b = _equilibrium(torch.full_like(rho, side.rho), ux, uy)
        return b + fn - _equilibrium(rho, ux, uy)

    def solid(self):
        """Covered nodes: (flat node, particle, fraction, offset from the centre) of each node's owner."""
        nx, ny = self.p.nx, self.p.ny
        K = int(math.ceil(float(self.r.max()) + self.cut)) + 1
        o = torch.arange(-K, K + 1, device=self.dev)
        ix = torch.floor(self.x).long()[:, None, None] + o[None, None, :]
        iy = torch.floor(self.y).long()[:, None, None] + o[None, :, None]
        dx, dy = ix - self.x[:, None, None], iy - self.y[:, None, None]
        r = self.r[:, None, None]
        dist = torch.sqrt(dx * dx + dy * dy)
        l = r - dist
        ok = l >= -self.cut
        if not self.px:
            ok = ok & (ix >= 0) & (ix < nx)
        if not self.py:
            ok = ok & (iy >= 0) & (iy < ny)
        pid = torch.arange(self.n, device=self.dev)[:, None, None].expand_as(ok)[ok]
        node = ((iy % ny) * nx + (ix % nx))[ok]
        dx, dy, r, l = (v.expand_as(ok)[ok] for v in (dx, dy, r, l))
        if self.ps:
            phi = (_quadrant(dx + 0.5, dy + 0.5, r) - _quadrant(dx - 0.5, dy + 0.5, r)
                   - _quadrant(dx + 0.5, dy - 0.5, r) + _quadrant(dx - 0.5, dy - 0.5, r))
            phi = torch.where(l >= self.cut, torch.ones_like(phi), torch.clamp(phi, 0.0, 1.0))
        else:
            phi = 1.0 / (1.0 + torch.exp(-4.0 * l / self.p.eps))
        top = torch.zeros(nx * ny, dtype=torch.float64, device=self.dev).scatter_reduce_(0, node, phi, "amax")
        lead = (phi == top[node]) & (phi > 0)
        node, pid, phi, dx, dy = node[lead], pid[lead], phi[lead], dx[lead], dy[lead]
        who = torch.full((nx * ny,), self.n, device=self.dev).scatter_reduce_(0, node, pid, "amin")
        own = pid == who[node]
        return node[own], pid[own], phi[own], dx[own], dy[own]

    def coupled(self, rho, ux, uy):
        """The corrected velocity in place; what the force term needs at the covered nodes."""
        node, pid, phi, rx, ry = self.solid()
        r, ax, ay = (v.reshape(-1)[node] for v in (rho, ux, uy))
        sx, sy = self.ux[pid] - self.om[pid] * ry, self.uy[pid] + self.om[pid] * rx
        if not self.ps:
            ux.reshape(-1)[node] = ax + 0.5 * phi * (sx - ax)
            uy.reshape(-1)[node] = ay + 0.5 * phi * (sy - ay)
        return node, pid, phi, rx, ry, r, ax, ay, sx, sy

    def step(self):
        p = self.p
        f = self.pulled()
        rho, ux, uy = self.moments(f)
        c = self.coupled(rho, ux, uy) if self.n else None
        eq = _equilibrium(rho, ux, uy)
        f += self.w * (eq - f)
        del eq
        if self.n:
            node, pid, phi, rx, ry, r, ax, ay, sx, sy = c
            k = self.kf * r * phi
            mxx, myy, mxy = k * (sx * sx - ax * ax), k * (sy * sy - ay * ay), k * (sx * sy - ax * ay)
            flat = f.reshape(9, -1)
            for i in range(9):
                cx, cy = _CX[i], _CY[i]
                flat[i][node] += _WT[i] * (3.0 * k * (cx * (sx - ax) + cy * (sy - ay))
                                           + 4.5 * (cx * cx * mxx + cy * cy * myy + 2 * cx * cy * mxy)
                                           - 1.5 * (mxx + myy))
            gx, gy = -self.kforce * phi * r * (sx - ax), -self.kforce * phi * r * (sy - ay)
            self.F = torch.zeros_like(self.F).index_add_(0, pid, torch.stack([gx, gy, rx * gy - ry * gx], 1))
            self.bodies()
        self.f = f
        if self.x_ref is not None:
            self.follow()

    def bodies(self):
        p = self.p
        e_p, e_p2, e_w, e_w2, xi = p.wan_turek

        def spring(d, rr, near, touch):
            s = torch.where(d <= rr + xi, (rr + xi - d) ** 2 / near, torch.zeros_like(d))
            return torch.where(d <= rr, (rr - d) / touch, s)
        fc = torch.zeros_like(self.Fc)
        if self.n > 1:
            dx, dy = self.x[:, None] - self.x[None, :], self.y[:, None] - self.y[None, :]
            if self.px:
                dx = dx - p.nx * torch.round(dx / p.nx)
            if self.py:
                dy = dy - p.ny * torch.round(dy / p.ny)
            d = torch.sqrt(dx * dx + dy * dy)
            s = spring(d, self.r[:, None] + self.r[None, :], e_p, e_p2)
            s.fill_diagonal_(0.0)
            fc[:, 0], fc[:, 1] = (s * dx).sum(1), (s * dy).sum(1)
        if not self.px:
            for wall in (0.0, p.nx - 1.0):
                dx = 2.0 * (self.x - wall)
                fc[:, 0] += spring(torch.abs(dx), 2.0 * self.r, e_w, e_w2) * dx
        if not self.py:
            for wall in (0.0, p.ny - 1.0):
                dy = 2.0 * (self.y - wall)
                fc[:, 1] += spring(torch.abs(dy), 2.0 * self.r, e_w, e_w2) * dy
        self.Fc = fc
        area = math.pi * self.r * self.r
        m = self.rs * area
        free = self.fx == 0
        weight = (self.rs - p.rho_f) * area
        self.x_old = self.x
        self.ux = torch.where(free, self.ux + (self.F[:, 0] + fc[:, 0] + weight * p.gravity[0]) / m, self.ux)
        self.uy = torch.where(free, self.uy + (self.F[:, 1] + fc[:, 1] + weight * p.gravity[1]) / m, self.uy)
        self.om = torch.where(free, self.om + self.F[:, 2] / (0.5 * m * self.r * self.r), self.om)
        self.th = torch.where(free, self.th + self.om, self.th)
        self.x = torch.where(free, self.x + self.ux, self.x)
        self.y = torch.where(free, self.y + self.uy, self.y)
        if self.px:
            self.x = self.x % p.nx
        if self.py:
            self.y = self.y % p.ny

    def follow(self):
        d = float(self.x_old[0] - self.x_ref)
        s = 1 if d >= 1.0 else -1 if d <= -1.0 else 0
        if s:
            cols = torch.clamp(torch.arange(self.p.nx, device=self.dev) + s, 0, self.p.nx - 1)
            self.f = self.f[:, :, cols]
            self.x = self.x - s
            self.offset += s

    def fields(self):
        rho, ux, uy = self.moments(self.pulled())
        phi = torch.zeros(rho.numel(), dtype=torch.float64, device=self.dev)
        if self.n:
            c = self.coupled(rho, ux, uy)
            phi[c[0]] = c[2]
        return [rho, ux, uy, phi.reshape(rho.shape)]

    def state(self):
        return torch.stack([self.x, self.y, self.r, self.ux, self.uy, self.om, self.th, self.rs], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        steps = [j[3] for j in _layout(case)]
        if sum(steps) > 12000:
            return None
        sims = [_Exact(p) for p in _problems(case, seed)]
        for e, n in zip(sims, steps):
            for _ in range(n):
                e.step()
        out = {"force": torch.cat([e.F for e in sims]), "state": torch.cat([e.state() for e in sims])}
        if kind == "batch":
            out["repulsion"] = torch.cat([e.Fc for e in sims])
            fields = [e.fields() for e in sims]
            out["fields"] = torch.stack([torch.cat([f[q].reshape(-1) for f in fields]) for q in range(4)])
        return out
    e = _Exact(_problem(case, seed), frame=kind == "frame")
    for _ in range(10 if kind == "checkpoint" else case["steps"]):
        e.step()
    if kind == "checkpoint":
        return {"populations": e.f}
    if kind == "coupled":
        return {"force": e.F, "state": e.state()}
    out = {"fields": e.fields()}
    if case["discs"]:
        out["force"], out["repulsion"], out["state"] = e.F, e.Fc, e.state()
    if kind == "frame":
        out["offset"] = None
    return out
