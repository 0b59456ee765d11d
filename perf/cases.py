"""Performance cases: the work a user of this library has it do.

A pass advances one or many simulations by some steps through the public
binding and reads back what a run looks at: the particles' motion and, at a
snapshot, velocity and temperature.  The kinds of use:

track    a small case advanced one step at a time, the particles read after
         every step (a trajectory recorder or a control loop)
cavity   a square cavity of cold disks, advanced to the next snapshot
channel  one disk settling in a closed channel
held     the same with a disk held at its temperature and heated walls
ellipse  an elliptical particle in a channel with an open lower end
batch    many channels of different sizes stepped together
serve    a set of cavity requests through the served mode

Sizes, densities and parameters are those of paper_2410_23802_gb300.workloads,
the tests and bench.py.  `exact` restates the time step in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2410_23802_gb300 import vlb as V
from paper_2410_23802_gb300 import workloads as W

STORAGE = {"fp64": V.VLB_FP64, "fp32": V.VLB_FP32, "fp16": V.VLB_FP16_STORE, "bf16": V.VLB_BF16_STORE}
STORED_BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
MOTION = ("x", "y", "theta", "ux", "uy", "omega")
# 16-bit runs keep half-precision snapshots; velocities and angles (about 1e-4) are
# scaled by 2^12 as the FP16 storage does, which keeps them clear of subnormals
HALF_SCALE = 4096.0
# no drawn case advances more cells than this in a pass (the largest listed one: 2048^2 x 1000)
MOST_CELL_STEPS = 2048 * 2048 * 1000


def listed():
    return [
        # the smallest call: four disks in a 64^2 box, one step and one particle read at a time
        {"name": "track_64", "kind": "track", "side": 64, "disks": 4, "storage": "fp32", "steps": 20},
        # one settling disk (the oracle's reference channel), between two snapshots
        {"name": "channel_100x400", "kind": "channel", "width": 100, "storage": "fp32", "steps": 500},
        # the same channel as a double-precision validation run
        {"name": "channel_100x400_fp64", "kind": "channel", "width": 100, "storage": "fp64", "steps": 200},
        # the paper's held-temperature sedimentation (width 4 D, 80 D long, Dirichlet walls)
        {"name": "held_80x1600", "kind": "held", "length": 80, "grashof": 1000.0, "hold": 1, "storage": "fp32",
         "steps": 500},
        # the paper's elliptical particle in a 104-wide channel with an open end
        {"name": "ellipse_104x3120", "kind": "ellipse", "length": 30, "storage": "fp32", "steps": 300},
        # a medium cavity: the size of the README's example
        {"name": "cavity_512", "kind": "cavity", "side": 512, "disks": 128, "spread": False, "storage": "fp32",
         "steps": 500},
        # an odd side, so that rows and tiles are ragged, and conductivities over two decades
        {"name": "cavity_1001_spread", "kind": "cavity", "side": 1001, "disks": 500, "spread": True,
         "storage": "fp32", "steps": 400},
        # the throughput configuration of bench.py
        {"name": "cavity_2048", "kind": "cavity", "side": 2048, "disks": 2048, "spread": False, "storage": "fp32",
         "steps": 1000},
        # the same with half-precision population storage
        {"name": "cavity_2048_fp16", "kind": "cavity", "side": 2048, "disks": 2048, "spread": False,
         "storage": "fp16", "steps": 500},
        # the largest lattice of the tests, 16-bit storage, per-particle conductivity
        {"name": "cavity_4096_bf16", "kind": "cavity", "side": 4096, "disks": 8192, "spread": True,
         "storage": "bf16", "steps": 200},
        # a parameter study: many small channels resident together
        {"name": "batch_48", "kind": "batch", "count": 48, "widest": 256, "layout": 20241104, "storage": "fp32",
         "steps": 200},
        # requests of mixed sizes and storage through the server
        {"name": "serve_10", "kind": "serve", "count": 10, "largest": 1024, "layout": 20241105, "steps": 300},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["track", "channel", "held", "ellipse", "cavity", "cavity", "cavity", "batch", "serve"])
    if kind == "track":
        side = _log_int(rng, 48, 160)
        return {"kind": kind, "side": side, "disks": rng.randint(1, max(1, side * side // 1200)), "storage": "fp32",
                "steps": rng.randint(10, 40)}
    if kind == "channel":
        storage = rng.choice(["fp32", "fp32", "fp16", "fp64"])
        return {"kind": kind, "width": _log_int(rng, 64, 256), "storage": storage,
                "steps": rng.randint(60, 150) if storage == "fp64" else rng.randint(200, 600)}
    if kind == "held":
        return {"kind": kind, "length": rng.randint(30, 150), "grashof": float(rng.choice([564, 1000, 2000, 2500])),
                "hold": rng.choice([1, 2]), "storage": "fp32", "steps": rng.randint(200, 600)}
    if kind == "ellipse":
        return {"kind": kind, "length": rng.randint(6, 40), "storage": "fp32", "steps": rng.randint(100, 500)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(8, 48), "widest": rng.randint(96, 256),
                "layout": rng.getrandbits(30), "storage": "fp32", "steps": rng.randint(60, 200)}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(4, 10), "largest": _log_int(rng, 128, 1024),
                "layout": rng.getrandbits(30), "steps": rng.randint(100, 300)}
    side = _log_int(rng, 96, 4096)
    steps = min(int(MOST_CELL_STEPS * rng.uniform(0.3, 1.0) / side ** 2), rng.randint(200, 500))
    return {"kind": kind, "side": side, "disks": max(1, int(side * side * rng.uniform(0.1, 1.0) / 2048)),
            "spread": rng.random() < 0.5, "storage": rng.choice(["fp32", "fp32", "fp16", "bf16"]),
            "steps": max(20, steps)}


# ---- inputs -----------------------------------------------------------------

def _simulations(case, seed):
    """The case's simulations as workloads.Case objects: sizes from the case,
    placements and temperatures from the seed.  Particles given to a handle
    are released with a small velocity (c.uv) and spin (c.omega); a served
    request starts at rest."""
    rng = W.SplitMix64(0x5EED0000 + seed)
    kind, storage = case["kind"], case.get("storage", "fp32")
    if kind in ("track", "cavity"):
        cases = [W.cavity(side=case["side"], n=case["disks"], diameter=16.0 if kind == "cavity" else 8.0,
                          seed=rng.next_u64(), precision=storage, k_log_uniform=case.get("spread", False))]
    elif kind == "channel":
        w = case["width"]
        c = W.channel(storage)
        c.params.update(nx=w, ny=4 * w, beta=W.gr_beta(100.0, 0.1, 1e-5, 1.0, 0.2 * w))
        c.x, c.y, c.radius = [w * rng.uniform(0.4, 0.6)], [w * rng.uniform(2.9, 3.1)], [0.1 * w]
        c.T0 = [rng.uniform(0.0, 0.2)]
        cases = [c]
    elif kind == "held":
        c = W.fixed_temperature_sedimentation(case["grashof"], float(case["length"]), storage, hold=case["hold"])
        c.x, c.y = [c.x[0] + rng.uniform(-2.0, 2.0)], [c.y[0] + rng.uniform(-2.0, 2.0)]
        cases = [c]
    elif kind == "ellipse":
        cases = [W.ellipse_sedimentation(float(case["length"]), rng.uniform(0.2, 1.3), rng.uniform(-6.0, 6.0), storage)]
    elif kind == "batch":
        cases = W.channels(n=case["count"], seed=case["layout"], w_max=case["widest"], precision=storage)
        for c in cases:
            c.x = [c.x[0] + c.params["nx"] * rng.uniform(-0.1, 0.1)]
    else:
        cases = [W.cavity(side=c.params["nx"], n=len(c.x), diameter=2.0 * c.radius[0], seed=rng.next_u64(),
                          precision=c.params["precision"])
                 for _, c, _ in W.served_cases(n=case["count"], seed=case["layout"], max_solid=0.2,
                                               side_log2=(6.0, math.log2(case["largest"])))]
    for c in cases:
        c.uv = [0.0 if kind == "serve" else rng.uniform(-2e-3, 2e-3) for _ in range(2 * len(c.x))]
        c.omega = [0.0 if kind == "serve" else rng.uniform(-1e-3, 1e-3) for _ in c.x]
    return cases


def _params(c):
    prm = {k: v for k, v in c.params.items() if k != "precision"}
    return V.vlb_params_default(precision=STORAGE[c.params["precision"]], max_particles=len(c.x), **prm)


class _Run:
    """Handles of a run, closed with the state that holds them."""

    def __init__(self):
        self.lattices, self.server = [], None

    def __del__(self):
        for lat in self.lattices:
            lat.close()
        if self.server is not None:
            self.server.close()


def prepare(case, seed):
    state = {"case": case, "run": _Run(), "sims": _simulations(case, seed)}
    if case["kind"] == "serve":
        state["requests"] = [(_params(c), np.column_stack([c.x, c.y]), c.radius, c.T0) for c in state["sims"]]
        state["run"].server = V.Server(hbm_budget=2 << 30, steps_per_round=100)
        return state
    for c in state["sims"]:
        lat = V.Lattice(_params(c))
        state["run"].lattices.append(lat)
        xy = np.column_stack([c.x, c.y])
        if c.semi_minor is not None:
            lat.add_ellipses(xy, c.radius, c.semi_minor, c.theta0, c.T0, uv=c.uv, omega=c.omega)
        else:
            lat.add_particles(xy, c.radius, c.T0, k_ratio=c.k_ratio, uv=c.uv, omega=c.omega)
        if c.fixed_T is not None:
            V.vlb_set_fixed_temperature(lat.h, c.fixed_T)
        lat.step(0)  # the initial state
        V.vlb_synchronize(lat.h)
    return state


# ---- one pass ---------------------------------------------------------------

def _keep(a, storage, velocity=False):
    """A read-back array as the program keeps it: in the run's own precision."""
    t = torch.from_numpy(np.ascontiguousarray(a))
    if storage == "fp64":
        return t
    if storage == "fp32":
        return t.float()
    return (t * HALF_SCALE if velocity else t).half()


def _keep_motion(p, storage, turning=True):
    out = {"uv": _keep(np.stack([p["ux"], p["uy"]]), storage, velocity=True)}
    # positions in a 16-bit run need more than 11 bits
    out["xy"] = _keep(np.stack([p["x"], p["y"]]), "fp64" if storage == "fp64" else "fp32")
    if turning:
        out["turn"] = _keep(np.stack([p["theta"], p["omega"]]), storage, velocity=True)
    return out


def _keep_fields(f, storage):
    return {k: _keep(f[k], storage, velocity=k != "T") for k in ("ux", "uy", "T") if k in f}


def _joined(parts):
    return {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in parts[0]} if parts else {}


def run(state):
    case, lattices = state["case"], state["run"].lattices
    steps = case["steps"]
    if case["kind"] == "serve":
        srv = state["run"].server
        ids = [srv.submit(prm, xy, radius, T0, steps) for prm, xy, radius, T0 in state["requests"]]
        while True:
            queued, active, _ = srv.poll()
            if queued + active == 0:
                break
        out = {"fp32": [], "fp16": []}
        for cid, c in zip(ids, state["sims"]):
            fields, motion = srv.take(cid)
            storage = c.params["precision"]
            # (the spin of a disk released at rest is mostly rounding: not kept)
            out[storage].append(_keep_fields(fields, storage) | _keep_motion(motion, storage, turning=False))
        return {storage: _joined(parts) for storage, parts in out.items()}
    storage = case["storage"]
    if case["kind"] == "track":
        path = []
        for _ in range(steps):
            lattices[0].step(1)
            path.append(lattices[0].particles())
        return _keep_motion({k: np.stack([p[k] for p in path]) for k in MOTION}, storage)
    if case["kind"] == "batch":
        V.vlb_step_batch([lat.h for lat in lattices], steps)
        motion = [lat.particles() for lat in lattices]
        fields = [_keep_fields(lat.fields(V.VLB_FIELD_T), storage) for lat in lattices]
        return {"motion": _keep_motion({k: np.concatenate([m[k] for m in motion]) for k in MOTION}, storage),
                "fields": _joined(fields)}
    lattices[0].step(steps)
    return {"motion": _keep_motion(lattices[0].particles(), storage),
            "fields": _keep_fields(lattices[0].fields(V.VLB_FIELD_UX | V.VLB_FIELD_UY | V.VLB_FIELD_T), storage)}


# ---- the work of a pass -----------------------------------------------------

def work(case):
    """Each step reads and writes the 18 populations of every cell once, in
    the storage type; about 400 operations per cell (two nine-moment
    transforms there and back, both equilibria, the temperature solve)."""
    nbytes = flops = 0.0
    for c in _simulations(case, 1):
        updates = c.cells * case["steps"]
        nbytes += updates * 2 * 18 * STORED_BYTES[c.params["precision"]]
        flops += updates * 400
    return {"bytes": nbytes, "flops": flops}


# ---- the time step in 64 bits -----------------------------------------------
# D2Q9 velocities, weights and opposites; rows of the moment basis
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WEIGHT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _basis():
    e2 = [x * x + y * y for x, y in zip(EX, EY)]
    rows = [[1] * 9, [3 * s - 4 for s in e2], [4 - 10.5 * s + 4.5 * s * s for s in e2], EX,
            [(3 * s - 5) * x for s, x in zip(e2, EX)], EY, [(3 * s - 5) * y for s, y in zip(e2, EY)],
            [x * x - y * y for x, y in zip(EX, EY)], [x * y for x, y in zip(EX, EY)]]
    return torch.tensor(rows, dtype=torch.float64, device="cuda")


def _covered(x, y, X, Y, a, b, theta):
    """Area of the ellipse (centre X, Y, semi-axes a, b, angle theta) in the
    unit cell with lower-left corner (x, y): the cell's edges, seen in the
    frame where the ellipse is the unit disk, clipped to the disk, plus the
    sectors under the parts of the edges outside it."""
    c, s = torch.cos(theta), torch.sin(theta)
    us, vs = [], []
    for i, j in ((0, 0), (1, 0), (1, 1), (0, 1)):
        dx, dy = x + i - X, y + j - Y
        us.append((c * dx + s * dy) / a)
        vs.append((c * dy - s * dx) / b)

    def sector(u0, v0, u1, v1):
        return torch.atan2(u0 * v1 - v0 * u1, u0 * u1 + v0 * v1)

    twice = 0.0
    for k in range(4):
        u, v = us[k], vs[k]
        du, dv = us[(k + 1) % 4] - u, vs[(k + 1) % 4] - v
        q, p = du * du + dv * dv, u * du + v * dv
        disc = p * p - q * (u * u + v * v - 1.0)
        root = torch.sqrt(disc.clamp(min=0.0))
        t0, t1 = ((-p - root) / q).clamp(0.0, 1.0), ((-p + root) / q).clamp(0.0, 1.0)
        ua, va, ub, vb = u + t0 * du, v + t0 * dv, u + t1 * du, v + t1 * dv
        cut = sector(u, v, ua, va) + (ua * vb - va * ub) + sector(ub, vb, u + du, v + dv)
        twice = twice + torch.where((disc > 0.0) & (t1 > t0), cut, sector(u, v, u + du, v + dv))
    return (0.5 * a * b * twice).clamp(0.0, 1.0)


class _Exact:
    """The coupled time step of one simulation, in 64 bits, phase by phase."""

    def __init__(self, c):
        def vec(values):
            return torch.tensor(values, dtype=torch.float64, device="cuda")

        q = c.params
        self.q, self.nx, self.ny = q, q["nx"], q["ny"]
        self.nu = (q["tau_f"] - 0.5) / 3.0
        self.lam_f, self.cvs = self.nu / q["prandtl"], q["cv_ratio"]
        self.cref = 2.0 * self.cvs / (1.0 + self.cvs)
        self.force = [-q["beta"] * g for g in q["gravity"]]
        self.M = _basis()
        self.Minv = torch.linalg.inv(self.M)
        self.w = vec(WEIGHT)[:, None, None]
        self.open = q.get("outflow", (0, 0, 0, 0))
        n = len(c.x)
        self.X, self.Y = vec(c.x), vec(c.y)
        self.a = vec(c.radius)
        self.b = self.a if c.semi_minor is None else vec(c.semi_minor)
        self.theta = torch.zeros_like(self.X) if c.theta0 is None else vec(c.theta0)
        self.U, self.V, self.O = vec(c.uv[0::2]), vec(c.uv[1::2]), vec(c.omega)
        self.before = (self.U, self.V, self.O)
        self.T0, self.lam_s = vec(c.T0), vec(c.k_ratio or [q["k_ratio_default"]] * n) * self.lam_f
        self.hold = vec(c.fixed_T or [0] * n)
        self.any_hold = bool(c.fixed_T and any(c.fixed_T))
        area = math.pi * self.a * self.b
        self.inside = (area, 0.25 * area * (self.a ** 2 + self.b ** 2))
        self.weight = (q["rho_ratio"] - 1.0) * area
        self.stiff = abs(q["rho_ratio"] - 1.0) * math.hypot(*q["gravity"]) * math.pi
        half = int(math.ceil(float(self.a.max()))) + 2
        span = torch.arange(-half, half + 1, device="cuda", dtype=torch.float64)
        self.box = (span.repeat(span.numel()), span.repeat_interleave(span.numel()))
        # the initial state: fluid at rest, each cell's energy the mix of its parts
        self._cover()
        shape = (9, self.ny, self.nx)
        f = self._correct(self.w.expand(shape).clone())
        T = ((1.0 - self.fs) * q["T_fluid_init"] + self.solid_eps) / self.cv
        g = self._energy(self.cv * T, T)
        self.dfs = torch.zeros_like(self.fs)
        rho, j = f.sum(0), self._flux(f)
        self._collide(f, g, rho, self._velocity(rho, j, T), T, self.cv * T, torch.zeros_like(T))

    @staticmethod
    def _flux(f):
        return f[1] - f[3] + f[5] - f[6] - f[7] + f[8], f[2] - f[4] + f[5] + f[6] - f[7] - f[8]

    def _energy(self, eps, T):
        g = self.w * self.cref * T
        g[0] = eps - 5.0 / 9.0 * self.cref * T
        return g

    def _spread(self, per_cell):
        """Values [particle, box cell] added up over the lattice."""
        total = torch.zeros(self.ny * self.nx, dtype=torch.float64, device="cuda")
        return total.index_add_(0, self.at, per_cell.reshape(-1)[self.pick]).view(self.ny, self.nx)

    def _cover(self):
        """Solid fraction, rigid-body velocity sums and properties at the current positions."""
        x = torch.floor(self.X)[:, None] + self.box[0]
        y = torch.floor(self.Y)[:, None] + self.box[1]
        col = [v[:, None] for v in (self.X, self.Y, self.a, self.b, self.theta)]
        share = _covered(x, y, *col)
        share = torch.where(share > 1e-11, share, 0.0)  # (rounding of cells that it does not reach)
        on = (share > 0.0) & (x >= 0) & (x < self.nx) & (y >= 0) & (y < self.ny)
        self.pick = on.reshape(-1).nonzero()[:, 0]  # the (particle, box cell) pairs that count, and their cells
        self.at = (y * self.nx + x).reshape(-1)[self.pick].long()
        rx, ry = x + 0.5 - col[0], y + 0.5 - col[1]
        ux, uy = self.U[:, None] - self.O[:, None] * ry, self.V[:, None] + self.O[:, None] * rx
        self.share, self.arm, self.us = share, (rx, ry), (ux, uy)
        self.fs = self._spread(share)
        self.moving = [self._spread(share * m) for m in (ux, uy, ux * ux, ux * uy, uy * uy)]
        self.lam = (1.0 - self.fs) * self.lam_f + self._spread(share * self.lam_s[:, None])
        self.cv = (1.0 - self.fs) + self.fs * self.cvs
        self.solid_eps = self._spread(share * self.cvs * self.T0[:, None])

    def _correct(self, f):
        """Volumetric correction of f; the exchange force and torque."""
        rho, (jx, jy) = f.sum(0), self._flux(f)
        rho_p, jx_p, jy_p = (torch.zeros_like(self.share) for _ in range(3))
        inside = torch.zeros_like(self.share)
        for to, field in ((rho_p, rho), (jx_p, jx), (jy_p, jy)):
            to.view(-1)[self.pick] = field.reshape(-1)[self.at]
        inside.view(-1)[self.pick] = self.share.reshape(-1)[self.pick]
        px, py = -inside * (rho_p * self.us[0] - jx_p), -inside * (rho_p * self.us[1] - jy_p)
        self.exchange = (px.sum(1), py.sum(1), (self.arm[0] * py - self.arm[1] * px).sum(1))
        mx, my, mxx, mxy, myy = self.moving
        keep = 1.0 - self.fs
        out = torch.empty_like(f)
        for i in range(9):
            feq = (self.fs + 3.0 * (EX[i] * mx + EY[i] * my) - 1.5 * (mxx + myy)
                   + 4.5 * (EX[i] ** 2 * mxx + 2 * EX[i] * EY[i] * mxy + EY[i] ** 2 * myy))
            out[i] = keep * f[i] + WEIGHT[i] * rho * feq
        return out

    def _hold(self, g):
        """Held particles: their part of each cell, or the whole cell, at T0."""
        share = self.share * (self.hold > 0)[:, None]
        share = torch.where((self.hold == 2)[:, None] & (share > 0.0), 1.0, share)
        total, T = self._spread(share), self._spread(share * self.T0[:, None])
        scale = 1.0 / total.clamp(min=1.0)
        return (1.0 - total * scale) * g + self._energy(self.cvs * T * scale, T * scale)

    def _velocity(self, rho, j, T):
        free = 0.5 * (1.0 - self.fs) * (T - self.q["T_ref"]) / rho
        return j[0] / rho + free * self.force[0], j[1] / rho + free * self.force[1]

    def _stream(self, s, wall_T=None):
        """Pull streaming; closed sides bounce back (to wall_T where given), open ones copy."""
        out = torch.empty_like(s)

        def bounced(i, rows, cols, wall):
            back = s[OPP[i]][rows, cols]
            if wall_T is None or not self.q["thermal_wall"][wall]:
                return back
            return 2.0 * WEIGHT[i] * self.cref * wall_T[wall] - back

        every = slice(None)
        for i in range(9):
            to = torch.roll(s[i], (EY[i], EX[i]), (0, 1))
            x_wall, y_wall = (0 if EX[i] > 0 else 1), (2 if EY[i] > 0 else 3)
            column, row = (0 if EX[i] > 0 else -1), (0 if EY[i] > 0 else -1)
            if EX[i]:
                to[:, column] = (torch.roll(s[i][:, column], EY[i], 0) if self.open[x_wall]
                                 else bounced(i, every, column, x_wall))
            if EY[i]:
                if self.open[y_wall]:
                    to[row] = torch.roll(s[i][row], EX[i], 0)
                    if EX[i]:
                        to[row, column] = (s[i][row, column] if self.open[x_wall]
                                           else bounced(i, row, column, x_wall))
                else:
                    to[row] = bounced(i, row, every, y_wall)
            out[i] = to
        return out

    def _collide(self, f, g, rho, u, T, eps, qc):
        q = self.q
        ux, uy = u
        free = (1.0 - self.fs) * (T - q["T_ref"])
        Fx, Fy = free * self.force[0], free * self.force[1]
        sq = 1.0 / (0.5 + (1.0 / 12.0) / (q["tau_f"] - 0.5))
        u2, Fu = ux * ux + uy * uy, Fx * ux + Fy * uy
        equal = (rho, rho * (3.0 * u2 - 2.0), rho * (1.0 - 3.0 * u2), rho * ux, -rho * ux, rho * uy, -rho * uy,
                 rho * (ux * ux - uy * uy), rho * ux * uy)
        push = (0.0, 6.0 * Fu, -6.0 * Fu, Fx, -Fx, Fy, -Fy, 2.0 * (Fx * ux - Fy * uy), Fx * uy + Fy * ux)
        rates = (1.0, 1.25, 1.25, 1.0, sq, 1.0, sq, 1.0 / q["tau_f"], 1.0 / q["tau_f"])
        m = torch.tensordot(self.M, f, 1)
        for k in range(9):
            m[k] += rates[k] * (equal[k] - m[k]) + (1.0 - 0.5 * rates[k]) * push[k]
        self.f = torch.tensordot(self.Minv, m, 1)
        tau = 0.5 + 3.0 * self.lam / self.cref
        sj = 1.0 / tau
        se = 1.0 / (0.5 + 0.25 / (tau - 0.5)) if q["thermal_rates_mode"] == 0 else 1.0
        ct = self.cref * T
        m = torch.tensordot(self.M, g, 1)
        m[0] = eps + 0.5 * qc
        m[1] += se * (2.0 * ct - 4.0 * eps - m[1]) - (1.0 - 0.5 * se) * 4.0 * qc
        m[2] += se * (4.0 * eps - 3.0 * ct - m[2]) + (1.0 - 0.5 * se) * 4.0 * qc
        for k in (3, 4, 5, 6):
            m[k] *= 1.0 - sj
        for k in (7, 8):
            m[k] *= 1.0 - se
        self.g = torch.tensordot(self.Minv, m, 1)
        self.u, self.T = u, T

    def _contacts(self):
        """Repulsion between particles (on their circumscribed disks) and by closed walls."""
        q, zeta = self.q, 2.0
        dx, dy = self.X[:, None] - self.X, self.Y[:, None] - self.Y
        d = torch.sqrt(dx * dx + dy * dy).fill_diagonal_(1e9)
        gap = (self.a[:, None] + self.a + zeta - d).clamp(min=0.0)
        push = self.stiff / 0.01 * torch.maximum(self.a[:, None], self.a) ** 2 * (gap / zeta) ** 2 / d
        Fx, Fy = (push * dx).sum(1), (push * dy).sum(1)
        c, s = torch.cos(self.theta), torch.sin(self.theta)
        reach = (torch.sqrt((self.a * c) ** 2 + (self.b * s) ** 2), torch.sqrt((self.a * s) ** 2 + (self.b * c) ** 2))
        away = []
        for wall, dist in enumerate((self.X, self.nx - self.X, self.Y, self.ny - self.Y)):
            gap = (2.0 * reach[wall // 2] + zeta - 2.0 * dist).clamp(min=0.0)
            away.append(0.0 if self.open[wall] else self.stiff / 0.005 * self.a ** 2 * (gap / zeta) ** 2)
        return Fx + away[0] - away[1], Fy + away[2] - away[3]

    def step(self):
        # particles: forward Euler with the force of the last level
        gx, gy = self.q["gravity"]
        Cx, Cy = self._contacts()
        Fx = self.exchange[0] + self.inside[0] * (self.U - self.before[0]) + self.weight * gx + Cx
        Fy = self.exchange[1] + self.inside[0] * (self.V - self.before[1]) + self.weight * gy + Cy
        Tc = self.exchange[2] + self.inside[1] * (self.O - self.before[2])
        self.before = (self.U, self.V, self.O)
        self.X, self.Y, self.theta = self.X + self.U, self.Y + self.V, self.theta + self.O
        ratio = self.q["rho_ratio"]
        self.U = self.U + Fx / (ratio * self.inside[0])
        self.V = self.V + Fy / (ratio * self.inside[0])
        self.O = self.O + Tc / (ratio * self.inside[1])
        # lattice
        fs_old = self.fs
        self._cover()
        f = self._correct(self._stream(self.f))
        g = self._stream(self.g, self.q["wall_T"])
        if self.any_hold:
            g = self._hold(g)
        self.dfs = 2.0 * (self.fs - fs_old) - self.dfs
        rho, j, G = f.sum(0), self._flux(f), g.sum(0)
        slope = -3.0 / (self.cref * (0.5 + 3.0 * self.lam / self.cref))
        Tx, Ty = (slope * v for v in self._flux(g))
        extra = (self.cvs - 1.0) * self.dfs
        still = self._velocity(rho, j, torch.full_like(rho, self.q["T_ref"]))
        lift = 0.5 * (1.0 - self.fs) / rho * (self.force[0] * Tx + self.force[1] * Ty)
        T = ((G - 0.5 * self.cv * (still[0] * Tx + still[1] * Ty - self.q["T_ref"] * lift))
             / (self.cv - 0.5 * extra + 0.5 * self.cv * lift))
        u = self._velocity(rho, j, T)
        qc = -self.cv * (u[0] * Tx + u[1] * Ty) + extra * T
        self._collide(f, g, rho, u, T, G + 0.5 * qc, qc)

    def motion(self):
        return dict(zip(MOTION, (self.X, self.Y, self.theta, self.U, self.V, self.O)))

    def fields(self):
        return {"ux": self.u[0], "uy": self.u[1], "T": self.T}


def _exact_motion(m, storage, turning=True):
    scale = HALF_SCALE if storage in ("fp16", "bf16") else 1.0
    out = {"uv": scale * torch.stack([m["ux"], m["uy"]]), "xy": torch.stack([m["x"], m["y"]])}
    return out | ({"turn": scale * torch.stack([m["theta"], m["omega"]])} if turning else {})


def _exact_fields(f, storage):
    scale = HALF_SCALE if storage in ("fp16", "bf16") else 1.0
    return {k: v * (1.0 if k == "T" else scale) for k, v in f.items()}


def exact(case, seed):
    sims = _simulations(case, seed)
    if sum(c.cells for c in sims) * case["steps"] > MOST_CELL_STEPS:
        return None  # over about 20 seconds
    kind, done, path = case["kind"], [], []
    for c in sims:
        e = _Exact(c)
        for _ in range(case["steps"]):
            e.step()
            if kind == "track":
                path.append(e.motion())
        done.append((c.params["precision"], e.motion(), e.fields()))
        del e
    if kind == "serve":
        return {s: _joined([_exact_fields(f, s) | _exact_motion(m, s, False) for t, m, f in done if t == s])
                for s in ("fp32", "fp16")}
    storage = case["storage"]
    if kind == "track":
        return _exact_motion({k: torch.stack([p[k] for p in path]) for k in MOTION}, storage)
    if kind == "batch":
        return {"motion": _exact_motion(_joined([m for _, m, _ in done]), storage),
                "fields": _joined([_exact_fields({"T": f["T"]}, storage) for _, _, f in done])}
    return {"motion": _exact_motion(done[0][1], storage), "fields": _exact_fields(done[0][2], storage)}
