"""Performance cases of the IB-LBM library: what a user's program has it do, through its public calls.

Six kinds of case, each a whole piece of work as a program asks for it:

* ``cylinder``  the 2D validation runs: a rigid cylinder in a body-force-driven channel (D2Q9), started from
                rest, advanced some hundred steps; the fields and the drag/lift history are read back.
* ``foils``     the paper's own runs: two elliptic foils doing clap and fling, or one hovering foil (D2Q9).
* ``wings``     the 3D clap-and-fling wing pair (D3Q19) started from rest: force histories of both wings, the
                marker state and the flow at a set of wake probes (the whole field of a large box is dumped
                rarely; the probes and the forces are what a run returns).
* ``tgv``       pure lattice Boltzmann (Taylor-Green vortex): set the velocity field, advance, read the fields.
* ``points``    the two immersed-boundary transfers on a cloud of points (device arrays), without the solve.
* ``serving``   a batch of clap-and-fling requests given to the server, which advances them together.

A run restarts its fluid, so every pass on a state does the same work.  Runs with bodies return their results
in the precision in which they store their populations (the calls hand out doubles whatever the storage); the
large fields of the pure runs stay the arrays that the calls fill.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_2102_01305_gb300 import ibl

DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16dev": torch.float16, "bf16dev": torch.bfloat16}
BYTES = {"fp64": 8, "fp32": 4, "fp16dev": 2, "bf16dev": 2}
SERVED_GRIDS = ((96, 96, 96, 8.0), (160, 128, 112, 12.0))


def listed():
    return [
        # the smallest run in earnest: the 2D cylinder configuration, FP64; every kernel is tiny, launches,
        # barriers and latencies are all there is
        {"name": "cylinder-200x100-fp64", "kind": "cylinder", "nx": 200, "ny": 100, "diameter": 20.0, "markers": 63,
         "precision": "fp64", "steps": 500},
        # the paper's clap-and-fling foils (Sec. 3.3), velocity inlet and pressure outlet, FP32
        {"name": "foils-800x400-fp32", "kind": "foils", "motion": "clap", "chord": 16, "precision": "fp32",
         "steps": 300},
        # the wing pair in the serving sweep's smallest box, 16-bit storage
        {"name": "wings-96-fp16", "kind": "wings", "nx": 96, "ny": 96, "nz": 96, "chord": 8.0, "Re": 75.0,
         "u_tip": 0.035, "precision": "fp16dev", "steps": 200, "probes": 20000},
        # the wing pair of the 3D configuration, FP32
        {"name": "wings-256x192x160-fp32", "kind": "wings", "nx": 256, "ny": 192, "nz": 160, "chord": 20.0,
         "Re": 100.0, "u_tip": 0.0209, "precision": "fp32", "steps": 100, "probes": 20000},
        # the largest single-GPU run: 63 million cells, 2 x 6292 markers
        {"name": "wings-512x384x320-fp32", "kind": "wings", "nx": 512, "ny": 384, "nz": 320, "chord": 40.0,
         "Re": 150.0, "u_tip": 0.0209, "precision": "fp32", "steps": 40, "probes": 20000},
        # pure LBM: the sweep's smallest cube (it fits the L2 cache) ...
        {"name": "tgv-64-fp32", "kind": "tgv", "nx": 64, "ny": 64, "nz": 64, "precision": "fp32", "steps": 500},
        # ... an ordinary cube in FP32 and in 16-bit storage ...
        {"name": "tgv-256-fp32", "kind": "tgv", "nx": 256, "ny": 256, "nz": 256, "precision": "fp32", "steps": 500},
        {"name": "tgv-256-fp16", "kind": "tgv", "nx": 256, "ny": 256, "nz": 256, "precision": "fp16dev",
         "steps": 500},
        # ... and a ragged box whose odd width rules out two cells a thread
        {"name": "tgv-151x97x83-bf16", "kind": "tgv", "nx": 151, "ny": 97, "nz": 83, "precision": "bf16dev",
         "steps": 500},
        # the transfers alone: a marker set of ordinary size, and one that covers the whole grid
        {"name": "points-256-1e4", "kind": "points", "nx": 256, "ny": 256, "nz": 256, "points": 10000,
         "precision": "fp32"},
        {"name": "points-256-1e6", "kind": "points", "nx": 256, "ny": 256, "nz": 256, "points": 1000000,
         "precision": "fp32"},
        # eight requests of mixed grids and storage types, run together
        {"name": "serving-8", "kind": "serving", "runs": 8, "steps": 400},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cylinder", "foils", "wings", "wings", "wings", "tgv", "tgv", "tgv", "points", "points",
                       "points", "serving"])
    if kind == "cylinder":
        ny = _log_int(rng, 60, 240)
        nx = int(ny * rng.uniform(1.5, 2.5))
        d = round(ny * rng.uniform(0.15, 0.25), 2)
        return {"kind": kind, "nx": nx, "ny": ny, "diameter": d, "markers": max(16, int(round(math.pi * d))),
                "precision": rng.choice(["fp64", "fp32"]), "steps": rng.randint(200, 500)}
    if kind == "foils":
        return {"kind": kind, "motion": rng.choice(["clap", "hover"]), "chord": _log_int(rng, 10, 24),
                "precision": rng.choice(["fp64", "fp32"]), "steps": rng.randint(100, 300)}
    if kind == "wings":
        nx = _log_int(rng, 64, 320)
        ny, nz = int(nx * rng.uniform(0.75, 1.0)), int(nx * rng.uniform(0.75, 1.0))
        chord = round(min((nz - 10) / 5.0, (ny - 10) / 3.0) * rng.uniform(0.6, 0.85), 1)
        steps = max(40, min(200, int(1.2e9 / (nx * ny * nz))))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "chord": chord,
                "Re": round(min(rng.uniform(60.0, 150.0), 6.0 * chord), 1),
                "u_tip": round(rng.uniform(0.02, 0.04), 4),
                "precision": rng.choice(["fp32", "fp32", "fp16dev", "bf16dev"]), "steps": steps,
                "probes": _log_int(rng, 1000, 50000)}
    if kind == "tgv":
        n = _log_int(rng, 48, 256)
        nx, ny, nz = (max(32, int(n * rng.uniform(0.7, 1.0))) for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz,
                "precision": rng.choice(["fp32", "fp32", "fp16dev", "bf16dev", "fp64"]),
                "steps": rng.randint(100, 300)}
    if kind == "points":
        n = rng.choice([96, 131, 192, 256])
        return {"kind": kind, "nx": n, "ny": int(n * rng.uniform(0.7, 1.0)), "nz": int(n * rng.uniform(0.7, 1.0)),
                "points": _log_int(rng, 1000, 1000000),
                "precision": rng.choice(["fp32", "fp32", "fp16dev", "fp64"])}
    return {"kind": kind, "runs": rng.randint(3, 8), "steps": rng.randint(150, 400)}


# ------------------------------------------------------------------ inputs
def _workload(case, seed):
    """Workload dict of a stepping case; the seed moves the bodies (position, phase) or the vortex."""
    r = np.random.default_rng([20210203, seed])
    k = case["kind"]
    if k == "cylinder":
        cfg = W.cylinder_channel(nx=case["nx"], ny=case["ny"], diameter=case["diameter"],
                                 center=(0.25 * case["nx"] + r.uniform(-1, 1), 0.5 * case["ny"] + r.uniform(-1, 1)),
                                 m=case["markers"], u_mean=0.05 * r.uniform(0.9, 1.1), precision=case["precision"])
    elif k == "foils":
        if case["motion"] == "clap":
            cfg = W.clap_fling_2d(chord=case["chord"], Re=50.0, period=50.0 * case["chord"], precision=case["precision"])
        else:
            cfg = W.figure_eight_2d(chord=case["chord"], period=125.0 * case["chord"], precision=case["precision"])
        phi = r.uniform(0.0, 2.0 * math.pi)
        off = r.uniform(-0.5, 0.5, size=2)
        for b in cfg["bodies"]:
            b["phi"] = phi
            b["origin"] = (b["origin"][0] + off[0], b["origin"][1] + off[1], 0.0)
    elif k == "wings":
        period = 2.0 * math.radians(120.0) * case["chord"] / case["u_tip"]
        cfg = W.clap_fling_3d(nx=case["nx"], ny=case["ny"], nz=case["nz"], chord=case["chord"], Re=case["Re"], J=0.0,
                              period=period, precision=case["precision"], faces="periodic",
                              hinge_x=round(case["nx"] / 3.0) + r.uniform(-0.5, 0.5),
                              phase=r.uniform(0.0, 2.0 * math.pi))
    else:
        n = (case["nx"], case["ny"], case["nz"])
        cfg = W.taylor_green_3d(n=8, precision=case["precision"])
        cfg["grid"].update(nx=n[0], ny=n[1], nz=n[2])
        u = W.tgv3d_velocity(*n, 0.05)
        u = np.roll(u, [int(r.integers(0, m)) for m in n], axis=(3, 2, 1))
        cfg["u_field"] = np.ascontiguousarray(u * r.uniform(0.9, 1.1))
    return cfg


def _requests(case, seed):
    r = np.random.default_rng([64, seed])
    out = []
    for i in range(case["runs"]):
        nx, ny, nz, c = SERVED_GRIDS[i % 2]
        out.append({"nx": nx, "ny": ny, "nz": nz, "chord": c, "Re": float(r.choice([75.0, 100.0])),
                    "period": 200.0 * c, "J": float(r.choice([1e-3, 1e-2])),
                    "precision": ("fp32", "fp16dev")[(i // 2) % 2], "steps": case["steps"]})
    return out


def _cloud(case, seed, m, margin=2.0):
    r = np.random.default_rng([7, seed])
    n = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64)
    return margin + r.uniform(size=(m, 3)) * (n - 2.0 * margin), r.uniform(-0.05, 0.05, size=(m, 3))


def prepare(case, seed):
    k = case["kind"]
    if k == "serving":
        return {"kind": k, "server": ibl.Server(64 << 30, max_active=8), "requests": _requests(case, seed)}
    cfg = _workload(case, seed)
    s = {"kind": k, "ctx": ibl.from_workload(cfg, init=False), "steps": case.get("steps", 1),
         "dtype": DTYPE[case["precision"]], "bodies": [b["X0"].shape[0] for b in cfg["bodies"]]}
    if k == "tgv":
        s["u"] = cfg["u_field"]
    elif k == "wings":
        s["probes"] = torch.from_numpy(_cloud(case, seed, case["probes"])[0]).cuda()
    elif k == "points":
        s["ctx"].ibl_init_fluid(None, cfg["u_field"])
        s["ctx"].ibl_step(1)
        s["ctx"].ibl_sync()
        X, V = _cloud(case, seed, case["points"])
        s["X"], s["V"] = torch.from_numpy(X).cuda(), torch.from_numpy(V).cuda()
        s["ds"] = torch.ones(case["points"], dtype=torch.float64, device="cuda")
    return s


def run(s):
    k = s["kind"]
    if k == "serving":
        srv = s["server"]
        ids = [srv.ibl_server_submit(**rq) for rq in s["requests"]]
        srv.ibl_server_wait_all(60.0)
        out = []
        for i, rq in zip(ids, s["requests"]):
            res = srv.ibl_server_poll(i)
            vals = [res[q] for q in ("CL_max", "CL_mean", "CT_max", "CT_mean", "CL_last", "CT_last")]
            out.append({"status": res["status"], "coefficients": torch.tensor(vals, dtype=DTYPE[rq["precision"]])})
        return out
    ctx = s["ctx"]
    if k == "points":
        U, rho = ctx.ibl_interpolate_points(s["X"])
        return {"U": U, "rho": rho, "spread": ctx.ibl_spread_points(s["X"], s["V"], s["ds"])}

    def own(a):
        if k == "tgv" or s["dtype"] == torch.float64:
            return a
        return a.astype(np.float32) if s["dtype"] == torch.float32 else torch.from_numpy(a).to(s["dtype"])

    # the markers' single forces are left out: a sheet's system is nearly singular in its checkerboard mode, so
    # the library determines (and its tests judge) fields and coefficients, not single marker corrections
    ctx.ibl_init_fluid(None, s.get("u"))
    ctx.ibl_step(s["steps"])
    out = {"history": [own(ctx.ibl_force_history(b, s["steps"])) for b in range(len(s["bodies"]))],
           "markers": [[own(a) for a in ctx.ibl_get_markers(b, m)[:2]] for b, m in enumerate(s["bodies"])]}
    if k == "wings":
        out["probes"] = [t.to(s["dtype"]) for t in ctx.ibl_interpolate_points(s["probes"])]
    else:
        out["u"] = own(ctx.ibl_get_field(ibl.IBL_FIELD_U))
        out["rho"] = own(ctx.ibl_get_field(ibl.IBL_FIELD_RHO))
    return out


def _shape(case):
    """(cells, directions, dimensions) of a stepping or points case."""
    if case["kind"] == "foils":
        return 50 * case["chord"] * 25 * case["chord"], 9, 2
    if case["kind"] == "cylinder":
        return case["nx"] * case["ny"], 9, 2
    return case["nx"] * case["ny"] * case["nz"], 19, 3


def work(case):
    """Every step reads and writes each population once; the results (and a given velocity field) move once."""
    if case["kind"] == "serving":
        b = f = 0
        for i in range(case["runs"]):
            nx, ny, nz, _ = SERVED_GRIDS[i % 2]
            b += case["steps"] * nx * ny * nz * 38 * (4, 2)[(i // 2) % 2]
            f += case["steps"] * nx * ny * nz * 300
        return {"bytes": b, "flops": f}
    n, q, d = _shape(case)
    if case["kind"] == "points":
        m = case["points"]
        # interpolation: the populations of the covered cells once, points in, results out; spreading: points
        # in, the dense result out
        covered = n * (1.0 - math.exp(-64.0 * m / n))
        return {"bytes": q * BYTES[case["precision"]] * covered + m * (24 + 32) + m * (24 + 24 + 8) + 24 * n,
                "flops": m * 64 * (3 + 8 + 6)}
    e = BYTES[case["precision"]]
    b = case["steps"] * n * 2 * q * e
    if case["kind"] == "wings":
        b += case["probes"] * 56
    else:
        b += (d + 1) * n * 8 + (d * n * 8 if case["kind"] == "tgv" else 0)
    return {"bytes": b, "flops": case["steps"] * n * (120 if q == 9 else 300)}


# ------------------------------------------------------------------ the same runs in 64 bits
class _Exact:
    """The method in plain FP64 torch: BGK with the Guo source, halfway bounce-back and Zou-He faces, the
    4-point cosine delta and a dense solve of the implicit velocity correction."""

    def __init__(self, cfg):
        g = cfg["grid"]
        self.n = (g["nx"], g["ny"], g["nz"])
        self.d = d = 2 if cfg["lattice"] == 9 else 3
        c = [(x, y, z) for x in (0, 1, -1) for y in (0, 1, -1) for z in ((0, 1, -1) if d == 3 else (0,))
             if abs(x) + abs(y) + abs(z) <= 2]
        self.c = c
        first = {2: (4 / 9, 1 / 9, 1 / 36), 3: (1 / 3, 1 / 18, 1 / 36)}[d]
        self.w = [first[sum(map(abs, v))] for v in c]
        self.opp = [c.index(tuple(-x for x in v)) for v in c]
        self.bc, self.u_in, self.rho_out = g["bc"], g["u_in"], g["rho_out"]
        self.G, self.tau, self.cfg = g["body_force"], cfg["tau"], cfg
        self.dev = torch.device("cuda")
        self.t64 = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=self.dev)
        self.bodies = [(self.t64(np.pad(np.asarray(b["X0"])[:, :d], ((0, 0), (0, 3 - d)))), b) for b in cfg["bodies"]]
        self.history = [[] for _ in self.bodies]
        self.markers = None

    def start(self, u=None):
        shape = self.n[::-1]
        u = torch.zeros((3,) + shape, dtype=torch.float64, device=self.dev) if u is None else self.t64(u)
        self.f, self.step_no, self.streamed = self.equilibrium(torch.ones(shape, dtype=torch.float64, device=self.dev), u), 0, True

    def equilibrium(self, rho, u):
        usq = (u * u).sum(0)
        f = torch.empty((len(self.c),) + tuple(rho.shape), dtype=torch.float64, device=self.dev)
        for i, c in enumerate(self.c):
            cu = sum(c[a] * u[a] for a in range(3) if c[a]) if any(c) else 0.0
            f[i] = self.w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
        return f

    def stream(self):
        """Post-streaming populations of the present state."""
        if self.streamed:
            return self.f
        p, g = self.f, torch.empty_like(self.f)
        for i, c in enumerate(self.c):
            g[i] = torch.roll(p[i], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
        for face in range(2 * self.d):
            a, side = face // 2, face % 2
            if self.bc[face] == W.PERIODIC:
                continue
            s = -1 if side else 1                   # the inward normal is s e_a
            at = [slice(None)] * 3
            at[2 - a] = self.n[a] - 1 if side else 0
            at = tuple(at)
            into = [i for i, c in enumerate(self.c) if c[a] == s]
            if self.bc[face] == W.BOUNCEBACK:
                for i in into:
                    g[(i,) + at] = p[(self.opp[i],) + at]
                continue
            known = (sum(g[(i,) + at] for i, c in enumerate(self.c) if c[a] == 0)
                     + 2 * sum(g[(i,) + at] for i, c in enumerate(self.c) if c[a] == -s))
            u = [torch.zeros_like(known) for _ in range(3)]
            if self.bc[face] == W.VEL_INLET:
                u = [torch.full_like(known, v) for v in self.u_in]
                rho = known / (1 - s * u[a])
            else:
                rho = torch.full_like(known, self.rho_out)
                u[a] = s * (1 - known / rho)
            cross = {}
            for t in range(self.d):
                if t != a:
                    cross[t] = (0.5 * sum(c[t] * g[(i,) + at] for i, c in enumerate(self.c) if c[a] == 0 and c[t])
                                - rho * u[t] / 3)
            for i in into:
                c = self.c[i]
                v = g[(self.opp[i],) + at] + 6 * self.w[i] * rho * sum(c[b] * u[b] for b in range(3) if c[b])
                for t in cross:
                    if c[t]:
                        v = v - c[t] * cross[t]
                g[(i,) + at] = v
        return g

    def moments(self, g):
        rho = g.sum(0)
        m = torch.stack([sum(c[a] * g[i] for i, c in enumerate(self.c) if c[a]) if a < self.d else torch.zeros_like(rho)
                         for a in range(3)])
        return rho, m

    def fields(self):
        rho, m = self.moments(self.stream())
        return rho, (m + 0.5 * self.t64(self.G)[:, None, None, None]) / rho

    def stencil(self, X):
        """Nodes [m, 4] and weights [m, 4] per axis (Eq. 14), periodic indices."""
        out = []
        for a in range(self.d):
            fl = torch.floor(X[:, a])
            k = torch.arange(-1, 3, device=self.dev)
            r = (X[:, a] - fl)[:, None] - k
            out.append((torch.remainder(fl.long()[:, None] + k, self.n[a]), 0.25 * (1 + torch.cos(0.5 * math.pi * r))))
        return out

    def nodes(self, st):
        """Flat cells [m, 4^d] and delta weights of each point."""
        m = st[0][0].shape[0]
        idx, wt = st[0][0][:, None, :], st[0][1][:, None, :]
        idx, wt = st[1][0][:, :, None] * self.n[0] + idx, st[1][1][:, :, None] * wt
        idx, wt = idx.reshape(m, -1), wt.reshape(m, -1)
        if self.d == 3:
            idx = (st[2][0][:, :, None] * (self.n[0] * self.n[1]) + idx[:, None, :]).reshape(m, -1)
            wt = (st[2][1][:, :, None] * wt[:, None, :]).reshape(m, -1)
        return idx, wt

    def at_points(self, X, part=20000):
        rho, u = self.fields()
        flat = torch.cat([rho.reshape(1, -1), u[:self.d].reshape(self.d, -1)])
        out = []
        for k in range(0, X.shape[0], part):
            idx, wt = self.nodes(self.stencil(X[k:k + part]))
            out.append(torch.stack([(f[idx] * wt).sum(1) for f in flat], 1))
        out = torch.cat(out)
        return out[:, 1:], out[:, 0]

    def spread(self, X, V, part=20000):
        out = torch.zeros((self.d, self.n[0] * self.n[1] * self.n[2]), dtype=torch.float64, device=self.dev)
        for k in range(0, X.shape[0], part):
            idx, wt = self.nodes(self.stencil(X[k:k + part]))
            for a in range(self.d):
                out[a].index_add_(0, idx.reshape(-1), (wt * V[k:k + part, a:a + 1]).reshape(-1))
        return out.reshape((self.d,) + self.n[::-1])

    def wave(self, w, b, t):
        th = 2 * math.pi * b["f"] * t + b["phi"]
        om, amp, off = 2 * math.pi * b["f"], w["amp"], w["offset"]
        if w["kind"] == W.WAVE_COS:
            return off + amp * math.cos(th), -amp * om * math.sin(th)
        if w["kind"] == W.WAVE_SIN:
            return off + amp * math.sin(th), amp * om * math.cos(th)
        if w["kind"] == W.WAVE_ABS_SIN:
            return off + amp * abs(math.sin(th)), amp * om * math.cos(th) * (1 if math.sin(th) >= 0 else -1)
        return off, 0.0

    def body_motion(self, X0, b, t):
        A, Ad = self.wave(b["A"], b, t)
        al, ald = self.wave(b["alpha"], b, t)
        es = self.t64([math.cos(b["beta"]), math.sin(b["beta"]), 0.0])
        e, h = self.t64(b["axis"]).expand_as(X0), self.t64(b["hinge"])
        r = X0 - h
        r = r * math.cos(al) + torch.cross(e, r, dim=1) * math.sin(al) + e * (e * r).sum(1, keepdim=True) * (1 - math.cos(al))
        return self.t64(b["origin"]) + h + r + A * es, Ad * es + ald * torch.cross(e, r, dim=1)

    def advance(self, steps):
        for _ in range(steps):
            g = self.stream()
            rho, m = self.moments(g)
            G = self.t64(self.G)[:, None, None, None]
            F = G.expand_as(m)
            if self.bodies:
                XU = [self.body_motion(X0, b, self.step_no) for X0, b in self.bodies]
                X, U = torch.cat([x for x, _ in XU]), torch.cat([u for _, u in XU])
                st = self.stencil(X)
                idx, wt = self.nodes(st)
                us = ((m + 0.5 * G) / rho).reshape(3, -1)
                B = U[:, :self.d] - torch.stack([(us[a][idx] * wt).sum(1) for a in range(self.d)], 1)
                A = torch.ones((X.shape[0], X.shape[0]), dtype=torch.float64, device=self.dev)
                for a in range(self.d):
                    D = torch.zeros((X.shape[0], self.n[a]), dtype=torch.float64, device=self.dev)
                    D.scatter_add_(1, st[a][0], st[a][1])
                    A *= D @ D.T
                w = torch.linalg.solve(A, B)
                rl = (rho.reshape(-1)[idx] * wt).sum(1)
                du = torch.zeros_like(us)
                for a in range(self.d):
                    du[a].index_add_(0, idx.reshape(-1), (wt * w[:, a:a + 1]).reshape(-1))
                F = G + 2 * rho * du.reshape(m.shape)
                mf = 2 * rl[:, None] * w
                self.markers, o = [], 0
                ref = self.cfg["reference"]
                q = 0.5 * ref["rho_ref"] * ref["U_ref"] ** 2 * ref["L"]
                for k, (X0, b) in enumerate(self.bodies):
                    e = o + X0.shape[0]
                    self.markers.append([X[o:e, :self.d], U[o:e, :self.d]])
                    Fb = (-mf[o:e].sum(0) / q).cpu().numpy()
                    lift = np.asarray(b.get("lift_axis", (0.0, 1.0, 0.0)))[:self.d]
                    self.history[k].append((float(Fb @ lift), -float(Fb[0]), float(Fb[0])))
                    o = e
            u = (m + 0.5 * F) / rho
            eq = self.equilibrium(rho, u)
            uF = (u * F).sum(0)
            for i, c in enumerate(self.c):
                cu = sum(c[a] * u[a] for a in range(3) if c[a]) if any(c) else torch.zeros_like(rho)
                cF = sum(c[a] * F[a] for a in range(3) if c[a]) if any(c) else torch.zeros_like(rho)
                src = (1 - 0.5 / self.tau) * self.w[i] * (3 * (cF - uF) + 9 * cu * cF)
                eq[i] = g[i] - (g[i] - eq[i]) / self.tau + src
            self.f, self.streamed = eq, False
            self.step_no += 1


def exact(case, seed):
    k = case["kind"]
    if k == "serving":
        return None
    n, q, _ = _shape(case)
    if k != "points" and case["steps"] * n > 9e8:   # over about 20 seconds
        return None
    cfg = _workload(case, seed)
    x = _Exact(cfg)
    x.start(cfg.get("u_field"))
    x.advance(case.get("steps", 1))
    if k == "points":
        X, V = (torch.from_numpy(a).cuda() for a in _cloud(case, seed, case["points"]))
        U, rho = x.at_points(X)
        return {"U": U, "rho": rho, "spread": x.spread(X, V)}
    out = {"history": [torch.tensor(h, dtype=torch.float64) for h in x.history], "markers": x.markers or []}
    if k == "wings":
        out["probes"] = list(x.at_points(torch.from_numpy(_cloud(case, seed, case["probes"])[0]).cuda()))
    else:
        rho, u = x.fields()
        out["u"], out["rho"] = u[:x.d], rho
    return out
