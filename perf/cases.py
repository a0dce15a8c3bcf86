"""Performance cases of the lattice Boltzmann library.

Every case is what a program that uses the library does between two looks at
its flow: advance a domain (or a batch of domains, or a two-component mixture)
by some steps and take the result back, through the public Python front end
(`Solver`, `Batch`, `CGSolver`) with the fields left on the GPU.  Sizes,
relaxation times, flows, storages and batch mixes are those of bench.py, of
the tests and of the serving workload, and ragged sizes between them.

A case is a dict of plain values:
  kind      "solver" | "batch" | "cg"
  lattice   "D2Q9" | "D3Q19" | "D3Q27" (batch: "D2Q9+D3Q19" or "D3Q19")
  nx,ny,nz  fluid nodes (nz = 1 in 2D)
  flow      "cavity" (moving lid at +y), "tg" (periodic vortex), "duct" (body
            force along x, walls on the other axes), "channel" (body force
            along x, walls at +-y, periodic elsewhere)
  storage   "f32" | "f16s" | "bf16s" | "f64"
  tau       relaxation time
  steps     time steps of one lb_step call, and
  calls     how many such calls one pass makes
  fresh     1: every pass sets the state from moment fields first (a solve of
            its own); 0: the run goes on from where the last pass left it
  monitor   1: the FP64 reductions with the convergence residual are read too
Every pass of a solver or batch ends with the fields rho and u and the
populations (what a checkpoint keeps) in the caller's device buffers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

Q = {"D2Q9": 9, "D3Q19": 19, "D3Q27": 27}
BYTES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}
LID = 0.05     # lid speed of the cavities
DUCT_U = 0.05  # centre-line speed the driven flows are forced towards


# ------------------------------------------------------------------ the cases
def _solver(name, lattice, dims, flow, storage, tau, steps, calls=1, fresh=0, monitor=0):
    nx, ny, nz = (list(dims) + [1])[:3]
    return dict(name=name, kind="solver", lattice=lattice, nx=nx, ny=ny, nz=nz, flow=flow, storage=storage,
                tau=tau, steps=steps, calls=calls, fresh=fresh, monitor=monitor)


def listed():
    return [
        # the smallest request of the serving workload, 100 steps a round: all latency
        _solver("cavity_d3q19_f32_32", "D3Q19", (32, 32, 32), "cavity", "f32", 0.6, 100),
        # a small 2D cavity with ragged sides, run on its own and checkpointed
        _solver("cavity_d2q9_f32_301x257", "D2Q9", (301, 257), "cavity", "f32", 0.56, 100),
        # a force-driven ragged duct that another program looks at every ten steps
        _solver("duct_d3q19_f32_97x61x113", "D3Q19", (97, 61, 113), "duct", "f32", 0.55, 10, calls=5),
        # the ordinary 3D cavity, watched for convergence
        _solver("cavity_d3q19_f32_256", "D3Q19", (256, 256, 256), "cavity", "f32", 0.52, 50, monitor=1),
        # the largest: the 512^3 cavity, advanced and checkpointed
        _solver("cavity_d3q19_f32_512", "D3Q19", (512, 512, 512), "cavity", "f32", 0.52, 20),
        # a whole solve of the 3D Taylor-Green vortex: fields in, steps, fields out
        _solver("tg_d3q27_f32_256", "D3Q27", (256, 256, 256), "tg", "f32", 0.8, 20, fresh=1),
        # 2D vortex decay over a large square
        _solver("tg_d2q9_f32_4096", "D2Q9", (4096, 4096), "tg", "f32", 0.8, 50, fresh=1),
        # 16-bit storage: half the memory per domain, used by half of the served requests
        _solver("cavity_d3q19_f16s_160", "D3Q19", (160, 160, 160), "cavity", "f16s", 0.55, 50),
        # reduced-precision channel of the accuracy study, ragged
        _solver("channel_d3q27_f16s_200x130x90", "D3Q27", (200, 130, 90), "channel", "f16s", 0.6, 50),
        # double precision, for reference solutions
        _solver("tg_d3q19_f64_96", "D3Q19", (96, 96, 96), "tg", "f64", 0.8, 20),
        # one round of the solve server: a mixed batch, 100 steps, then every member's residual
        dict(name="batch_d2q9_d3q19_f32_24", kind="batch", lattice="D2Q9+D3Q19", members=24, storage="f32",
             mix=11, steps=100),
        # an emulsion in 2D with near-contact repulsion (the two-component model)
        dict(name="cg_d2q9_f32_2048x1536_nci", kind="cg", lattice="D2Q9", nx=2048, ny=1536, nz=1, storage="f32",
             tau=1.0, sigma=0.01, beta=0.7, drops=400, rmin=8, rmax=24, nci=1, steps=50),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["solver", "batch", "cg"], weights=[8, 1, 2])[0]
    if kind == "batch":
        return dict(kind="batch", lattice=rng.choice(["D2Q9+D3Q19", "D3Q19"]), members=rng.randint(6, 32),
                    storage=rng.choice(["f32", "f32", "f16s"]), mix=rng.randint(1, 10 ** 6),
                    steps=rng.choice([10, 50, 100]))
    if kind == "cg":
        lattice = rng.choice(["D2Q9", "D3Q19"])
        if lattice == "D2Q9":
            nx, ny, nz = _logint(rng, 96, 3000), _logint(rng, 96, 3000), 1
            rmin, rmax = 8, 24
        else:
            nx, ny, nz = (_logint(rng, 40, 200) for _ in range(3))
            rmin, rmax = 6, 16
        fill = nx * ny * nz / ((4.0 * rmax) ** (2 if nz == 1 else 3))
        return dict(kind="cg", lattice=lattice, nx=nx, ny=ny, nz=nz, storage=rng.choice(["f32", "f32", "f32", "f64"]),
                    tau=round(rng.uniform(0.8, 1.1), 3), sigma=0.01, beta=0.7,
                    drops=max(2, min(500, int(4 * fill))), rmin=rmin, rmax=rmax, nci=rng.choice([0, 1]),
                    steps=rng.choice([5, 20, 50]))
    lattice = rng.choice(["D2Q9", "D3Q19", "D3Q19", "D3Q27"])
    storage = rng.choice(["f32", "f32", "f32", "f16s", "bf16s", "f64"])
    if lattice == "D2Q9":
        nx, ny, nz = _logint(rng, 24, 6000), _logint(rng, 24, 6000), 1
    else:
        side = _logint(rng, 16, 320)
        nx, ny, nz = (max(8, int(round(side * rng.uniform(0.6, 1.5)))) for _ in range(3))
    flow = rng.choice(["cavity", "cavity", "tg", "duct", "channel"])
    calls, steps = rng.choice([(1, 20), (1, 50), (1, 100), (1, 7), (5, 10), (10, 2), (20, 1)])
    # a pass of the largest draw stays below the largest listed case's work
    limit = 512 ** 3 * 20 * 38 * 4 / (8.0 if storage == "f64" else 2.0)
    while nx * ny * nz * steps * calls * 2.0 * Q[lattice] * BYTES[storage] > limit:
        if steps > 2:
            steps = max(2, steps // 2)
        else:
            nx, ny = max(8, nx // 2), max(8, ny // 2)
    return dict(kind="solver", lattice=lattice, nx=nx, ny=ny, nz=nz, flow=flow, storage=storage,
                tau=round(rng.uniform(0.55, 1.2), 3), steps=steps, calls=calls, fresh=rng.choice([0, 1]),
                monitor=rng.choice([0, 0, 1]))


# ------------------------------------------------------------------ flows
def _faces(flow, d):
    """(face kinds, wall velocities, body force direction) of a flow."""
    if flow == "cavity":
        faces = [1, 1, 1, 2, 1, 1] if d == 3 else [1, 1, 1, 2, 0, 0]
        return faces, [[0, 0, 0]] * 3 + [[LID, 0, 0]] + [[0, 0, 0]] * 2
    if flow == "duct":
        return ([0, 0, 1, 1, 1, 1] if d == 3 else [0, 0, 1, 1, 0, 0]), None
    if flow == "channel":
        return [0, 0, 1, 1, 0, 0], None
    return [0] * 6, None


def _force(case):
    if case["flow"] not in ("duct", "channel"):
        return (0.0, 0.0, 0.0)
    nu = (case["tau"] - 0.5) / 3.0
    # the force that gives the target centre-line speed of a square duct
    # (0.0737 F L^2 / nu) or of a plane channel (F L^2 / (8 nu))
    L = case["ny"]
    c = 0.0737 if case["flow"] == "duct" and case["nz"] > 1 else 0.125
    return (min(DUCT_U * nu / (c * L * L), 1e-3), 0.0, 0.0)


def _wave(n, k, phase):
    x = torch.arange(n, dtype=torch.float64, device="cuda")
    return torch.sin(2.0 * math.pi * k * x / n + phase)


def _modes(g, dims, count, amp):
    """A sum of `count` products of sines along the axes, of amplitude amp."""
    nx, ny, nz = dims
    out = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    for _ in range(count):
        k = g.integers(1, 4, size=3)
        p = g.uniform(0.0, 2.0 * math.pi, size=3)
        a = amp * g.uniform(0.5, 1.0) / count
        wz = _wave(nz, k[2], p[2]) if nz > 1 else torch.ones(1, dtype=torch.float64, device="cuda")
        out += (a * wz).view(nz, 1, 1) * (_wave(ny, k[1], p[1]).view(1, ny, 1) * _wave(nx, k[0], p[0]).view(1, 1, nx))
    return out.reshape(-1)


def _fields(case, seed):
    """Initial rho [N], u [d][N] of a single-component case (FP64, on the GPU):
    the flow's base state with seeded smooth disturbances."""
    g = np.random.Generator(np.random.PCG64([20230412, int(seed)]))
    dims = (case["nx"], case["ny"], case["nz"])
    nx, ny, nz = dims
    d = 2 if case["lattice"] == "D2Q9" else 3
    rho = 1.0 + _modes(g, dims, 2, 1e-3)
    u = torch.empty((d, nx * ny * nz), dtype=torch.float64, device="cuda")
    amp = 0.03 if case["flow"] == "tg" else 0.01
    for k in range(d):
        u[k] = _modes(g, dims, 3, amp)
    if case["flow"] in ("duct", "channel"):
        y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
        u[0].view(nz, ny, nx).add_((4.0 * 0.5 * DUCT_U * y * (1.0 - y)).view(1, ny, 1))
    return rho, u


# ------------------------------------------------------------------ prepare
def _member_cases(case):
    """The domains of a batch: sides, relaxation times and flows drawn from
    the case's own `mix` as the batch and serving workloads draw theirs."""
    g = np.random.Generator(np.random.PCG64(case["mix"]))
    out = []
    for i in range(case["members"]):
        two = case["lattice"].startswith("D2Q9") and i % 2 == 0
        lo, hi = (32, 1024) if two else (16, 128)
        L = int(round(math.exp(g.uniform(math.log(lo), math.log(hi)))))
        out.append(dict(lattice="D2Q9" if two else "D3Q19", nx=L, ny=L, nz=1 if two else L,
                        flow=("tg", "cavity", "duct")[int(g.integers(0, 3))], storage=case["storage"],
                        tau=round(float(g.uniform(0.55, 1.2)), 3)))
    return out


def _make_solver(case):
    from paper_2304_06437_gb300 import Solver
    d = 2 if case["lattice"] == "D2Q9" else 3
    faces, wall_u = _faces(case["flow"], d)
    return Solver(case["lattice"], (case["nx"], case["ny"], case["nz"]), case["tau"], faces=faces, wall_u=wall_u,
                  storage=case["storage"], force=_force(case))


def _drops(case, seed):
    """Seeded droplets (red) in a blue matrix: phi is the largest over the
    drops of tanh((R - r) / 2); returns rho_R, rho_B."""
    g = np.random.Generator(np.random.PCG64([20230412, int(seed)]))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    phi = torch.full((nz, ny, nx), -1.0, dtype=torch.float64, device="cuda")
    for _ in range(case["drops"]):
        R = g.uniform(case["rmin"], case["rmax"])
        idx, r2 = [], None
        for axis, n in enumerate((nz, ny, nx)):
            c = g.uniform(0, n)
            w = min(n, int(2 * (R + 8)) + 1) if n > 1 else 1
            i = np.arange(w) + int(c) - w // 2
            dist = np.zeros(1) if n == 1 else i - c
            idx.append(torch.from_numpy(np.mod(i, n) if n > 1 else np.zeros(1, dtype=np.int64)).cuda())
            shape = [1, 1, 1]
            shape[axis] = w
            t = torch.from_numpy(dist * dist).cuda().view(shape)
            r2 = t if r2 is None else r2 + t
        at = (idx[0].view(-1, 1, 1), idx[1].view(1, -1, 1), idx[2].view(1, 1, -1))
        phi[at] = torch.maximum(phi[at], torch.tanh(0.5 * (R - torch.sqrt(r2))))
    phi = phi.reshape(-1)
    return ((1.0 + phi) / 2.0).contiguous(), ((1.0 - phi) / 2.0).contiguous()


def prepare(case, seed):
    if case["kind"] == "cg":
        from paper_2304_06437_gb300 import CGSolver
        dims = (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])
        s = CGSolver(case["lattice"], dims, case["tau"], case["sigma"], case["beta"], storage=case["storage"])
        if case["nci"]:
            s.set_nci(0.01, 0.1, 2)
        rr, rb = _drops(case, seed)
        s.init(rr, rb)
        out = [torch.empty_like(rr), torch.empty_like(rb),
               torch.empty((s.d, s.n), dtype=torch.float64, device="cuda")]
        return dict(case=case, solver=s, out=out)
    if case["kind"] == "batch":
        from paper_2304_06437_gb300 import Batch
        doms = []
        for i, m in enumerate(_member_cases(case)):
            s = _make_solver(m)
            s.init_moments(*_fields(m, 1000 * int(seed) + i))
            s.reduce(residual=True)  # the residual's baseline, as the server takes it at admission
            doms.append(s)
        b = Batch(doms)
        # every member's rho and u, one after the other in one buffer, and
        # every member's populations in another
        fields = torch.empty(sum((1 + s.d) * s.n for s in doms), dtype=torch.float64, device="cuda")
        pops = torch.empty(sum(s.q * s.n for s in doms), dtype=torch.float64, device="cuda")
        views, at, ap = [], 0, 0
        for s in doms:
            views.append((fields[at:at + s.n], fields[at + s.n:at + (1 + s.d) * s.n].view(s.d, s.n),
                          pops[ap:ap + s.q * s.n].view(s.q, s.n)))
            at += (1 + s.d) * s.n
            ap += s.q * s.n
        return dict(case=case, batch=b, solvers=doms, fields=fields, pops=pops, views=views)
    s = _make_solver(case)
    rho0, u0 = _fields(case, seed)
    s.init_moments(rho0, u0)
    state = dict(case=case, solver=s, rho=torch.empty_like(rho0), u=torch.empty_like(u0),
                 f=torch.empty((s.q, s.n), dtype=torch.float64, device="cuda"))
    if case["fresh"]:
        state["init"] = (rho0, u0)
    if case["monitor"]:
        s.reduce(residual=True)
    return state


# ------------------------------------------------------------------ run
def run(state):
    case = state["case"]
    if case["kind"] == "cg":
        s = state["solver"]
        s.step(case["steps"])
        rr, rb, u = s.fields(*state["out"])
        return {"rho_r": rr, "rho_b": rb, "u": u}
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        sums = state["batch"].reduce(residual=True)
        for s, (rho, u, f) in zip(state["solvers"], state["views"]):
            s.moments(rho, u)
            s.get_populations(f)
        return {"fields": state["fields"], "populations": state["pops"],
                "sums": np.array([[r["mass"], *(r["momentum"] + [0.0])[:3], r["residual"]] for r in sums])}
    s = state["solver"]
    if case["fresh"]:
        s.init_moments(*state["init"])
    for _ in range(case["calls"]):
        s.step(case["steps"])
    out = {}
    if case["monitor"]:
        r = s.reduce(residual=True)
        out["sums"] = np.array([r["mass"], *r["momentum"], r["residual"]])
    s.moments(state["rho"], state["u"])
    out["rho"], out["u"] = state["rho"], state["u"]
    out["f"] = s.get_populations(state["f"])
    return out


# ------------------------------------------------------------------ work
def work(case):
    """Bytes and operations of one pass.  A step has to read and write the
    state once; a flow's state of second-order regularized collisions is its
    hydrodynamic moments (1 + d + d (d + 1) / 2 per node, one density more for
    two components) in the arithmetic precision, or its populations where
    those take fewer bytes; the outputs are written once.  Operations: the
    moment sums, the equilibrium and the projection, about 10 per population."""
    if case["kind"] == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for m in _member_cases(case):
            w = work(dict(m, kind="solver", steps=case["steps"], calls=1, fresh=0, monitor=1))
            for k in tot:
                tot[k] += w[k]
        return tot
    n = float(case["nx"] * case["ny"] * case["nz"])
    d = 2 if case["lattice"] == "D2Q9" else 3
    q = Q[case["lattice"]]
    es = BYTES[case["storage"]]
    rs = 8 if case["storage"] == "f64" else 4
    mom = 1 + d + d * (d + 1) // 2
    if case["kind"] == "cg":
        per_step = min(2 * 2 * q * es, 2 * (mom + 1) * rs)
        return {"bytes": n * (case["steps"] * per_step + 8 * (2 + d)), "flops": n * case["steps"] * 25.0 * q}
    per_step = min(2 * q * es, 2 * mom * rs)
    steps = case["steps"] * case["calls"]
    b = steps * per_step + 8 * (1 + d) + 8 * q
    if case["fresh"]:
        b += 8 * (1 + d)
    if case["monitor"]:
        b += 2 * 4 * d
    return {"bytes": n * b, "flops": n * steps * 10.0 * q}


# ------------------------------------------------------------------ exact
def _velocities(lattice):
    """Velocities in the library's order (rest, |c|^2, lexicographic) and weights."""
    d = 2 if lattice == "D2Q9" else 3
    cmax = {"D2Q9": 2, "D3Q19": 2, "D3Q27": 3}[lattice]
    r = (-1, 0, 1)
    c = [(x, y, z) for x in r for y in r for z in (r if d == 3 else (0,)) if x * x + y * y + z * z <= cmax]
    c.sort(key=lambda v: (v[0] ** 2 + v[1] ** 2 + v[2] ** 2, v))
    w = {"D2Q9": (4 / 9, 1 / 9, 1 / 36), "D3Q19": (1 / 3, 1 / 18, 1 / 36),
         "D3Q27": (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[lattice]
    return c, [w[x * x + y * y + z * z] for x, y, z in c]


def _dot(v, c):
    """sum_k c_k v_k over the non-zero components of c (None if there is none)."""
    out = None
    for k, ck in enumerate(c):
        if ck:
            t = v[k] if ck > 0 else -v[k]
            out = t if out is None else out + t
    return out


class _Reference:
    """The regularized step in plain FP64 torch: deviations f_a - t_a (rho0 = 1)
    of each population on a (z, y, x) grid, collided in place of two arrays."""

    def __init__(self, lattice, dims, tau, faces, wall_u, force):
        self.c, self.w = _velocities(lattice)
        self.q, self.d = len(self.c), 2 if lattice == "D2Q9" else 3
        self.dims, self.om = dims, 1.0 / tau
        self.faces, self.wall_u, self.F = faces, wall_u, force
        self.forced = any(force)
        self.opp = [self.c.index((-x, -y, -z)) for x, y, z in self.c]

    def grid(self, a):
        nx, ny, nz = self.dims
        return a.view(nz, ny, nx)

    def project(self, a, A, B, C):
        """w_a [A + B.c + c.C.c], C[(i, j)] for i <= j, off-diagonals doubled."""
        c, out = self.c[a], A.clone()
        for i in range(self.d):
            if c[i]:
                out.add_(B[i], alpha=c[i])
                for j in range(i, self.d):
                    if c[j]:
                        out.add_(C[(i, j)], alpha=c[i] * c[j])
        return out.mul_(self.w[a])

    def init(self, rho, u):
        r = self.grid(rho) - 1.0
        u = [self.grid(u[k]) for k in range(self.d)]
        A = r - 1.5 * sum(v * v for v in u)
        B = [3.0 * u[k] - 1.5 * self.F[k] for k in range(self.d)]
        C = {(i, j): (4.5 if i == j else 9.0) * u[i] * u[j] for i in range(self.d) for j in range(i, self.d)}
        return [self.project(a, A, B, C) for a in range(self.q)]

    def moments(self, f):
        r = f[0].clone()
        j = [torch.zeros_like(r) for _ in range(self.d)]
        for a in range(1, self.q):
            r += f[a]
            for k in range(self.d):
                if self.c[a][k]:
                    j[k].add_(f[a], alpha=self.c[a][k])
        for k in range(self.d):
            if self.F[k]:
                j[k] += 0.5 * self.F[k]
        return r, j  # rho - 1 and u

    def coefficients(self, f, F=None):
        d, om = self.d, self.om
        F = F if F is not None else (self.F if self.forced else None)
        r, u = self.moments(f)
        P = {}
        for i in range(d):
            for j in range(i, d):
                p = None
                for a in range(1, self.q):
                    cc = self.c[a][i] * self.c[a][j]
                    if cc:
                        p = f[a] * cc if p is None else p.add_(f[a], alpha=cc)
                p -= u[i] * u[j]
                if i == j:
                    p.sub_(r, alpha=1.0 / 3.0)
                P[(i, j)] = p
        g = 1.0 - 0.5 * om
        A = r - 1.5 * sum(v * v for v in u) - 1.5 * (1.0 - om) * sum(P[(k, k)] for k in range(d))
        if F is not None:
            A -= 3.0 * g * sum(u[k] * F[k] for k in range(d))
        B = [3.0 * u[k] + (1.5 * F[k] if F is not None else 0.0) for k in range(d)]
        C = {}
        for (i, j), p in P.items():
            t = u[i] * u[j] + (1.0 - om) * p
            if F is not None:
                t += g * (u[i] * F[j] + u[j] * F[i])
            C[(i, j)] = t.mul_(4.5 if i == j else 9.0)
        return A, B, C

    def stream(self, post):
        """Pull streaming with halfway bounce-back of the post-collision set."""
        out = []
        for a, c in enumerate(self.c):
            shift, dims = [], []
            for k in range(3):
                if c[k]:
                    shift.append(c[k])
                    dims.append(2 - k)
            t = torch.roll(post[a], shift, dims) if shift else post[a].clone()
            out.append(t)
        for a, c in enumerate(self.c):
            walls = [2 * k + (0 if c[k] > 0 else 1) for k in range(self.d)
                     if c[k] and self.faces[2 * k + (0 if c[k] > 0 else 1)] != 0]
            for sub in range(1, 1 << len(walls)):
                crossed = [walls[i] for i in range(len(walls)) if sub >> i & 1]
                term = 0.0
                if all(self.faces[f] == 2 for f in crossed):
                    uw = self.wall_u[crossed[0]]
                    term = 6.0 * self.w[a] * sum(c[k] * uw[k] for k in range(3))
                # nodes on all of these faces; the masks ascend, so a set of faces
                # comes after every set it contains and decides the corner
                idx = [slice(None)] * 3
                for f in crossed:
                    ax = 2 - f // 2
                    n = out[a].shape[ax]
                    idx[ax] = slice(0, 1) if f % 2 == 0 else slice(n - 1, n)
                out[a][tuple(idx)] = post[self.opp[a]][tuple(idx)] + term
        return out

    def step(self, f):
        A, B, C = self.coefficients(f)
        return self.stream([self.project(a, A, B, C) for a in range(self.q)])


def _exact_solver(case, seed, steps):
    d = 2 if case["lattice"] == "D2Q9" else 3
    faces, wall_u = _faces(case["flow"], d)
    ref = _Reference(case["lattice"], (case["nx"], case["ny"], case["nz"]), case["tau"], faces, wall_u, _force(case))
    f = ref.init(*_fields(case, seed))
    _, u0 = ref.moments(f)
    for _ in range(steps):
        f = ref.step(f)
    r, u = ref.moments(f)
    u = torch.stack([v.reshape(-1) for v in u])
    u0 = torch.stack([v.reshape(-1) for v in u0])
    return ref, f, r.reshape(-1), u, u0


def _exact_sums(ref, r, u, u0):
    n = r.numel()
    mom = [float((u[k] - 0.5 * ref.F[k]).sum()) for k in range(ref.d)]
    return [n + float(r.sum()), *mom, float((u - u0).norm() / u.norm())]


def _populations(ref, f):
    full = torch.empty((ref.q, f[0].numel()), dtype=torch.float64, device="cuda")
    for a in range(ref.q):
        full[a] = f[a].reshape(-1) + ref.w[a]
        f[a] = None
    return full


def exact(case, seed):
    if case["kind"] == "cg":
        return None if case["nci"] else _exact_cg(case, seed)
    if case["kind"] == "batch":
        members = _member_cases(case)
        if sum(m["nx"] * m["ny"] * m["nz"] for m in members) * case["steps"] > 3e9:
            return None
        fields, pops, sums = [], [], []
        for i, m in enumerate(members):
            ref, f, r, u, u0 = _exact_solver(m, 1000 * int(seed) + i, case["steps"])
            fields += [r + 1.0, u.reshape(-1)]
            pops.append(_populations(ref, f).reshape(-1))
            s = _exact_sums(ref, r, u, u0)
            sums.append([s[0], *(s[1:1 + ref.d] + [0.0])[:3], s[-1]])
        return {"fields": torch.cat(fields), "populations": torch.cat(pops), "sums": np.array(sums)}
    steps = case["steps"] * case["calls"]
    if case["nx"] * case["ny"] * case["nz"] * steps * Q[case["lattice"]] > 6e10:
        return None
    ref, f, r, u, u0 = _exact_solver(case, seed, steps)
    out = {"rho": r + 1.0, "u": u}
    if case["monitor"]:
        # a fresh pass sets the state from outside, which restarts the residual
        s = _exact_sums(ref, r, u, u0)
        out["sums"] = np.array(s[:-1] + ([1.0] if case["fresh"] else s[-1:]))
    out["f"] = _populations(ref, f)
    return out


def _exact_cg(case, seed):
    dims = (case["nx"], case["ny"], case["nz"])
    if dims[0] * dims[1] * dims[2] * case["steps"] > 1.5e9:
        return None
    ref = _Reference(case["lattice"], dims, case["tau"], [0] * 6, None, (0.0, 0.0, 0.0))
    rr, rb = (ref.grid(v) for v in _drops(case, seed))
    d, q, w = ref.d, ref.q, ref.w
    shell = [sum(x * x for x in c) for c in ref.c]
    Bw = ((-4 / 27, 2 / 27, 5 / 108) if d == 2 else (-2 / 9, 1 / 54, 1 / 27))
    # each colour as deviations from half the rest population, at rest
    fr = [w[a] * (rr - 0.5) for a in range(q)]
    fb = [w[a] * (rb - 0.5) for a in range(q)]
    pk = 2.25 * case["sigma"] * ref.om
    for _ in range(case["steps"]):
        A, B, C = ref.coefficients([fr[a] + fb[a] for a in range(q)])
        rr, rb = sum(fr) + 0.5, sum(fb) + 0.5
        rho = rr + rb
        phi, cr, crb = (rr - rb) / rho, rr / rho, case["beta"] * rr * rb / rho
        grad = [torch.zeros_like(phi) for _ in range(d)]
        for a, c in enumerate(ref.c):
            shift = [(-c[k], 2 - k) for k in range(3) if c[k]]
            if not shift:
                continue
            p = torch.roll(phi, [s for s, _ in shift], [ax for _, ax in shift])
            for k in range(d):
                if c[k]:
                    grad[k].add_(p, alpha=3.0 * w[a] * c[k])
        gn = torch.sqrt(sum(v * v for v in grad))
        n = [torch.where(gn > 0, v / torch.where(gn > 0, gn, torch.ones_like(gn)), torch.zeros_like(gn)) for v in grad]
        pr, pb = [], []
        for a, c in enumerate(ref.c):
            cn = _dot(n, c)
            cn = torch.zeros_like(gn) if cn is None else cn
            g = ref.project(a, A, B, C) + w[a] + pk * gn * (w[a] * cn * cn - Bw[shell[a]])
            red = cr * g
            if shell[a]:
                red = red + crb * (w[a] / math.sqrt(shell[a])) * cn
            pr.append(red - 0.5 * w[a])
            pb.append(g - red - 0.5 * w[a])
        fr, fb = ref.stream(pr), ref.stream(pb)
    rr, rb = sum(fr) + 0.5, sum(fb) + 0.5
    _, u = ref.moments([fr[a] + fb[a] for a in range(q)])
    return {"rho_r": rr.reshape(-1), "rho_b": rb.reshape(-1), "u": torch.stack([v.reshape(-1) for v in u])}
