"""Measured cases: what a user of the framework has it do, through its public entry points.

A pass of a single-domain case advances one resident domain by ``steps`` time
steps, reads the force / torque series of those steps (every form, FP64) and
the density and velocity fields -- the loop of a user's program between two
field outputs.  A domain goes on from where the last pass left it.  Bodies with
prescribed translation turn back at the start of each pass (an update of their
kinematics), so they stay on the collision-free stretch they were placed for.
A pass of the serving case takes a set of requests through a resident batch:
admission, the steps of every request, reading each series, release.

Sizes are those of ``paper_1407_4524_gb300.workloads`` (the framework's own
configurations) and ragged ones of the same kinds.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1407_4524_gb300 import lbm, workloads

BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}
# operations of a node's step (moments, equilibrium, relaxation) in the plain formulas
FLOPS = {"D2Q9": 110, "D3Q19": 260}
SIZES_2D = workloads.SERVING_D2Q9_SIZES
SIZES_3D = workloads.SERVING_D3Q19_SIZES


def listed():
    return [
        # drag and lift of a cylinder in a small channel at full precision: few cells, every step waits for the last
        dict(name="channel_2d_fp64", kind="channel_2d", precision="fp64", nx=200, ny=80, nz=1, steps=1002),
        # translating and rotating cylinders: geometry, covered and uncovered nodes every step, still a small domain
        dict(name="moving_2d_fp32", kind="moving_2d", precision="fp32", nx=512, ny=256, nz=1, steps=1002),
        # a sedimenting disc between Zou-He walls, moved by the flow, at full precision (the paper's own test)
        dict(name="disc_2d_fp64", kind="disc_2d", precision="fp64", nx=135, ny=1073, nz=1, steps=402),
        # flow past a sphere (inlet, outlet) in each precision mode: single, half storage, and the FP64 comparison run
        dict(name="channel_3d_fp32", kind="channel_3d", precision="fp32", nx=256, ny=128, nz=128, steps=642),
        dict(name="channel_3d_fp16", kind="channel_3d", precision="fp16", nx=256, ny=128, nz=128, steps=642),
        dict(name="channel_3d_fp64", kind="channel_3d", precision="fp64", nx=256, ny=128, nz=128, steps=130),
        # walled duct driven by a body force, ragged sizes
        dict(name="duct_3d_fp32", kind="duct_3d", precision="fp32", nx=93, ny=61, nz=57, steps=802),
        # a few spheres, half of them moving, on an odd ragged grid; then many of them: the largest domains
        dict(name="swarm_3d_ragged_fp32", kind="swarm_3d", precision="fp32", nx=151, ny=97, nz=84, bodies=4, steps=802),
        dict(name="swarm_3d_fp32", kind="swarm_3d", precision="fp32", nx=512, ny=256, nz=256, bodies=64, steps=602),
        dict(name="swarm_3d_fp16", kind="swarm_3d", precision="fp16", nx=512, ny=256, nz=256, bodies=64, steps=602),
        # continuous batching of uneven requests, half-precision storage
        dict(name="serving_16_fp16", kind="serving", precision="fp16", requests=16, slots=16, shift=0, steps=2000),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["channel_2d", "moving_2d", "disc_2d", "channel_3d", "duct_3d", "swarm_3d", "serving"])
    # (flows that start at rest and stay slow are solved in the modes that resolve them)
    precision = rng.choice(["fp64", "fp32"] if kind in ("disc_2d", "duct_3d") else ["fp64", "fp32", "fp16"])
    if kind == "serving":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp16"]), requests=rng.randint(3, 24),
                    slots=rng.choice([8, 16, 40]), shift=rng.randint(0, 27), steps=rng.randint(1200, 1600))
    c = dict(kind=kind, precision=precision)
    if kind == "channel_2d":
        c.update(nx=log(96, 2048), ny=log(48, 1024), nz=1)
    elif kind == "moving_2d":
        c.update(nx=log(128, 1200), ny=log(96, 900), nz=1)
    elif kind == "disc_2d":
        c.update(nx=rng.randint(90, 202), ny=rng.randint(500, 1300), nz=1)
    elif kind == "channel_3d":
        c.update(nx=log(56, 320), ny=log(32, 160), nz=log(32, 160))
    elif kind == "duct_3d":
        c.update(nx=log(40, 160), ny=log(32, 120), nz=log(32, 120))
    else:
        c.update(nx=log(72, 512), ny=log(64, 256), nz=log(64, 256))
        c["bodies"] = max(2, min(64, c["nx"] * c["ny"] * c["nz"] // 400000))
    cells = c["nx"] * c["ny"] * c["nz"]
    c["steps"] = max(18, min(1002, int((2e8 if precision == "fp64" else 2e9) / cells)))
    return c


# ------------------------------------------------------------------- inputs --


def _spec(case, seed):
    """The problem dict of a single-domain case: the sizes are the case's, the body and the flow the seed's."""
    rng = np.random.default_rng(seed)
    kind, n = case["kind"], (case["nx"], case["ny"], case["nz"])
    jit = rng.uniform(-0.5, 0.5, 3)
    speed = float(rng.uniform(0.9, 1.1))
    if kind == "channel_2d":
        R = min(8.0, 0.1 * n[1] + 0.2)
        return dict(lattice="D2Q9", n=n[:2], tau=0.8, precision=case["precision"],
                    edges={"x": ("inlet", "outlet"), "y": ("wall", "wall")},
                    inlet={"profile": "parabolic", "u": 0.05 * speed},
                    bodies=[dict(shape="cylinder", R=R, X0=(min(40.0, 0.2 * n[0]) + jit[0], 0.5 * n[1] + jit[1]))])
    if kind == "moving_2d":
        s = min(1.0, n[1] / 128.0)
        return dict(lattice="D2Q9", n=n[:2], tau=0.6, precision=case["precision"],
                    bodies=[dict(shape="cylinder", R=12.0 * s, X0=(0.25 * n[0] + jit[0], 0.25 * n[1] + jit[1]),
                                 U=(0.02 * speed, 0.0)),
                            dict(shape="cylinder", R=10.0 * s, X0=(0.75 * n[0] + jit[2], 0.75 * n[1]), W=0.002 * speed)])
    if kind == "disc_2d":  # workloads.sedimenting_disc_2d, released at rest higher or lower by the seed
        return dict(lattice="D2Q9", n=n[:2], tau=0.6, precision=case["precision"], edge_rule="zouhe",
                    edges={"x": ("wall", "wall"), "y": ("wall", "wall")},
                    gravity=(0.0, -2.9e-4 * (134.0 / (n[0] - 1)) ** 3),
                    bodies=[dict(shape="cylinder", R=(n[0] - 1) / 8.0, free=True, density_ratio=1.01,
                                 X0=(0.69 * (n[0] - 1) + jit[0], 0.78 * (n[1] - 1) + 8 * jit[1]))])
    if kind == "channel_3d":
        u = 0.04 * speed
        R = min(12.0, 0.094 * min(2 * n[0], 4 * n[1], 4 * n[2]) / 2)
        return dict(lattice="D3Q19", n=n, tau=0.55, precision=case["precision"], edges={"x": ("inlet", "outlet")},
                    inlet={"profile": "uniform", "u": u}, u0=(u, 0.0, 0.0),
                    bodies=[dict(shape="sphere", R=R, X0=tuple(0.25 * n[0] if a == 0 else 0.5 * n[a]
                                                               for a in range(3)) + jit)])
    if kind == "duct_3d":
        return dict(lattice="D3Q19", n=n, tau=0.8, precision=case["precision"], force=(1e-5 * speed, 0.0, 0.0),
                    edges={"y": ("wall", "wall"), "z": ("wall", "wall")},
                    bodies=[dict(shape="sphere", R=0.15 * min(n), X0=tuple(0.5 * v for v in n) + jit)])
    return workloads.sphere_swarm_3d(precision=case["precision"], n=n, n_bodies=case["bodies"], seed=seed)


def _requests(case, seed):
    """Requests as workloads.serving_request draws them, sizes and steps by the request's number."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["requests"]):
        q = k + case["shift"]
        flat = q % 2 == 0
        n = SIZES_2D[(q // 2) % 4] if flat else SIZES_3D[(q // 2) % 3]
        while True:
            r = workloads.serving_request(rng, lattice="D2Q9" if flat else "D3Q19", precision=case["precision"])
            if tuple(r["n"]) == tuple(n):
                break
        out.append(dict(r, steps=case["steps"] - (q * 37) % (case["steps"] // 2)))
    return out


def prepare(case, seed):
    if case["kind"] == "serving":
        return {"requests": _requests(case, seed), "batch": lbm.Batch(64 << 30, max_slots=case["slots"])}
    spec = _spec(case, seed)
    return {"domain": lbm.Domain(spec), "bodies": spec["bodies"], "steps": case["steps"],
            "turning": case["kind"] == "swarm_3d"}


def run(state):
    if "batch" in state:
        return _serve(state["batch"], state["requests"])
    dom, first = state["domain"], state["domain"].t
    if state["turning"]:
        sign = -1.0 if first else 1.0
        state["bodies"] = [dict(b, X0=tuple(x + (first - b.get("t0", 0)) * u for x, u in zip(b["X0"], b["U"])),
                                U=tuple(sign * u for u in b["U"]), W=tuple(sign * w for w in b["W"]), t0=first)
                           for b in state["bodies"]]
        dom.update_bodies(state["bodies"])
    dom.step(state["steps"])
    return {"series": dom.series(first, state["steps"]), "fields": dom.macros()}


def _serve(batch, requests):
    waiting = list(range(len(requests)))
    resident, out = {}, {}
    while waiting or resident:
        while waiting:
            slot = batch.admit(requests[waiting[0]])
            if slot is None:
                break
            resident[slot] = waiting.pop(0)
        batch.run()
        for slot in batch.poll():
            out["request_%02d" % resident.pop(slot)] = batch.force_torque(slot)
            batch.release(slot)
    return out


def work(case):
    """Every population of a cell read and written once a step, the series and the fields written once a pass."""
    if case["kind"] == "serving":
        each = [(r["lattice"], workloads.cells(r), r["steps"], 0) for r in _requests(case, 0)]
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        each = [("D2Q9" if case["nz"] == 1 else "D3Q19", cells, case["steps"], 32 * cells)]
    q = {"D2Q9": 9, "D3Q19": 19}
    return {"bytes": float(sum(2 * q[lat] * BYTES[case["precision"]] * c * s + more for lat, c, s, more in each)),
            "flops": float(sum(FLOPS[lat] * c * s for lat, c, s, _ in each))}


# -------------------------------------------------------- results in 64 bits --


def exact(case, seed):
    if case["kind"] == "serving":  # the first two requests: all of them would take a minute
        reqs = _requests(case, seed)
        return {"request_%02d" % k: _Solver(r).advance(r["steps"])[:, :, :6] if k < 2 else None
                for k, r in enumerate(reqs)}
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["steps"] * (6e-3 + 1.8e-9 * cells) > 20.0:  # seconds, as measured
        return None
    s = _Solver(_spec(case, seed))
    series = s.advance(case["steps"])
    return {"series": series, "fields": s.fields()}


class _Solver:
    """The method (quasi-incompressible BGK, curved-wall links, momentum exchange, prescribed and free bodies, half-way
    or, in 2-D closed boxes, Zou-He faces) on dense torch arrays in 64 bits, post-collision f of shape [Q, nz, ny, nx]."""

    def __init__(self, spec):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.n = tuple(spec["n"]) + (1,) * (3 - len(spec["n"]))
        self.flat = spec["lattice"] == "D2Q9"
        self.tau, self.zouhe = float(spec["tau"]), spec.get("edge_rule") == "zouhe"
        self.g = self._vec((tuple(spec.get("force") or ()) + (0.0,) * 3)[:3])
        self.forced = spec.get("force") is not None
        top = (3, 3, 1) if self.flat else (3, 3, 3)
        cs = [c for c in itertools.product((0, 1, -1), repeat=3) if sum(map(abs, c)) < 3 and (c[2] == 0 or top[2] > 1)]
        self.c = cs
        self.Q = len(cs)
        rest = {9: (4 / 9, 1 / 9, 1 / 36), 19: (1 / 3, 1 / 18, 1 / 36)}[self.Q]
        self.w = [rest[sum(map(abs, c))] for c in cs]
        self.opp = [cs.index(tuple(-v for v in c)) for c in cs]
        self.cT, self.wT = torch.tensor(cs, dtype=torch.int64, device=self.dev), self._vec(self.w)
        self.oppT = torch.tensor(self.opp, device=self.dev)
        self.cF = self.cT.double()
        self.shape = self.n[::-1]
        edges = spec.get("edges", {})
        self.edge = [(edges.get(a, "periodic"),) * 2 if isinstance(edges.get(a, "periodic"), str) else edges[a] for a in "xyz"]
        self.inlet = spec.get("inlet", {})
        self._faces()
        self.f = torch.empty((self.Q,) + self.shape, dtype=torch.float64, device=self.dev)
        u0 = self._vec((tuple(spec.get("u0", ())) + (0.0,) * 3)[:3])
        for i in range(self.Q):
            self.f[i] = self._feq_of(torch.ones((), dtype=torch.float64, device=self.dev), u0[:, None], i)[0]
        self._collide(self.f)
        self.t = 0
        self._place(spec)

    def _vec(self, v):
        return torch.tensor(v, dtype=torch.float64, device=self.dev)

    # ---- fluid ----
    def _feq_of(self, rho, u, i):
        cu = sum(k * u[a] for a, k in enumerate(self.c[i]))
        return self.w[i] * (rho + 3.0 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def _moments(self, f, sign):
        """rho and u; `sign` +1 for streamed, -1 for collided populations (the body force adds g to them)."""
        rho, u = f.sum(0), []
        for a in range(3):
            j = torch.zeros_like(rho)
            for i, c in enumerate(self.c):
                if c[a]:
                    j += c[a] * f[i]
            u.append(j + sign * 0.5 * self.g[a])
        return rho, torch.stack(u)

    def _collide(self, f):
        om = 1.0 / self.tau
        rho, u = self._moments(f, 1.0)
        usq = 1.5 * (u * u).sum(0)
        for i, c in enumerate(self.c):
            cu = sum((k * u[a] for a, k in enumerate(c) if k), torch.zeros_like(rho))
            new = (1.0 - om) * f[i] + om * self.w[i] * (rho + 3.0 * cu + 4.5 * cu * cu - usq)
            if self.forced:
                cg, ug = (self.cF[i] * self.g).sum(), (u * self.g.view(3, *([1] * rho.dim()))).sum(0)
                new += (1.0 - 0.5 * om) * self.w[i] * (3.0 * (cg - ug) + 9.0 * cu * cg)
            f[i] = new

    def _index(self, p):
        return (p[2] * self.n[1] + p[1]) * self.n[0] + p[0]

    def _wrap(self, p):
        return torch.stack([p[a] % self.n[a] for a in range(3)])

    def _faces(self):
        """Per direction: cells whose pull bounces at a face (with 6 w c.u_B) and cells that take the outlet's last column."""
        self.face, self.zh = [], []
        hard = [[e in ("wall", "inlet") for e in self.edge[a]] for a in range(3)]
        ax = [torch.arange(v, device=self.dev) for v in self.n]
        on = torch.zeros(self.shape, dtype=torch.bool, device=self.dev)
        for a in range(3):
            if self.edge[a][0] != "periodic":
                sl = [slice(None)] * 3
                for end in (0, -1):
                    sl[2 - a] = end
                    on[tuple(sl)] = True
        z, y, x = torch.nonzero(on, as_tuple=True)
        cells = torch.stack([x, y, z])
        for i, c in enumerate(self.c):
            s = cells - self.cT[i][:, None]
            wall = torch.zeros(cells.shape[1], dtype=torch.bool, device=self.dev)
            inl, out = wall.clone(), wall.clone()
            for a in range(3):
                for end, beyond in ((0, s[a] < 0), (1, s[a] >= self.n[a])):
                    kind = self.edge[a][end]
                    wall |= beyond & (kind == "wall")
                    inl |= beyond & (kind == "inlet")
                    out |= beyond & (kind == "outlet")
                    if kind == "outlet":
                        s[a] = torch.where(beyond, torch.full_like(s[a], self.n[a] - 1), s[a])
            bounce = wall | inl
            uB = torch.zeros(cells.shape[1], dtype=torch.float64, device=self.dev)
            u = float(self.inlet.get("u", 0.0))
            if self.inlet.get("profile", "uniform") == "parabolic":
                ny = float(self.n[1])
                yb = cells[1].double() - 0.5 * c[1]
                uB += torch.where(inl & ~wall, 4.0 * u * (yb + 0.5) * (ny - 0.5 - yb) / ny ** 2, uB)
            else:
                uB += (inl & ~wall).double() * u
            keep = out & ~bounce
            self.face.append((self._index(cells[:, bounce]), 6.0 * self.w[i] * c[0] * uB[bounce],
                              self._index(cells[:, keep]), self._index(self._wrap(s[:, keep]))))
        if self.zouhe:  # 2-D closed box: (cells, normal axis, side) of the faces, (cell, inner neighbour) of the corners
            assert self.flat and all(all(h) for h in hard[:2])
            nx, ny = self.n[0], self.n[1]
            for a, end in itertools.product((0, 1), (0, 1)):
                along = ax[1 - a][1:-1]
                fixed = torch.full_like(along, 0 if end == 0 else self.n[a] - 1)
                p = (fixed, along) if a == 0 else (along, fixed)
                self.zh.append((p[1] * nx + p[0], a, -1 if end == 0 else 1))
            self.corners = [(y * nx + x, (y + (1 if y == 0 else -1)) * nx + x + (1 if x == 0 else -1),
                             1 if x == 0 else -1, 1 if y == 0 else -1) for x in (0, nx - 1) for y in (0, ny - 1)]

    def _zouhe(self, old, new):
        for cells, a, side in self.zh:
            f = new[:, cells]
            along = sum(c[1 - a] * f[i] for i, c in enumerate(self.c) if c[a] == 0) * 0.5
            for i, c in enumerate(self.c):
                if c[a] * side < 0:
                    new[i][cells] = f[self.opp[i]] - c[1 - a] * along
        for cell, inner, sx, sy in self.corners:
            unknown = [c[0] == sx or c[1] == sy for c in self.c]
            buried = [u and unknown[o] for u, o in zip(unknown, self.opp)]
            f = new[:, cell].clone()
            for i in range(self.Q):
                if unknown[i] and not buried[i]:
                    f[i] = new[self.opp[i], cell]
            share = (old[:, inner].sum() - sum(f[i] for i in range(self.Q) if not buried[i])) / sum(buried)
            for i in range(self.Q):
                new[i, cell] = share if buried[i] else f[i]

    # ---- bodies ----
    def _place(self, spec):
        b = spec["bodies"]
        three = lambda v: (tuple(v) + (0.0,) * 3)[:3]  # noqa: E731
        spin = lambda v: (0.0, 0.0, float(v)) if np.isscalar(v) else tuple(v)  # noqa: E731
        self.R = self._vec([k["R"] for k in b])
        self.X, self.U = self._vec([three(k["X0"]) for k in b]), self._vec([three(k.get("U", ())) for k in b])
        self.W = self._vec([spin(k.get("W", 0.0)) for k in b])
        self.X0 = self.X.clone()
        self.free = any(k.get("free") for k in b)
        self.moving = self.free or bool((self.U != 0).any() or (self.W != 0).any())
        if self.free:
            self.gravity, self.ratio = self._vec(three(spec["gravity"])), float(b[0]["density_ratio"])
        k = int(math.ceil(float(self.R.max()))) + 4
        r = torch.arange(-k, k + 2, device=self.dev)
        z = torch.zeros(1, dtype=torch.int64, device=self.dev) if self.flat else r
        self.box = torch.stack(torch.meshgrid(r, r, z, indexing="ij")).reshape(3, -1)
        self.own, self.links = self._geometry(self.X)

    def _around(self, X):
        """Cells near each body, their displacement from its centre and the body's number."""
        base = torch.floor(X).long()
        if self.flat:
            base[:, 2] = 0
        p = base.T[:, :, None] + self.box[:, None, :]
        d = p.double() - X.T[:, :, None]
        if self.flat:
            d[2] = 0.0
        dist = (d * d).sum(0).sqrt()
        near = dist <= self.R[:, None] + 2.0
        body = torch.arange(len(self.R), device=self.dev)[:, None].expand_as(dist)[near]
        return p[:, near], d[:, near], (dist <= self.R[:, None])[near], body

    def _geometry(self, X):
        p, d, inside, body = self._around(X)
        cell = self._index(self._wrap(p))
        own = torch.full((math.prod(self.n),), -1, dtype=torch.int32, device=self.dev)
        own[cell[inside]] = body[inside].int()
        keep = own[cell] < 0
        p, d, cell, body = p[:, keep], d[:, keep], cell[keep], body[keep]
        got = []
        for i in range(1, self.Q):
            A = self._index(self._wrap(p - self.cT[i][:, None]))
            m = own[A] == body
            got.append((cell[m], torch.full_like(cell[m], i), d[:, m], body[m],
                        self._index(self._wrap(p + self.cT[i][:, None]))[m]))
        F, i, d, b, G = (torch.cat(v, -1) for v in zip(*got))
        c = self.cF[i].T
        a, bb, cc = (c * c).sum(0), (d * c).sum(0), (d * d).sum(0) - self.R[b] ** 2
        s = (cc / (bb + (bb * bb - a * cc).clamp_min(0.0).sqrt())).clamp(0.0, 1.0)
        return own, (F, i, d, b, G, s)

    def _at(self, f, cells):
        return self._moments(f.reshape(self.Q, -1)[:, cells], -1.0)

    def _per_body(self, v, body, out):
        out.index_add_(0, body, v.T)

    def _wall(self):
        """Wall value of every cut link, and the link sums of the row: static force, torque, moving frame."""
        F, i, d, b, G, s = self.links
        c = self.cF[i].T
        f = self.f.reshape(self.Q, -1)
        fb = f[self.oppT[i], F]
        rho, uF = self._at(self.f, F)
        _, uG = self._at(self.f, G)
        uB = self.U[b].T + torch.linalg.cross(self.W[b].T, d - s * c, dim=0)
        low, lone = s < 0.5, self.own[G] >= 0
        ubf = torch.where(low, torch.where(lone, uF, uG), uF + 1.5 / s.clamp_min(0.25) * (uB - uF))
        chi = torch.where(low, torch.where(lone, 0.0, (2.0 * s - 1.0) / (self.tau - 2.0)), (2.0 * s - 1.0) / (self.tau + 0.5))
        w = self.wT[i]
        g = w * (rho - 3.0 * (c * ubf).sum(0) + 4.5 * (c * uF).sum(0) ** 2 - 1.5 * (uF * uF).sum(0))
        fa = (1.0 - chi) * fb + chi * g + 6.0 * w * (c * uB).sum(0)
        ps = -c * (fa + fb)
        pm = ps + uB * (fa - fb)
        row = torch.zeros((len(self.R), 18), dtype=torch.float64, device=self.dev)
        for at, v in ((0, ps), (3, torch.linalg.cross(d, ps, dim=0)), (12, pm), (15, torch.linalg.cross(d, pm, dim=0))):
            self._per_body(v, b, row[:, at:at + 3])
        return fa, row

    def _displace(self, new, X1, row):
        """Covered and uncovered nodes between t and t+1: impulsive terms into `row`, refill into `new`."""
        own1, links1 = self._geometry(X1)
        nf = new.reshape(self.Q, -1)
        at = torch.nonzero(own1 != self.own).squeeze(1)
        for gone in (False, True):
            cell = at[(self.own[at] >= 0) == gone]
            b = (self.own if gone else own1)[cell].long()
            p = torch.stack([cell % self.n[0], cell // self.n[0] % self.n[1], cell // (self.n[0] * self.n[1])])
            half = self._vec(self.n)[:, None]
            image = lambda X: (lambda v: v - half * torch.floor(v / half + 0.5))(p.double() - X[b].T)  # noqa: E731
            r, r1 = image(self.X), image(X1)
            if self.flat:
                r[2] = r1[2] = 0.0
            if gone:
                q = self._wrap(p[:, None, :] + self.cT[1:].T[:, :, None])
                q = self._index(q.reshape(3, -1))
                ok = (self.own[q] < 0).double()
                rho = (self._at(self.f, q)[0] * ok).reshape(self.Q - 1, -1).sum(0)
                cnt = ok.reshape(self.Q - 1, -1).sum(0)
                rho = torch.where(cnt > 0, rho / cnt.clamp_min(1.0), torch.ones_like(rho))
                u = self.U[b].T + torch.linalg.cross(self.W[b].T, r1, dim=0)
                for i in range(self.Q):
                    nf[i][cell] = self._feq_of(rho, u, i)
            m = self.cF.T @ nf[:, cell] * (-1.0 if gone else 1.0)
            self._per_body(m, b, row[:, 6:9])
            self._per_body(torch.linalg.cross(r, m, dim=0), b, row[:, 9:12])
        return own1, links1

    def advance(self, steps):
        rows = []
        for _ in range(steps):
            fa, row = self._wall()
            new = torch.empty_like(self.f)
            for i, c in enumerate(self.c):
                new[i] = torch.roll(self.f[i], (c[2], c[1], c[0]), (0, 1, 2))
                bounce, add, keep, src = self.face[i]
                o, nf = self.f.reshape(self.Q, -1), new[i].reshape(-1)
                if len(bounce):
                    nf[bounce] = o[self.opp[i]][bounce] + add
                if len(keep):
                    nf[keep] = o[i][src]
            F, i = self.links[0], self.links[1]
            new.reshape(self.Q, -1)[i, F] = fa
            if self.zouhe:
                self._zouhe(self.f.reshape(self.Q, -1), new.reshape(self.Q, -1))
            if self.moving:
                X1 = self.X + self.U if self.free else self.X0 + (self.t + 1) * self.U
                geometry = self._displace(new, X1, row)
                if self.free:
                    V = math.pi * float(self.R[0]) ** 2
                    M = self.ratio * V
                    self.U = self.U + (row[:, 0:3] + row[:, 6:9] + (self.ratio - 1.0) * V * self.gravity) / M
                    self.W[:, 2] += (row[:, 5] + row[:, 11]) / (0.5 * M * float(self.R[0]) ** 2)
                self.X, (self.own, self.links) = X1, geometry
            self._collide(new)
            self.f = new
            self.t += 1
            rows.append(row)
        return torch.stack(rows).cpu().numpy()

    def fields(self):
        rho, u = self._moments(self.f, -1.0)
        out = torch.cat([rho[None], u])
        out.reshape(4, -1)[:, self.own >= 0] = 0.0
        return out.cpu().numpy()
