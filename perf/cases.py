"""Performance cases of the library: what its users run, through the Python
binding of the C ABI (``lbib.Simulation``, ``lbib.Ensemble``, ``lbib_adjoint_*``).

A pass of a simulation advances it by ``steps`` time steps and takes the state
back as a program does between two outputs: populations into a device tensor,
marker positions and bonds to the host.  A pass of the adjoint records
``steps`` time steps, sweeps back and reads every gradient.  The simulation
goes on from pass to pass, as in a long run.

``exact`` is the same computation written out in plain torch, FP64, from the
method's equations (Coclite, arXiv 1907.00080); gradients by torch.autograd.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1907_00080_gb300 import inputs, lbib

PREC = ("f64", "f32", "f16", "bf16")
STORED_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


def listed():
    return [
        # the smallest call: one FP64 step of the capsule in a 128 x 32 channel, read back
        # after each step (set-up, debugging, coupling to other code): latency and launches
        {"name": "capsule_f64_1", "kind": "capsule", "prec": "f64", "steps": 1},
        # the production run of one coarse capillary between two outputs (the lattice stays in L2)
        {"name": "capillary_f32", "kind": "capillary", "nx": 640, "ny": 160, "prec": "f32",
         "carriers": "kinematic", "steps": 100},
        # the same in FP64, the reference precision of every error that users state
        {"name": "capillary_f64", "kind": "capillary", "nx": 640, "ny": 160, "prec": "f64",
         "carriers": "kinematic", "steps": 48},
        # a capillary of other, ragged sizes (odd NX: no vector loads), read back often
        {"name": "capillary_odd_f32", "kind": "capillary", "nx": 403, "ny": 121, "prec": "f32",
         "carriers": "kinematic", "steps": 7},
        # the cell-free layer study: Couette walls, one rigid dynamic carrier near the wall
        {"name": "couette_dynamic_f32", "kind": "couette", "carrier": "rigid", "carriers": "dynamic",
         "prec": "f32", "steps": 64},
        # the fine mesh: free carriers in 16-bit storage, carriers adhering to the walls in FP32
        {"name": "fine_f16", "kind": "fine", "carrier": "rigid", "release": "free", "prec": "f16", "steps": 50},
        {"name": "fine_f32", "kind": "fine", "carrier": "soft", "release": "wall", "prec": "f32", "steps": 50},
        # the parameter sweep: 64 capillaries of different lengths in the tuned shape
        {"name": "ensemble64_f32", "kind": "ensemble", "members": 64, "prec": "f32", "vec": 2, "ty": 0, "steps": 64},
        # a small sweep in 16-bit storage, in the default shape
        {"name": "ensemble10_bf16", "kind": "ensemble", "members": 10, "prec": "bf16", "vec": 4, "ty": 1, "steps": 48},
        # the lattice alone on an odd size with Zou-He walls (no bulk copies: rows are not 16-byte multiples)
        {"name": "lattice_odd_f32", "kind": "lattice", "nx": 1501, "ny": 333, "prec": "f32", "walls": 2, "steps": 40},
        # a lattice far beyond L2 with dilute carriers: HBM-bound, the largest
        {"name": "probe_f32", "kind": "probe", "nx": 8192, "ny": 2048, "prec": "f32", "steps": 32},
        # the sensitivity study: recorded run and backward sweep
        {"name": "adjoint_f64", "kind": "adjoint", "prec": "f64", "steps": 60, "every": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["capsule", "capillary", "capillary", "couette", "fine", "ensemble", "lattice", "probe",
                       "adjoint"])
    prec = rng.choice(PREC)
    # the scaled FP16 storage overflows where bonds or random starts move the populations by
    # more than a few times the flow itself: such studies take BF16
    if prec == "f16" and kind in ("couette", "lattice"):
        prec = "bf16"
    c = {"kind": kind, "prec": prec}
    even = 2 if prec in ("f16", "bf16") else 1
    if kind == "capsule":
        c["steps"] = _log(rng, 1, 100)
    elif kind == "capillary":
        c.update(nx=_log(rng, 300, 1500) // even * even, ny=rng.randint(100, 260),
                 carriers=rng.choice(["kinematic", "kinematic", "dynamic"]), steps=_log(rng, 1, 60))
    elif kind == "couette":
        c.update(carrier=rng.choice(["rigid", "soft"]), carriers=rng.choice(["kinematic", "dynamic"]),
                 steps=_log(rng, 1, 100))
    elif kind == "fine":
        c.update(carrier=rng.choice(["rigid", "soft"]), release="free" if prec == "f16" else rng.choice(["free", "wall"]),
                 steps=_log(rng, 4, 40))
    elif kind == "ensemble":
        c.update(members=_log(rng, 2, 64), steps=_log(rng, 4, 40))
        c["vec"], c["ty"] = rng.choice({"f64": [(2, 1), (1, 2)], "f32": [(2, 0), (1, 0), (4, 1), (2, 2)],
                                        "f16": [(2, 0), (4, 0), (4, 2), (8, 1)],
                                        "bf16": [(2, 0), (4, 0), (4, 2), (8, 1)]}[prec])
    elif kind == "lattice":
        c.update(nx=max(4, _log(rng, 8, 4096)) // even * even, ny=_log(rng, 8, 1024), walls=rng.randint(0, 2),
                 steps=_log(rng, 1, 100))
    elif kind == "probe":
        c.update(prec=rng.choice(["f32", "f16", "bf16"]), nx=_log(rng, 2000, 8000) // 2 * 2,
                 ny=_log(rng, 600, 2000), steps=rng.randint(4, 24))
    else:
        c.update(prec=rng.choice(["f64", "f64", "f32"]), steps=rng.randint(10, 60), every=rng.randint(5, 60))
    return c


# ------------------------------------------------------------------ inputs
def _workloads(case, seed):
    """the synthetic set-ups of a case (one, or an ensemble's members)"""
    kind, prec, seed = case["kind"], case["prec"], int(seed) % (1 << 31)
    if kind == "capsule":
        wl = inputs.capsule_128x32(prec, bonds="stress")
        # released at a random place near the lower wall, which carries the receptors
        rng = np.random.default_rng(seed)
        wl.membranes[0].xy = wl.membranes[0].xy + [rng.uniform(-20.0, 60.0), rng.uniform(0.0, 1.0)]
        wl.seed = seed
        return [wl]
    if kind == "capillary":
        nx, ny = case["nx"], case["ny"]
        return [inputs.capillary(nx=nx, ny=ny, n_rbc=max(1, round(8 * nx / 640 * 160 / ny)), rbc_alpha=0.4 * ny,
                                 rbc_markers=round(1.25 * ny), carrier_radius=0.05 * ny,
                                 carrier_markers=round(0.3125 * ny), seed=seed, precision=prec,
                                 carrier_model=case["carriers"])]
    if kind == "couette":
        return [inputs.couette_cfl_600x200(prec, carrier=case["carrier"], carrier_model=case["carriers"], seed=seed)]
    if kind == "fine":
        make = inputs.fine_capillary_adhering if case["release"] == "wall" else inputs.fine_capillary_2000x667
        return [make(prec, carriers=case["carrier"], seed=seed)]
    if kind == "ensemble":
        return _sweep(case["members"], prec, seed)
    if kind == "lattice":
        # a developing channel flow (or a decaying one between periodic rows)
        ny = case["ny"]
        g = inputs.body_force_for(inputs.u_max_for_re(1.0, ny), ny) if case["walls"] else 0.0
        return [inputs.Workload("lattice", case["nx"], ny, body_force=(g, 0.0), walls=case["walls"], init="rest",
                                precision=prec, wall_velocity=(0.0, 0.01) if case["walls"] else (0.0, 0.0))]
    if kind == "probe":
        wl = inputs.probe_lattice(case["nx"], case["ny"], prec)
        # each carrier at a random place of its own cell of a grid, so that no two overlap
        rng, n = np.random.default_rng(seed), len(wl.membranes)
        cols = math.ceil(math.sqrt(n * wl.nx / wl.ny))
        dx, dy = wl.nx / cols, wl.ny / math.ceil(n / cols)
        for k, m in enumerate(wl.membranes):
            m.xy = inputs.circle(dx * (k % cols) + rng.uniform(12, dx - 12), dy * (k // cols) + rng.uniform(12, dy - 12),
                                 8.0, 50)
        return [wl]
    wl = inputs.adjoint_capillary_320x160(seed=seed, precision=prec, bonds="stress")
    return [wl]


@functools.lru_cache(maxsize=None)
def _layouts(prec):
    return inputs.capillary_ensemble(8, seed=0, precision=prec)


def _sweep(members, prec, seed):
    """an ensemble as inputs.capillary_ensemble makes it (64 members of 512-1008 x 160), from a few of its
    layouts, which are slow to place: each member one of them, moved along x in a channel of its own length"""
    rng, out = np.random.default_rng(seed), []
    for i in range(members):
        wl = _layouts(prec)[i % 8]
        shift, nx = rng.uniform(0, wl.nx), min(wl.nx + 8 * (7 * i % 24), max(wl.nx, 1008))
        out.append(dataclasses.replace(wl, nx=nx, seed=seed + i, receptors=inputs.wall_receptors(nx, wl.ny),
                                       membranes=[dataclasses.replace(m, xy=m.xy + [shift, 0.0])
                                                  for m in wl.membranes]))
    return out


def _start(wl, seed, device):
    """random initial populations of a lattice without membranes: the rest state,
    perturbed by 1 %, (9, ny, nx) on the device"""
    gen = torch.Generator(device=device).manual_seed(int(seed))
    r = torch.rand((9, wl.ny, wl.nx), generator=gen, device=device, dtype=torch.float64)
    return _W.to(device)[:, None, None] * (1.0 + 0.01 * (2.0 * r - 1.0))


def _bars(nv, seed):
    """adjoint seed: weights of the final marker positions in the objective"""
    return np.random.default_rng(int(seed) + 1).standard_normal((nv, 2))


class _State:
    """a prepared case; frees the library's objects with itself"""

    def __init__(self):
        self.ens = self.sim = self.adj = None

    def __del__(self):
        if self.adj is not None:
            lbib.lbib_adjoint_destroy(self.adj)
        for owner in (self.ens, self.sim):
            if owner is not None:
                owner.close()


def prepare(case, seed):
    lbib.load()
    s = _State()
    s.case = case
    s.wls = _workloads(case, seed)
    if case["kind"] == "ensemble":
        s.ens = lbib.Ensemble(s.wls, tiling=(case["vec"], case["ty"]))
        s.xy = np.zeros((sum(wl.n_vertices for wl in s.wls), 2))
        s.views = np.split(s.xy, np.cumsum([wl.n_vertices for wl in s.wls])[:-1])
        s.f = torch.empty(sum(9 * wl.nx * wl.ny for wl in s.wls), dtype=torch.float64, device="cuda")
        return s
    wl = s.wls[0]
    s.sim = lbib.Simulation(wl)
    if case["kind"] == "adjoint":
        s.adj = lbib.lbib_adjoint_create(s.sim.ctx, case["every"])
        s.bars = _bars(wl.n_vertices, seed)
        return s
    s.f = torch.empty((9, wl.ny, wl.nx), dtype=torch.float64, device="cuda")
    if case["kind"] == "lattice":
        f0 = _start(wl, seed, "cuda")
        torch.cuda.synchronize()
        lbib.lbib_write_populations(s.sim.ctx, f0.data_ptr(), on_device=1)
    return s


def run(state):
    s, n = state, state.case["steps"]
    if s.ens is not None:
        s.ens.step(n)
        s.ens.sync()
        at = 0
        for m in s.ens.members:
            lbib.lbib_read_populations(m.ctx, s.f.data_ptr() + 8 * at, on_device=1)
            at += 9 * m.nx * m.ny
        s.ens.read_markers(s.views)
        return {"f": s.f, "xy": s.xy, "bonds": np.concatenate([m.bonds() for m in s.ens.members])}
    if s.adj is not None:
        lbib.lbib_adjoint_record(s.sim.ctx, s.adj, n)
        lbib.lbib_adjoint_seed(s.sim.ctx, s.adj, s.bars)
        lbib.lbib_adjoint_reverse(s.sim.ctx, s.adj)
        out = lbib.lbib_adjoint_read(s.sim.ctx, s.adj, s.sim.nv, len(s.wls[0].membranes))
        return {k: out[k] for k in ("xy", "xy_prev", "k_s", "k_b", "sigma")}
    s.sim.step(n)
    lbib.lbib_read_populations(s.sim.ctx, s.f.data_ptr(), on_device=1)
    return {"f": s.f, "xy": s.sim.markers(), "bonds": s.sim.bonds()}


def work(case):
    """Per time step, every population read and written once in its storage type;
    per marker its two positions read and written; the state read back once.
    The adjoint reads the state and the adjoint populations of a step and writes
    the latter, and needs the state again (a second forward step or its tape)."""
    wls = _workloads(case, 0) if case["kind"] != "adjoint" else [inputs.adjoint_capillary_320x160()]
    nodes = sum(wl.nx * wl.ny for wl in wls)
    markers = sum(wl.n_vertices for wl in wls)
    e = STORED_BYTES[case["prec"]]
    n = case["steps"]
    if case["kind"] == "adjoint":
        return {"bytes": float(n * (2 * (18 * e * nodes + 64 * markers) + (18 * 8 + 9 * e) * nodes)),
                "flops": float(n * (2 * 130 + 260) * nodes)}
    return {"bytes": float(n * (18 * e * nodes + 64 * markers) + (9 * (8 + e)) * nodes + 16 * markers),
            "flops": float(n * (130 * nodes + 500 * markers))}


# ------------------------------------------------------------------ exact
_E = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_W = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64)


def _roma(r):
    a = r.abs()
    near = (1 + torch.sqrt(1 - 3 * a.clamp(max=0.5) ** 2)) / 3
    b = 1 - a.clamp(min=0.5, max=1.5)
    far = (2 + 3 * b - torch.sqrt(1 - 3 * b * b)) / 6
    return torch.where(a <= 0.5, near, torch.where(a <= 1.5, far, torch.zeros_like(a)))


def _uniform(step, lig, rec, tag, seed, instance):
    """Philox4x64-10 (Salmon et al. 2011), the top 53 bits of its first word"""
    m64 = (1 << 64) - 1
    c = [step, lig, rec, tag]
    k0, k1 = seed & m64, instance & m64
    for _ in range(10):
        p0, p1 = 0xD2E7470EE14C6C93 * c[0], 0xCA5A826395121157 * c[2]
        c = [(p1 >> 64) ^ c[1] ^ k0, p1 & m64, (p0 >> 64) ^ c[3] ^ k1, p0 & m64]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & m64, (k1 + 0xBB67AE8584CAA73B) & m64
    return (c[0] >> 11) * 2.0 ** -53


class _Plain:
    """one simulation in FP64 torch operations"""

    def __init__(self, wl, device):
        self.wl, self.dev = wl, device
        self.t = t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=device)
        self.long = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.int64, device=device)
        self.ex, self.ey, self.w9 = t(_E[:, 0]), t(_E[:, 1]), _W.to(device)
        self.n = 0
        mems = wl.membranes
        sizes = [len(m.xy) for m in mems]
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(int)
        self.rings = [slice(off[k], off[k + 1]) for k in range(len(mems))]
        ring = lambda d: self.long(np.concatenate([o + (np.arange(k) + d) % k for o, k in zip(off, sizes)] or [[]]))
        self.L, self.R = ring(-1), ring(1)
        self.mem = self.long(np.repeat(np.arange(len(mems)), sizes))
        self.ks, self.kb = t([m.ks for m in mems]), t([m.kb for m in mems])
        self.ka, self.sigma = t([m.ka for m in mems]), t(wl.sigma_lu)
        self.X = t(np.concatenate([m.xy for m in mems]) if mems else np.zeros((0, 2)))
        self.Xp = self.X
        self.rest_len, self.rest_angle, self.rest_area = self._geometry(self.X)[:3]
        self.lig_a = self.long(np.concatenate([off[k] + m.ligands for k, m in enumerate(mems)] or [[]]))
        self.rec = t(wl.receptors) if wl.receptors is not None and len(wl.receptors) else None
        self.bond = -np.ones(wl.n_ligands, dtype=np.int32)
        self.owner = -np.ones(0 if self.rec is None else len(self.rec), dtype=np.int32)
        # dynamic particles: vertex velocity, rigid state (u, v, omega and the step before), mass, moment
        self.V = torch.zeros_like(self.X)
        self.rigid = {k: (np.zeros(3), np.zeros(3)) for k, m in enumerate(mems) if m.kind == 3}
        self.dyn = {k: m.rho_p * np.array(self._polygon(self.X[self.rings[k]])[:2])
                    for k, m in enumerate(mems) if m.kind >= 2}
        nu, y = (wl.tau - 0.5) / 3, torch.arange(wl.ny, dtype=torch.float64, device=device)
        if wl.init == "poiseuille":
            gx = wl.body_force[0]
            u = gx / (2 * nu) * (y + 0.5) * (wl.ny - 0.5 - y) + 0.25 * gx
        else:
            gx, (ub, ut) = 0.0, wl.wall_velocity
            u = (ub + (ut - ub) * (y + 0.5) / wl.ny) if wl.init == "couette" else torch.zeros_like(y)
        u = u[:, None].expand(wl.ny, wl.nx)
        if wl.init == "rest":
            self.f = self.w9[:, None, None].expand(9, wl.ny, wl.nx).contiguous()
        else:
            post = self._equilibrium(1.0, u, 0 * u) + self._source(u, 0 * u, gx + 0 * u, 0 * u)
            self.f = self._stream(post)

    # ---- lattice
    def _equilibrium(self, rho, u, v):
        eu = self.ex[:, None, None] * u + self.ey[:, None, None] * v
        return self.w9[:, None, None] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u + v * v))

    def _source(self, u, v, gx, gy):
        ex, ey = self.ex[:, None, None], self.ey[:, None, None]
        eu = ex * u + ey * v
        s = (3 * (ex - u) + 9 * eu * ex) * gx + (3 * (ey - v) + 9 * eu * ey) * gy
        return (1 - 0.5 / self.wl.tau) * self.w9[:, None, None] * s

    def _stream(self, post):
        rows = []
        for i, (cx, cy) in enumerate(_E):
            p = torch.roll(post[i], (int(cy), int(cx)), (0, 1))
            if self.wl.walls and cy:
                y, u_wall = (0, self.wl.wall_velocity[0]) if cy > 0 else (self.wl.ny - 1, self.wl.wall_velocity[1])
                back = post[_OPP[i]][y] + 6 * float(_W[i]) * float(cx) * u_wall
                p = torch.cat([back[None], p[1:]]) if cy > 0 else torch.cat([p[:-1], back[None]])
            rows.append(p)
        f = torch.stack(rows)
        return self._zou_he(f, 0.0, 0.0) if self.wl.walls == 2 else f

    def _zou_he(self, f, gx, gy):
        """wall rows y = 0, NY - 1 at the wall velocity: j = rho (u_w, 0) - G / 2"""
        f = f.clone()
        for y, s, (n, a, b), uw in ((0, 1, (2, 5, 6), self.wl.wall_velocity[0]),
                                    (self.wl.ny - 1, -1, (4, 7, 8), self.wl.wall_velocity[1])):
            gxy = [g[y] if torch.is_tensor(g) else g for g in (gx, gy)]
            jn = -0.5 * s * gxy[1]
            r = f[:, y]
            rho = r[0] + r[1] + r[3] + 2 * (r[_OPP[n]] + r[_OPP[a]] + r[_OPP[b]]) + jn
            shift = 0.5 * (r[1] - r[3]) - 0.5 * (rho * uw - 0.5 * gxy[0])
            f[n, y] = r[_OPP[n]] + 2 / 3 * jn
            f[a, y] = r[_OPP[a]] - s * shift + jn / 6
            f[b, y] = r[_OPP[b]] + s * shift + jn / 6
        return f

    def _moments(self, f, gx, gy):
        rho = f.sum(0)
        jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
        jy = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7])
        return rho, (jx + 0.5 * gx) / rho, (jy + 0.5 * gy) / rho

    # ---- membranes
    def _geometry(self, X):
        """per vertex: length of its element, turning angle; per membrane: area; per vertex: normal, edge shares"""
        if not len(X):
            z = X[:, 0]
            return z, z, self.ks, X, z
        eL, eR = X - X[self.L], X[self.R] - X
        lL, lR = eL.norm(dim=1), eR.norm(dim=1)
        angle = torch.atan2(eL[:, 0] * eR[:, 1] - eL[:, 1] * eR[:, 0], (eL * eR).sum(1))
        nrm = torch.stack([eL[:, 1] / lL + eR[:, 1] / lR, -eL[:, 0] / lL - eR[:, 0] / lR], 1)
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        first = X[self.long([r.start for r in self.rings])][self.mem]
        a, b = X - first, X[self.R] - first
        cross = 0.5 * (a[:, 0] * b[:, 1] - b[:, 0] * a[:, 1])
        area = torch.zeros_like(self.ks).index_add(0, self.mem, cross)
        return lR, angle, area, nrm, lL / (lL + lR)

    def _polygon(self, X):
        """area, polar moment about the area centroid, centroid of a ring"""
        a = X - X[0]
        b = torch.roll(a, -1, 0)
        c = a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]
        g = (c[:, None] * (a + b)).sum(0) / (3 * c.sum())
        j = (c * ((a * a).sum(1) + (a * b).sum(1) + (b * b).sum(1))).sum() / 12 - 0.5 * c.sum() * (g * g).sum()
        return float(0.5 * c.sum()), float(j), X[0] + g

    def _image(self, d):
        per = [float(self.wl.nx), float(self.wl.ny) if not self.wl.walls else math.inf]
        return torch.stack([d[..., k] - (per[k] * torch.floor(d[..., k].detach() / per[k] + 0.5)
                                         if per[k] < math.inf else 0.0) for k in (0, 1)], -1)

    def _forces(self, X):
        lR, angle, area, nrm, sL = self._geometry(X)
        F = torch.zeros_like(X)
        eR = X[self.R] - X
        pull = (self.ks[self.mem] * (lR - self.rest_len) / lR)[:, None] * eR
        F = F + pull - pull[self.L]
        m = (self.kb[self.mem] * (angle - self.rest_angle))[:, None] * nrm
        F = F - m + (m * sL[:, None])[self.R] + (m * (1 - sL)[:, None])[self.L]
        c = (-self.ka * (1 - area / self.rest_area) / 3)[self.mem]
        push = 0.5 * c[:, None] * torch.stack([-eR[:, 1], eR[:, 0]], 1)
        F = F + push + push[self.L]
        if len(self.rings) > 1 and self.wl.d_rep > 0:
            for k, ring in enumerate(self.rings):  # Eq. repFor, along each vertex's own inward normal
                with torch.no_grad():
                    d2 = (self._image(X[ring][:, None] - X[None]) ** 2).sum(-1)
                    close = (d2 < self.wl.d_rep ** 2) & (self.mem[None] != k)
                    i, j = close.nonzero(as_tuple=True)
                d = self._image(X[ring][i] - X[j]).norm(dim=1)
                mag = torch.zeros_like(X[ring][:, 0]).index_add(0, i, 1e-4 / (8 * math.sqrt(2.0)) * d ** -2.5)
                F = F.index_add(0, torch.arange(ring.start, ring.stop, device=self.dev), -mag[:, None] * nrm[ring])
        held = np.nonzero(self.bond >= 0)[0]
        if len(held):
            a = self.lig_a[self.long(held)]
            d = self._image(self.rec[self.long(self.bond[held])] - 0.5 * (X[a] + X[self.R[a]]))
            dist = d.norm(dim=1, keepdim=True)
            half = 0.5 * self.sigma * (dist - self.wl.bonds["y_eq"]) / dist * d
            F = F.index_add(0, a, half).index_add(0, self.R[a], half)
        return F

    def _fit(self, q):
        """moving least squares over the 3 x 3 nearest fluid nodes: the rows (value, d/dx, d/dy) and the node indices"""
        nx, ny = self.wl.nx, self.wl.ny
        o = torch.floor(q.detach() + 0.5)
        k = torch.arange(-1, 2, device=self.dev, dtype=torch.float64)
        rx, ry = o[:, :1] + k - q[:, :1], o[:, 1:] + k - q[:, 1:]
        jj = (o[:, 1:] + k).long()
        inside = ((jj >= 0) & (jj < ny)) if self.wl.walls else torch.ones_like(jj, dtype=torch.bool)
        w = (torch.where(inside, _roma(ry), torch.zeros_like(ry))[:, :, None] * _roma(rx)[:, None]).reshape(-1, 9)
        p = torch.stack([torch.ones_like(w), rx[:, None].expand(-1, 3, 3).reshape(-1, 9),
                         ry[:, :, None].expand(-1, 3, 3).reshape(-1, 9)], 1)
        A = (w[:, None] * p) @ p.transpose(1, 2)
        thin = (inside.sum(1) < 2)[:, None, None]  # one row or none: the normalised weights, no gradient
        phi = w[:, None] * torch.linalg.solve(torch.where(thin, torch.eye(3, device=self.dev, dtype=w.dtype), A), p)
        mean = torch.stack([w / w.sum(1, keepdim=True).clamp(min=1e-300), 0 * w, 0 * w], 1)
        phi = torch.where(thin, mean, phi)
        full = inside.all(1)[:, None]
        value = torch.where(full, w, phi[:, 0])  # exact on a full stencil
        ii = (o[:, :1] + k).long().remainder(nx)
        idx = (jj.clamp(0, ny - 1) if self.wl.walls else jj.remainder(ny))[:, :, None] * nx + ii[:, None]
        return value, phi, idx.reshape(-1, 9)

    def _hydro(self, k, w, idx, flow):
        """Eqs. hydroForP, hydroForNu on the vertices of dynamic ring k, and its forcing term on the fluid"""
        r = self.rings[k]
        X, nu = self.X[r], (self.wl.tau - 0.5) / 3
        e = torch.roll(X, -1, 0) - X
        ln = e.norm(dim=1, keepdim=True)
        nrm = torch.stack([e[:, 1], -e[:, 0]], 1) / ln
        _, phi, at = self._fit(X + 0.5 * e + 1.2 * nrm)
        g = phi @ flow[at]  # rows value, d/dx, d/dy of (p, u, v)
        p, ux, uy, vx, vy = g[:, 0, 0], g[:, 1, 1], g[:, 2, 1], g[:, 1, 2], g[:, 2, 2]
        t = torch.stack([(2 * nu * ux - p) * nrm[:, 0] + nu * (uy + vx) * nrm[:, 1],
                         nu * (uy + vx) * nrm[:, 0] + (2 * nu * vy - p) * nrm[:, 1]], 1) * ln
        H = 0.5 * (t + torch.roll(t, 1, 0))
        U = (w[r][:, None] @ flow[idx[r]])[:, 0, 1:]
        return H, (ln + torch.roll(ln, 1, 0)) * (self.V[r] - U)

    def _advance(self, k, m, F, U):
        """new positions of ring k; (X^n - X^{n-1}) is kept for the second-order forms"""
        r = self.rings[k]
        X, Xp, U = self.X[r], self.Xp[r], U[r]
        first = self.n == 0
        if m.kind == 2:
            new = X + U + 0.5 * F[r] / (self.dyn[k][0] / len(X))
            self.V[r] = (new - X) if first else 1.5 * (new - X) - 0.5 * (X - Xp)
            return new
        if m.kind == 3:
            mass, inertia = self.dyn[k]
            d = X - self._polygon(X)[2]
            acc = np.array([float(F[r][:, 0].sum()) / mass, float(F[r][:, 1].sum()) / mass,
                            float((d[:, 0] * F[r][:, 1] - d[:, 1] * F[r][:, 0]).sum()) / inertia])
            now, before = self.rigid[k]
            new = now + acc if first else (2.0 * now - 0.5 * before + acc) * (2 / 3)
            self.rigid[k] = (new, now)
            u, v, om = new
            c1, sn = -2 * math.sin(0.5 * om) ** 2, math.sin(om)
            turn = torch.stack([c1 * d[:, 0] - sn * d[:, 1], sn * d[:, 0] + c1 * d[:, 1]], 1)
            at = d + turn
            self.V[r] = torch.stack([u - om * at[:, 1], v + om * at[:, 0]], 1)
            return X + turn + self.t([u, v])
        if m.kind == 1:
            d, du = X - X.mean(0), U - U.mean(0)
            om = (d[:, 0] * du[:, 1] - d[:, 1] * du[:, 0]).sum() / (d * d).sum()
            U = U.mean(0) + om * torch.stack([-d[:, 1], d[:, 0]], 1)
        return X + U if first else (2 * X - 0.5 * Xp + U) * (2 / 3)

    def _bonds(self):
        """rupture, then formation, at the new positions"""
        b, wl = self.wl.bonds, self.wl
        X = self.X.detach()
        c = 0.5 * (X[self.lig_a] + X[self.R[self.lig_a]])
        dist = self._image(self.rec[None] - c[:, None]).norm(dim=2)
        was_free = self.owner < 0

        def prob(d, k, beta):
            return 1 - math.exp(-k * math.exp(beta * ((d - b["y_eq"]) / b["y_eq"]) ** 2))

        held = np.nonzero(self.bond >= 0)[0]
        at = dist[self.long(held), self.long(self.bond[held])].tolist()
        for lig, d in zip(held.tolist(), at):
            rec = int(self.bond[lig])
            if d >= b["d_break"] or _uniform(self.n, lig, rec, 1, wl.seed, wl.instance) < prob(d, b["kr0_dt"], b["beta_r"]):
                self.bond[lig] = self.owner[rec] = -1
        tried, claimed = set(), set()
        pairs = (dist < b["d_cut"]).nonzero()
        at = dist[pairs[:, 0], pairs[:, 1]].tolist()
        for (lig, rec), d in zip(pairs.tolist(), at):
            if lig in tried or self.bond[lig] >= 0 or not was_free[rec]:
                continue
            if _uniform(self.n, lig, rec, 0, wl.seed, wl.instance) < prob(d, b["kf_dt"], -b["beta_f"]):
                tried.add(lig)
                if rec not in claimed:
                    claimed.add(rec)
                    self.bond[lig], self.owner[rec] = rec, lig

    def step(self):
        wl, f = self.wl, self.f
        gx, gy = (torch.full_like(f[0], g) for g in wl.body_force)
        if len(self.X):
            F = self._forces(self.X)
            w, _, idx = self._fit(self.X)
            spread = F
            if self.dyn:
                rho, u, v = self._moments(f, *wl.body_force)
                flow = torch.stack([(rho - 1) / 3, u, v], -1).reshape(-1, 3)
                F, spread = F.clone(), F.clone()
                for k in self.dyn:
                    H, D = self._hydro(k, w, idx, flow)
                    F[self.rings[k]] += H
                    spread[self.rings[k]] = D
            gx, gy = (g.reshape(-1).index_add(0, idx.reshape(-1), (w * spread[:, k:k + 1]).reshape(-1)).reshape(g.shape)
                      for k, g in enumerate((gx, gy)))
        if wl.walls == 2:
            f = self._zou_he(f, gx, gy)
        rho, u, v = self._moments(f, gx, gy)
        post = f - (f - self._equilibrium(rho, u, v)) / wl.tau + self._source(u, v, gx, gy)
        self.f = self._stream(post)
        if len(self.X):
            U = torch.stack([(w * c.reshape(-1)[idx]).sum(1) for c in (u, v)], 1)
            new = torch.cat([self._advance(k, m, F, U) for k, m in enumerate(wl.membranes)])
            self.Xp, self.X = self.X, new
            if self.rec is not None and len(self.bond):
                self._bonds()
        self.n += 1


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    wls, n = _workloads(case, seed), case["steps"]
    if case["kind"] == "adjoint":
        return _exact_adjoint(wls[0], case, seed, device)
    sims = []
    with torch.no_grad():
        for wl in wls:
            s = _Plain(wl, device)
            if case["kind"] == "lattice":
                s.f = _start(wl, seed, device)
            for _ in range(n):
                s.step()
            sims.append(s)
    if case["kind"] != "ensemble":
        return {"f": sims[0].f, "xy": sims[0].X.cpu().numpy(), "bonds": sims[0].bond}
    return {"f": torch.cat([s.f.reshape(-1) for s in sims]),
            "xy": np.concatenate([s.X.cpu().numpy() for s in sims]), "bonds": np.concatenate([s.bond for s in sims])}


def _exact_adjoint(wl, case, seed, device):
    wl = dataclasses.replace(wl, precision="f64")
    s = _Plain(wl, device)
    leaves = [s.X.clone(), s.X.clone(), s.ks, s.kb, s.sigma]
    for x in leaves:
        x.requires_grad_(True)
    s.X, s.Xp, s.ks, s.kb, s.sigma = leaves
    for _ in range(case["steps"]):
        s.step()
    (s.X * s.t(_bars(wl.n_vertices, seed))).sum().backward()
    xy, xy_prev, k_s, k_b, sigma = (torch.zeros_like(x) if x.grad is None else x.grad for x in leaves)
    return {"xy": xy.cpu().numpy(), "xy_prev": xy_prev.cpu().numpy(), "k_s": k_s.cpu().numpy(),
            "k_b": k_b.cpu().numpy(), "sigma": float(sigma)}
