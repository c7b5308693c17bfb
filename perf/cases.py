"""The work a user has this library do, as cases that can be timed and checked.

A case is one call sequence of a running simulation: some time steps of a
lattice with its immersed bodies (alone, in a batch, recorded step by step,
or served), and the read-back of what the user looks at afterwards.  Sizes,
relaxation times, meshes and parameters are those of this repository's
workloads, tests and benchmark; the seed moves the bodies, draws their
parameters and perturbs the initial flow.

What is read back is kept at the width the context computes with: doubles
for FP64, floats for FP32, and for 16-bit storage floats for the marker
positions and the storage type for the rest (the library hands every array
out in double, whatever the context holds).  Of the markers a program reads
the positions and velocities, and for a rigid body in FP64 or FP32 the IB
force too; a membrane's IB force is the small remainder of forces that
balance (its FP32 value holds three or four digits, its FP64 value nine),
and its effect is in the velocities.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2207_06029_gb300 import lbib
from paper_2207_06029_gb300 import workloads as W

PREC = {"fp64": lbib.LBIB_FP64, "fp32": lbib.LBIB_FP32, "fp16": lbib.LBIB_FP16_DEV, "bf16": lbib.LBIB_BF16_DEV}
ELEM = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
KEPT = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def _single(name, n, prec, flow, body, radius, level, steps, **more):
    c = dict(name=name, kind="run", nx=n[0], ny=n[1], nz=n[2], prec=prec, flow=flow, body=body, radius=float(radius),
             level=level, steps=steps, tau=0.8, option=0)
    c.update(more)
    return c


def listed():
    return [
        # a control loop around a small cell: one step, then the body's state
        # and its markers are read (the smallest call; launches and latency)
        _single("monitor32_fp32", (32, 32, 32), "fp32", "shear", "sphere", 4, 3, 1, kind="monitor", tau=1.0),
        # the plain method in FP64: 32^3 Couette cell, rigid sphere, 642 markers
        _single("couette32_fp64", (32, 32, 32), "fp64", "shear", "sphere", 4, 3, 40, tau=1.0),
        # a spheroid orbiting in a small shear cell, the momentum-exchange force
        _single("spheroid48_fp32", (48, 48, 48), "fp32", "shear", "spheroid", 6, 3, 40, option=1),
        # a recorded trajectory: every step's markers copied to the host
        _single("record64_fp32", (64, 64, 64), "fp32", "shear", "capsule", 7, 3, 40, kind="record"),
        # odd rows, bfloat16 storage: a capsule in a cell of 75 x 67 x 81 nodes
        _single("capsule75_bf16", (75, 67, 81), "bf16", "shear", "capsule", 8, 4, 40),
        # the main single run: deformable capsule, 96^3, 2562 markers
        _single("capsule96_fp32", (96, 96, 96), "fp32", "shear", "capsule", 10, 4, 40),
        # the same in FP64, for reference runs
        _single("capsule96_fp64", (96, 96, 96), "fp64", "shear", "capsule", 10, 4, 10),
        # fluid alone: the lid-driven cavity on its finest grid
        _single("cavity193_fp32", (193, 193, 193), "fp32", "cavity", "none", 0, 0, 20),
        # the large run: a sphere settling in a closed box of 12.3 M nodes
        _single("settling160_fp32", (160, 160, 480), "fp32", "box", "sphere", 8, 5, 20, tau=0.7),
        # the same with populations stored as FP16 deviations
        _single("settling160_fp16", (160, 160, 480), "fp16", "box", "sphere", 8, 5, 20, tau=0.7),
        # a parameter study: 64 uneven capsule lattices advanced as one batch
        dict(name="batch64_fp32", kind="batch", count=64, nmin=48, nmax=112, mixed=0, prec="fp32", steps=30),
        # serving: small runs of both kinds submitted at once to a server
        dict(name="serve12_fp32", kind="serve", count=12, nmin=32, nmax=64, mixed=1, prec="fp32", steps=240),
    ]


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["record", "monitor", "batch", "batch", "serve"])
    if kind in ("batch", "serve"):
        nmin = rng.randint(48, 64) if kind == "batch" else rng.randint(32, 48)
        c = dict(kind=kind, count=rng.randint(3, 24 if kind == "batch" else 10), nmin=nmin,
                 nmax=nmin + rng.randint(4, 48 if kind == "batch" else 24), mixed=rng.randint(0, 1),
                 prec=rng.choice(["fp32", "fp32", "fp16", "bf16"]))
        c["steps"] = rng.randint(13, 40) if kind == "batch" else rng.randint(60, 240)
        return c
    prec = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16", "fp64"])
    body = rng.choice(["sphere", "sphere", "spheroid", "capsule", "capsule", "none"])
    if body == "none" and kind != "run":
        body = "sphere"
    least = 48 if body == "capsule" else 24
    most = 64 if kind == "monitor" else 96 if prec == "fp64" else 208
    side = math.exp(rng.uniform(math.log(least), math.log(most)))
    n = [max(least, min(2 * most, int(round(side * math.exp(rng.uniform(-0.3, 0.3)))))) for _ in range(3)]
    flow = rng.choice(["shear", "shear", "box"]) if body != "none" else rng.choice(["cavity", "channel"])
    if body == "capsule":
        flow = "shear"
    radius = max(3.5, min(n) / rng.uniform(8.0, 12.0))
    level = 3 if radius <= 7.0 else 4 if radius <= 14.0 else 5
    cells = n[0] * n[1] * n[2]
    steps = 1 if kind == "monitor" else max(7, min(40, int(2.4e8 / cells)))
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], prec=prec, flow=flow, body=body, radius=float(radius),
                level=level if body != "none" else 0, steps=steps, tau=rng.choice([0.7, 0.8, 1.0]),
                option=rng.randint(0, 1))


# ---- what a user's program has in hand ------------------------------------------------

@functools.lru_cache(maxsize=None)
def _unit_sphere(level):
    return W.icosphere(level)


def _walls(flow):
    """(bc, wall velocities, gext) of a flow."""
    w = np.zeros((6, 3))
    if flow == "shear":
        return (0, 0, 1), w, (0.0, 0.0, 0.0)
    if flow == "channel":  # driven along x between y walls
        return (0, 1, 0), w, (1e-6, 0.0, 0.0)
    return (1, 1, 1), w, (0.0, 0.0, 0.0)


def _plan(c, seed):
    """Everything that defines a single run, in plain host values."""
    rng = np.random.default_rng([int(seed), c["nx"], c["ny"], c["nz"]])
    n = (c["nx"], c["ny"], c["nz"])
    bc, wall_u, gext = _walls(c["flow"])
    if c["flow"] == "shear":
        U = float(rng.uniform(0.004, 0.008))
        wall_u = W.shear_walls(U)
    elif c["flow"] == "cavity":
        wall_u[3, 2] = float(rng.uniform(0.01, 0.02))
    p = dict(n=n, tau=c["tau"], bc=bc, wall_u=wall_u, gext=gext, prec=c["prec"], body=None,
             amp=1e-3, phase=rng.uniform(0, 2 * math.pi, 9))
    if c["body"] != "none":
        r = c["radius"]
        cen = (np.array(n) - 1) / 2.0 + rng.uniform(-0.5, 0.5, 3)
        if c["flow"] == "box":
            cen[2] = 0.7 * (n[2] - 1) + rng.uniform(-0.5, 0.5)
            cen[2] = min(cen[2], n[2] - 6 - r)
        v, f = _unit_sphere(c["level"])
        axes = np.array([r, r / 2, r / 2]) if c["body"] == "spheroid" else np.array([r, r, r])
        verts = v * axes + cen
        if c["body"] == "capsule":
            rate = 2 * U / (n[2] - 1)
            Ca = float(rng.uniform(0.05, 0.3))
            kw = dict(rigid=False, ks0=W.ks0_from_capillary(Ca, c["tau"], rate, r), Eb=0.01, kv=1.0, density_ratio=1.0,
                      ref_radius=r, mass_model=1, bend_variant=c["option"])
        else:
            gamma = float(rng.uniform(1.1, 1.5)) if c["flow"] == "box" else 1.0
            # terminal Reynolds number of a settling body: at most 5, and so
            # slow in small boxes that it stays clear of the floor for long
            d = 2 * r
            Re = min(5.0, 2e-6 * n[2] * d / W.viscosity(c["tau"]) * (1 if n[2] < 400 else 1e3))
            g = W.settling_gravity(Re, gamma, d, c["tau"]) if gamma > 1 else 0.0
            kw = dict(rigid=True, density_ratio=gamma, ref_radius=r, gravity=(0.0, 0.0, -g), rigid_force=c["option"])
        p["body"] = (verts, f, kw)
    return p


def _fields(p, device):
    """The initial density and velocity: the steady profile of the walls
    (shear flows) plus a smooth perturbation that vanishes on the walls."""
    nx, ny, nz = p["n"]
    ax = [torch.arange(m, dtype=torch.float64, device=device) for m in (nx, ny, nz)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    win = torch.ones((nz, ny, nx), dtype=torch.float64, device=device)
    for a, (q, m) in enumerate(((x, nx), (y, ny), (z, nz))):
        if p["bc"][a]:
            win = win * torch.sin(math.pi * q / (m - 1))
    th = [2 * math.pi * x / nx, 2 * math.pi * y / ny, 2 * math.pi * z / nz]
    ph = p["phase"]
    u = torch.empty((nz, ny, nx, 3), dtype=torch.float64, device=device)
    for a in range(3):
        b, d = (a + 1) % 3, (a + 2) % 3
        u[..., a] = p["amp"] * win * torch.sin(th[b] + ph[3 * a]) * torch.cos(th[d] + ph[3 * a + 1])
    lo, hi = float(p["wall_u"][4, 0]), float(p["wall_u"][5, 0])
    if lo != hi:
        u[..., 0] += lo + (hi - lo) * z / (nz - 1)
    rho = 1.0 + 1e-4 * win * torch.cos(th[0] + ph[2]) * torch.cos(th[2] + ph[5])
    return rho.reshape(-1).contiguous(), u.reshape(-1).contiguous()


def _context(p, stream):
    ctx = lbib.Context(p["n"], p["tau"], bc=p["bc"], wall_u=p["wall_u"], body_force=p["gext"], precision=PREC[p["prec"]],
                       stream=stream.cuda_stream)
    with torch.cuda.stream(stream):
        rho, u = _fields(p, "cuda")
        lbib.lbib_set_fields(ctx.h, rho, u)
        ctx.sync()
    if p["body"] is not None:
        verts, tris, kw = p["body"]
        ctx.add_body(verts, tris, **kw)
    return ctx


def _members(c, seed):
    """The runs of a batch or of a served stream: capsules in shear, or
    (mixed) capsules and settling spheres in turn, drawn as the repository's
    batch and serving streams draw them."""
    rng = np.random.default_rng([int(seed), c["count"], c["nmin"], c["nmax"]])
    # the sizes belong to the case, the rest to the seed
    sizes = np.random.default_rng([c["count"], c["nmin"], c["nmax"]]).integers(c["nmin"], c["nmax"] + 1, c["count"])
    out = []
    for k in range(c["count"]):
        capsule = not (c["mixed"] and k % 2)
        m = int(max(sizes[k], 48)) if capsule else int(sizes[k])
        r = m / 10.0
        sub = dict(nx=m, ny=m, nz=m, prec=c["prec"], flow="shear" if capsule else "box",
                   body="capsule" if capsule else "sphere", radius=max(r, 3.5), level=3 if r <= 7.0 else 4,
                   tau=0.8 if capsule else 0.7, option=0)
        out.append(_plan(sub, int(rng.integers(1 << 30))))
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.stream = case, torch.cuda.Stream()
    if case["kind"] == "serve":
        # the runs a client is about to submit; steps differ from run to run
        s.plans = _members(case, seed)
        s.steps = _serve_steps(case)
        return s
    if case["kind"] == "batch":
        s.plans = _members(case, seed)
        s.ctx = [_context(p, s.stream) for p in s.plans]
        s.batch = lbib.Batch(s.ctx, s.stream.cuda_stream)
    else:
        s.plans = [_plan(case, seed)]
        s.ctx = [_context(s.plans[0], s.stream)]
    return s


def _serve_steps(case):
    return [case["steps"] * (2 + k % 5) // 6 for k in range(case["count"])]


# ---- one pass -------------------------------------------------------------------------

def _fields_of(ctx, prec):
    rho = torch.empty(ctx.ncell, dtype=torch.float64, device="cuda")
    u = torch.empty(3 * ctx.ncell, dtype=torch.float64, device="cuda")
    lbib.lbib_get_fields(ctx.h, rho, u)
    return rho.to(KEPT[prec]), u.to(KEPT[prec])


def _reads_force(c):
    return c["kind"] in ("run", "monitor") and c["body"] != "capsule" and c["prec"] in ("fp64", "fp32")


def _markers_of(ctx, prec, force=False):
    X, V, F = (np.empty((ctx.nv[0], 3)) if k < 2 or force else None for k in range(3))
    lbib.lbib_get_markers(ctx.h, 0, X, V, F)
    return _kept_markers([X, V, F], prec)


def _kept_markers(arrays, prec):
    pos = torch.float64 if prec == "fp64" else torch.float32
    return [torch.as_tensor(a).to(t) for a, t in zip(arrays, (pos, KEPT[prec], KEPT[prec])) if a is not None]


def _joined(parts):
    return [torch.cat([p.reshape(-1) for p in col]) for col in zip(*parts)]


def run(state):
    c = state.case
    prec = c["prec"]
    with torch.cuda.stream(state.stream):
        if c["kind"] == "run":
            ctx = state.ctx[0]
            ctx.step(c["steps"])
            out = dict(zip(("rho", "u"), _fields_of(ctx, prec)))
            if ctx.nv:
                out.update(zip(("X", "V", "F"), _markers_of(ctx, prec, _reads_force(c))))
            return out
        if c["kind"] == "monitor":
            ctx = state.ctx[0]
            ctx.step(1)
            out = dict(zip(("X", "V", "F"), _markers_of(ctx, prec, _reads_force(c))))
            b = ctx.body(0)
            wide = KEPT[prec] if prec in ("fp64", "fp32") else torch.float32
            out["body"] = torch.as_tensor(np.concatenate([b["xc"], b["u"], b["omega"], b["q"], [b["volume"], b["area"]]])).to(wide)
            return out
        if c["kind"] == "record":
            ctx = state.ctx[0]
            rec = [torch.empty((c["steps"], ctx.nv[0], 3), dtype=torch.float64, pin_memory=True) for _ in range(2)]
            lbib.lbib_step_markers(ctx.h, c["steps"], 0, *rec)
            ctx.sync()
            return dict(zip(("X", "V"), _kept_markers(rec, prec)))
        if c["kind"] == "batch":
            state.batch.step(c["steps"])
            state.batch.sync()
            done = state.ctx
        else:
            # a client's session: start a server, submit, wait, collect
            server = lbib.lbib_serve_create(64 << 30, chunk_steps=100, max_active=64)
            ids = []
            for p, steps in zip(state.plans, state.steps):
                par = lbib.make_params(p["n"], p["tau"], bc=p["bc"], wall_u=p["wall_u"], precision=PREC[prec])
                req = lbib.lbib_request_create(par, steps, int(p["bc"] == (0, 0, 1)))
                verts, tris, kw = p["body"]
                lbib.lbib_request_add_body(req, verts, tris, lbib.make_body_params(**kw))
                ids.append(lbib.lbib_serve_submit(server, req))
            done = []
            for i, p in zip(ids, state.plans):
                rc, _ = lbib.lbib_serve_wait(server, i)
                h, times, rc = lbib.lbib_serve_take(server, i)
                if h is None:
                    raise RuntimeError("a served run failed: %s" % times["error"])
                done.append(lbib.Context.adopt(h, p["n"], [len(p["body"][0])]))
        fields = _joined([_fields_of(x, prec) for x in done])
        marks = _joined([_markers_of(x, prec) for x in done])
        if c["kind"] == "serve":
            for x in done:
                x.close()
            lbib.lbib_serve_destroy(server)
        return dict(zip(("rho", "u", "X", "V"), fields + marks))


def work(case):
    """Per time step: every population read and written once, every marker's
    position and velocity written once and its position read; per
    pass: the read-back.  About 220 operations a node, 4000 a fitted point."""
    def one(n, prec, nv, steps, fields):
        cells = n[0] * n[1] * n[2]
        pts = nv + 4 * nv  # markers, and two probes on each of about 2 nv triangles
        b = steps * (2 * 19 * ELEM[prec] * cells + 72 * nv) + (32 * cells if fields else 0) + 48 * nv
        return b, steps * (220.0 * cells + 4000.0 * pts)
    if case["kind"] in ("batch", "serve"):
        steps = [case["steps"]] * case["count"] if case["kind"] == "batch" else _serve_steps(case)
        parts = [one(p["n"], case["prec"], len(p["body"][0]), k, True) for p, k in zip(_members(case, 0), steps)]
    else:
        nv = 10 * 4 ** case["level"] + 2 if case["body"] != "none" else 0
        parts = [one((case["nx"], case["ny"], case["nz"]), case["prec"], nv, case["steps"], case["kind"] == "run")]
        if case["kind"] == "record":
            parts.append((48.0 * nv * case["steps"], 0.0))
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


# ---- the same in 64 bits, from the method's equations ---------------------------------

_E = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [1, -1, 0],
               [1, 0, 1], [1, 0, -1], [-1, 1, 0], [-1, -1, 0], [-1, 0, 1], [-1, 0, -1], [0, 1, 1], [0, 1, -1],
               [0, -1, 1], [0, -1, -1]])
_W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
_OPP = [int(np.where((_E == -e).all(axis=1))[0][0]) for e in _E]


class _Exact:
    """One lattice with at most one body (IB markers at the vertices), FP64."""

    def __init__(self, p, device, start="fields"):
        self.p, self.dev = p, device
        self.n, self.tau, self.bc = p["n"], p["tau"], p["bc"]
        if start == "fields":
            rho, u = _fields(p, device)
        else:  # a served run: density 1, the steady profile of the walls or rest
            rho, u = _fields(dict(p, amp=0.0), device)
            rho = torch.ones_like(rho)
        nx, ny, nz = self.n
        rho = rho.reshape(nz, ny, nx)
        u = u.reshape(nz, ny, nx, 3).movedim(-1, 0)
        self.w = torch.tensor(_W, device=device)
        self.e = torch.tensor(_E, dtype=torch.float64, device=device)
        self.g = self._feq(rho - 1, u)
        self.rho, self.u = rho, u
        self.gext = [float(v) for v in p["gext"]]
        if p["body"] is not None:
            self._body(*p["body"])

    def _eu(self, i, u):
        t = None
        for a in range(3):
            if _E[i, a]:
                t = u[a] * float(_E[i, a]) if t is None else t + u[a] * float(_E[i, a])
        return t

    def _feq(self, dr, u):
        g = torch.empty((19,) + dr.shape, dtype=torch.float64, device=self.dev)
        uu = (u * u).sum(0)
        for i in range(19):
            eu = self._eu(i, u)
            q = -1.5 * uu if eu is None else 3 * eu + 4.5 * eu * eu - 1.5 * uu
            g[i] = _W[i] * (dr + (1 + dr) * q)
        return g

    def _wall_velocity(self, faces):
        out = np.zeros(3)
        code = {a: s for a, s in faces}
        wu = self.p["wall_u"]
        for a in range(3):
            if a in code:
                out[a] = wu[2 * a + (code[a] < 0)][a]
            else:
                out[a] = np.mean([wu[2 * b + (s < 0)][a] for b, s in faces])
        return out

    def _walls(self, g):
        walled = [a for a in range(3) if self.bc[a]]
        for combo in itertools.product(*[(0, 1, -1) for _ in walled]):
            faces = [(a, s) for a, s in zip(walled, combo) if s]  # s: the inward normal's sign
            if not faces:
                continue
            at = [slice(None)] * 3
            for a in walled:
                at[a] = slice(1, -1)
            for a, s in faces:
                at[a] = slice(0, 1) if s > 0 else slice(-1, None)
            idx = (at[2], at[1], at[0])
            h = [g[i][idx].clone() for i in range(19)]
            uw = self._wall_velocity(faces)
            unknown = [any(s * _E[i, a] > 0 for a, s in faces) for i in range(19)]
            new = list(h)
            if len(faces) == 1:
                (a, s), = faces
                s0 = sum(h[i] for i in range(19) if _E[i, a] == 0)
                so = sum(h[i] for i in range(19) if s * _E[i, a] < 0)
                rho = (1 + s0 + 2 * so) / (1 - s * uw[a])
                N = {b: 0.5 * sum(float(_E[i, b]) * h[i] for i in range(19) if _E[i, a] == 0 and _E[i, b]) - rho * uw[b] / 3
                     for b in range(3) if b != a}
                for i in range(19):
                    if unknown[i]:
                        new[i] = h[_OPP[i]] + 6 * _W[i] * rho * float(_E[i] @ uw)
                        for b in N:
                            if _E[i, b]:
                                new[i] = new[i] - float(_E[i, b]) * N[b]
            else:
                uu = float(uw @ uw)
                for i in range(19):
                    if unknown[i]:
                        eu = float(_E[i] @ uw)
                        new[i] = h[_OPP[i]] + 6 * _W[i] * eu if not unknown[_OPP[i]] else torch.full_like(
                            h[i], _W[i] * (3 * eu + 4.5 * eu * eu - 1.5 * uu))
            for i in range(19):
                if unknown[i]:
                    g[i][idx] = new[i]

    def step(self):
        g = torch.stack([torch.roll(self.g[i], shifts=(int(_E[i, 2]), int(_E[i, 1]), int(_E[i, 0])), dims=(0, 1, 2))
                         for i in range(19)])
        F = None
        if self.p["body"] is not None:
            dr, j = self._moments(g)
            F = self._ib(dr, (j + 0.5 * torch.tensor(self.gext, device=self.dev)[:, None, None, None]) / (1 + dr))
        self._walls(g)
        dr, j = self._moments(g)
        if F is None:
            F = torch.zeros((3,) + dr.shape, dtype=torch.float64, device=self.dev)
        for a in range(3):
            F[a] += self.gext[a]
        for a in range(3):  # no body force on wall nodes
            if self.bc[a]:
                F.select(3 - a, 0).zero_()
                F.select(3 - a, -1).zero_()
        rho = 1 + dr
        u = (j + 0.5 * F) / rho
        om, cF = 1 / self.tau, 1 - 0.5 / self.tau
        uu, uF = (u * u).sum(0), (u * F).sum(0)
        for i in range(19):
            eu, eF = self._eu(i, u), self._eu(i, F)
            if eu is None:
                feq, guo = dr - 1.5 * rho * uu, -3 * uF
            else:
                feq = dr + rho * (3 * eu + 4.5 * eu * eu - 1.5 * uu)
                guo = 3 * (eF - uF) + 9 * eu * eF
            g[i] += om * (_W[i] * feq - g[i]) + _W[i] * cF * guo
        self.g, self.rho, self.u = g, rho, u

    def _moments(self, g):
        j = torch.zeros((3,) + g.shape[1:], dtype=torch.float64, device=self.dev)
        for i in range(1, 19):
            for a in range(3):
                if _E[i, a]:
                    j[a].add_(g[i], alpha=float(_E[i, a]))
        return g.sum(0), j

    # -- the immersed body --
    def _body(self, verts, tris, kw):
        d = self.dev
        self.kw = kw
        self.X = torch.tensor(verts, device=d)
        self.Xp = self.X.clone()
        self.T = torch.tensor(tris.astype(np.int64), device=d)
        self.off = torch.tensor([[x, y, z] for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)], device=d)
        self.V = torch.zeros_like(self.X)
        self.Fl = torch.zeros_like(self.X)
        a, b, c = (verts[tris[:, k]] for k in range(3))
        vol6 = np.einsum("ij,ij->i", a, np.cross(b, c))
        self.vol0 = vol6.sum() / 6
        if kw["rigid"]:
            s = a + b + c
            cen = (vol6[:, None] / 6 * s / 4).sum(0) / self.vol0
            C = sum(np.einsum("t,ti,tj->ij", vol6 / 120, q, q) for q in (a, b, c, s)) - self.vol0 * np.outer(cen, cen)
            I = np.trace(C) * np.eye(3) - C
            self.I, self.Ii = kw["density_ratio"] * I, np.linalg.inv(kw["density_ratio"] * I)
            self.m = kw["density_ratio"] * self.vol0
            self.xc, self.q = cen.copy(), np.array([1.0, 0, 0, 0])
            self.ub, self.ubp, self.om, self.omp = (np.zeros(3) for _ in range(4))
            self.Xb = self.X - torch.tensor(cen, device=d)
            return
        edge = {}
        for t in range(len(tris)):
            for k in range(3):
                edge[(int(tris[t, k]), int(tris[t, (k + 1) % 3]))] = (t, int(tris[t, (k + 2) % 3]))
        H = np.array([(i, j, w[1], edge[(j, i)][1]) for (i, j), w in edge.items() if i < j])
        HT = np.array([(w[0], edge[(j, i)][0]) for (i, j), w in edge.items() if i < j])
        area = 0.5 * np.linalg.norm(np.cross(b - a, c - a), axis=1)
        self.l0 = torch.tensor(np.linalg.norm(verts[H[:, 0]] - verts[H[:, 1]], axis=1), device=d)
        self.ks = kw["ks0"] * torch.tensor(area[HT].sum(1), device=d) / self.l0 ** 2
        self.kb = kw["Eb"] * self.ks * kw["ref_radius"] ** 2
        self.H = torch.tensor(H, device=d)
        self.th0 = self._hinge(self.X)[0]
        self.mv = (kw["density_ratio"] * self.vol0 if kw["mass_model"] else kw["density_ratio"] * area.sum()) / len(verts)

    def _hinge(self, X):
        xa, xb, xc, xd = (X[self.H[:, k]] for k in range(4))
        e, ac, ad = xb - xa, xc - xa, xd - xa
        N1, N2 = torch.linalg.cross(e, ac), torch.linalg.cross(ad, e)
        l1, l2, le = (v.norm(dim=1, keepdim=True) for v in (N1, N2, e))
        n1, n2 = N1 / l1, N2 / l2
        th = torch.atan2((torch.linalg.cross(n1, n2) * e).sum(1) / le[:, 0], (n1 * n2).sum(1))
        tc, td = (ac * e).sum(1, keepdim=True) / le ** 2, (ad * e).sum(1, keepdim=True) / le ** 2
        p1, p2 = n1 * le / l1, n2 * le / l2
        return th, e, le, [(1 - tc) * p1 + (1 - td) * p2, tc * p1 + td * p2, -p1, -p2]

    def _mls(self, P):
        base = torch.floor(P + 0.5)
        off = self.off.to(torch.float64)
        d = off[None] - (P - base)[:, None, :]
        node = base.to(torch.int64)[:, None, :] + self.off[None]
        for a in range(3):
            if not self.bc[a]:
                node[..., a] %= self.n[a]
        flat = node[..., 0] + self.n[0] * (node[..., 1] + self.n[1] * node[..., 2])
        r = (d * d).sum(-1).sqrt() / 1.3
        w = torch.where(r <= 1, torch.exp(-(r / 0.3) ** 2), torch.zeros_like(r))
        p = torch.cat([torch.ones_like(r)[..., None], d], dim=-1)
        A = torch.einsum("nk,nki,nkj->nij", w, p, p)
        psi = torch.linalg.solve(A, (w[..., None] * p).transpose(1, 2))  # (N, 4, 27)
        return psi, flat

    def _ib(self, dr, us):
        X, T = self.X, self.T
        fr, fu = dr.reshape(-1), us.reshape(3, -1)
        psi, node = self._mls(X)
        phi = psi[:, 0]
        U = (phi[None] * fu[:, node]).sum(-1).T
        x0, x1, x2 = (X[T[:, k]] for k in range(3))
        N = torch.linalg.cross(x1 - x0, x2 - x0)
        nn = N.norm(dim=1, keepdim=True)
        nrm, area, cen = N / nn, 0.5 * nn[:, 0], (x0 + x1 + x2) / 3
        nu = (self.tau - 0.5) / 3
        st = []
        for sg in (1.2, -1.2):
            ps, nd = self._mls(cen + sg * nrm)
            rho = 1 + (ps[:, 0] * fr[nd]).sum(-1)
            G = torch.einsum("nik,ank->nai", ps[:, 1:], fu[:, nd])
            tr = (rho * nu)[:, None] * ((G + G.transpose(1, 2)) @ nrm[..., None])[..., 0]
            st.append(((rho - 1) / 3, tr))
        Ft = (-(st[0][0] - st[1][0])[:, None] * nrm + st[0][1] - st[1][1]) * area[:, None]
        Av = torch.zeros(len(X), dtype=torch.float64, device=self.dev)
        for k in range(3):
            Av.index_add_(0, T[:, k], area / 3)
        if self.kw["rigid"]:
            Ub, Xn = self._rigid(Ft, cen, Av)
        else:
            Ub, Xn = self._membrane(Ft, nrm, area, U)
        Fl = Ub - U
        F = torch.zeros_like(fu)
        for a in range(3):
            F[a].index_add_(0, node.reshape(-1), ((Av * Fl[:, a])[:, None] * phi).reshape(-1))
        self.V, self.Fl = Ub, Fl
        self.Xp, self.X = X, Xn
        return F.reshape(us.shape)

    def _rigid(self, Ft, cen, Av):
        kw = self.kw
        if kw["rigid_force"]:
            fm, at = -Av[:, None] * self.Fl, self.X
        else:
            fm, at = Ft, cen
        F = fm.sum(0).cpu().numpy()
        M = torch.linalg.cross(at - torch.tensor(self.xc, device=self.dev), fm).sum(0).cpu().numpy()
        F = F + (kw["density_ratio"] - 1) * self.vol0 * np.array(kw["gravity"])
        R = self._R(self.q)
        if kw["rigid_force"]:
            F = F + self.vol0 * (self.ub - self.ubp)
            M = M + R @ self.I @ R.T @ (self.om - self.omp) / kw["density_ratio"]
        un = 2 / 3 * (2 * self.ub - 0.5 * self.ubp + F / self.m)
        wn = 2 / 3 * (2 * self.om - 0.5 * self.omp + R @ self.Ii @ R.T @ M)
        t = lambda v: torch.tensor(v, device=self.dev)  # noqa: E731
        Ub = t(un) + torch.linalg.cross(t(wn).expand_as(self.X), self.X - t(self.xc))
        self.ubp, self.ub, self.omp, self.om = self.ub, un, self.om, wn
        self.xc = self.xc + un
        th = float(np.linalg.norm(wn))
        if th > 0:
            w, v = math.cos(th / 2), math.sin(th / 2) / th * wn
            q0, qv = self.q[0], self.q[1:]
            self.q = np.concatenate([[w * q0 - v @ qv], w * qv + q0 * v + np.cross(v, qv)])
            self.q /= np.linalg.norm(self.q)
        return Ub, t(self.xc) + self.Xb @ t(self._R(self.q)).T

    @staticmethod
    def _R(q):
        w, x, y, z = q
        return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                         [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                         [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])

    def _membrane(self, Ft, nrm, area, U):
        X, kw = self.X, self.kw
        th, e, le, grad = self._hinge(X)
        F = torch.zeros_like(X)
        sp = (self.ks * (le[:, 0] - self.l0))[:, None] * e / le
        F.index_add_(0, self.H[:, 0], sp)
        F.index_add_(0, self.H[:, 1], -sp)
        dth = th - self.th0
        dE = self.kb * (dth if kw["bend_variant"] else torch.sin(dth))
        for k in range(4):
            F.index_add_(0, self.H[:, k], -dE[:, None] * grad[k])
        x0, x1, x2 = (X[self.T[:, k]] for k in range(3))
        vol = (x0 * torch.linalg.cross(x1, x2)).sum() / 6
        el = kw["kv"] * (1 - vol / self.vol0) * nrm * area[:, None] + Ft
        for k in range(3):
            F.index_add_(0, self.T[:, k], el / 3)
        acc = F / self.mv
        xt = X + U + 0.5 * acc
        return U + acc, X + (1.5 * xt - 2 * X + 0.5 * self.Xp) + 0.5 * acc

    def fields(self):
        return self.rho.reshape(-1), self.u.movedim(0, -1).reshape(-1)

    def body_numbers(self):
        x0, x1, x2 = (self.X[self.T[:, k]] for k in range(3))
        vol = float((x0 * torch.linalg.cross(x1, x2)).sum()) / 6
        area = 0.5 * float(torch.linalg.cross(x1 - x0, x2 - x0).norm(dim=1).sum())
        if self.kw["rigid"]:
            head = [self.xc, self.ub, self.om, self.q]
        else:
            head = [self.X.mean(0).cpu().numpy(), self.V.mean(0).cpu().numpy(), np.zeros(3), np.array([1.0, 0, 0, 0])]
        return torch.as_tensor(np.concatenate(head + [[vol, area]]))


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "serve" or (case["kind"] == "batch" and case["count"] * case["steps"] > 1200):
        return None  # thousands of coupled steps
    if case["kind"] == "batch":
        parts = []
        for p in _members(case, seed):
            x = _Exact(p, dev)
            for _ in range(case["steps"]):
                x.step()
            parts.append(x.fields() + (x.X, x.V))
        return dict(zip(("rho", "u", "X", "V"), _joined(parts)))
    x = _Exact(_plan(case, seed), dev)
    rec = []
    for _ in range(case["steps"]):
        x.step()
        if case["kind"] == "record":
            rec.append((x.X, x.V))
    if case["kind"] == "record":
        return {k: torch.stack([r[i] for r in rec]) for i, k in enumerate(("X", "V"))}
    out = {}
    if case["kind"] == "run":
        out.update(zip(("rho", "u"), x.fields()))
    if case["body"] != "none":
        out.update(X=x.X, V=x.V)
        if _reads_force(case):
            out.update(F=x.Fl)
    if case["kind"] == "monitor":
        out["body"] = x.body_numbers()
    return out
