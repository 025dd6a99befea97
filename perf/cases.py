"""Performance cases: the work a user of this package has it do, through its public entry points.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what
a program has in hand before the call (inputs on the GPU, or pinned host arrays for the
host-buffer step, and the grid or batch it keeps), ``run`` is one pass through the public entry
points, ``work`` the bytes and operations that pass cannot do without, and ``exact`` the same
results from plain torch in float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1803_01262_gb300 import cdi
from paper_1803_01262_gb300 import inputs as I
from paper_1803_01262_gb300.autograd import rollout
from paper_1803_01262_gb300.phase import euler_dt

DEV = "cuda"
L2_BYTES = 129e6          # a working set beyond this is read from memory again in every step
DTYPE = {"f32": torch.float32, "f64": torch.float64}
ESIZE = {"f32": 4, "f64": 8}


def listed():
    return [
        # The 2D single vortex (Section 3.3.1, Eq. 33) at the mesh the paper uses: the smallest
        # runs, where launches and latency count.
        dict(name="vortex_128_f32", kind="run", field="vortex", nx=128, ny=128, nz=1, dtype="f32", steps=32),
        # The 3D deformation sphere, the headline workload: consecutive Euler steps.
        dict(name="deformation_256_f32", kind="run", field="deformation", nx=256, ny=256, nz=256, dtype="f32",
             steps=8),
        # A production-size box (the inverse problem's 512^3 with a random solenoidal velocity).
        dict(name="random_512_f32", kind="run", field="random", nx=512, ny=512, nz=512, dtype="f32", steps=4),
        # A box whose edges are whatever the user's geometry asks for: odd rows, ragged tiles.
        dict(name="ragged_f32", kind="run", field="random", nx=301, ny=257, nz=211, dtype="f32", steps=8),
        # Double precision, the reference form every FP32 result is checked against.
        dict(name="deformation_128_f64", kind="run", field="deformation", nx=128, ny=128, nz=128, dtype="f64",
             steps=8),
        # One RK4 step (Section 2.3): the integrator of the paper's own experiments.
        dict(name="rk4_192_f32", kind="rk", scheme="rk4", nx=192, ny=192, nz=192, dtype="f32"),
        # One adjoint step: the inner operation of every gradient.
        dict(name="adjoint_256_f32", kind="adjoint", vel=False, nx=256, ny=256, nz=256, dtype="f32"),
        # One adjoint step with velocity gradients on a box with odd rows.
        dict(name="adjoint_ragged_vel_f32", kind="adjoint", vel=True, nx=203, ny=197, nz=187, dtype="f32"),
        # A checkpointed gradient through a rollout: forward, recompute, adjoint, velocity gradients.
        dict(name="gradient_128_f32", kind="gradient", nx=128, ny=128, nz=128, dtype="f32", steps=16, ckpt=8),
        # 64 independent boxes of uneven sizes (edges 32..160) advanced together.
        dict(name="batch_64_f32", kind="batch", nbox=64, nmin=32, nmax=160, dims_seed=0, dtype="f32", steps=8),
        # A phase-diagram sweep: the drop of Table 2 at 256 points of the (eps/dx, gamma/|u|) plane.
        dict(name="sweep_256_f64", kind="sweep", n=50, ne=16, ng=16, dtype="f64", sharpen="centre", steps=256),
        # The state in pinned host memory: in, one step, out, with its statistics.
        dict(name="host_256_f32", kind="host", nx=256, ny=256, nz=256, dtype="f32"),
    ]


def _dims3(rng, lo, hi):
    """Three edges around a log-uniform mean; half of the boxes with rows of whole 16-byte vectors."""
    m = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    d = [max(5, int(m * rng.uniform(0.75, 1.25))) for _ in range(3)]
    if rng.random() < 0.5:
        d[0] = max(8, d[0] // 4 * 4)
    return d


def draw(rng):
    """One more case of the listed ones' ranges (any edges, FP32 and FP64 as each path is used)."""
    kind = rng.choice(["run2", "run3", "run3", "run64", "rk", "adjoint", "adjoint", "gradient", "batch", "sweep",
                       "host"])
    if kind == "run2":
        n = int(math.exp(rng.uniform(math.log(24), math.log(1024))))
        return dict(kind="run", field="vortex", nx=n, ny=n, nz=1, dtype=rng.choice(["f32", "f32", "f64"]),
                    steps=rng.randrange(4, 65))
    if kind in ("run3", "run64"):
        nx, ny, nz = _dims3(rng, 24, 300) if kind == "run3" else _dims3(rng, 24, 140)
        return dict(kind="run", field="random", nx=nx, ny=ny, nz=nz, dtype="f32" if kind == "run3" else "f64",
                    steps=rng.randrange(1, 9))
    if kind == "rk":
        nx, ny, nz = _dims3(rng, 32, 256)
        return dict(kind="rk", scheme=rng.choice(["rk2", "rk3", "rk4", "rk4"]), nx=nx, ny=ny, nz=nz, dtype="f32")
    if kind == "adjoint":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        nx, ny, nz = _dims3(rng, 32, 300 if dtype == "f32" else 128)
        return dict(kind="adjoint", vel=rng.random() < 0.5, nx=nx, ny=ny, nz=nz, dtype=dtype)
    if kind == "gradient":
        nx, ny, nz = _dims3(rng, 32, 100)
        return dict(kind="gradient", nx=nx, ny=ny, nz=nz, dtype="f32", steps=rng.randrange(6, 17),
                    ckpt=rng.choice([4, 8, 16]))
    if kind == "batch":
        nmax = rng.randrange(48, 161)
        return dict(kind="batch", nbox=rng.randrange(8, 65), nmin=rng.randrange(16, 41), nmax=nmax,
                    dims_seed=rng.randrange(1, 1 << 20), dtype="f32", steps=rng.randrange(2, 9))
    if kind == "sweep":
        return dict(kind="sweep", n=rng.randrange(32, 57), ne=rng.randrange(4, 15), ng=rng.randrange(4, 15),
                    dtype="f64", sharpen=rng.choice(["centre", "centre", "face"]), steps=2 * rng.randrange(32, 101))
    nx, ny, nz = _dims3(rng, 64, 256)
    return dict(kind="host", nx=nx, ny=ny, nz=nz, dtype="f32")


# ---------------------------------------------------------------------------
# Inputs

def _curl(Ax, Ay, Az, h):
    """Discrete staggered curl of an edge-centred vector potential (None: zero), as inputs.staggered_curl."""
    def dm(a, dim):
        return a - torch.roll(a, 1, dims=dim) if a is not None else 0.0
    return ((dm(Az, 1) - dm(Ay, 0)) / h, (dm(Ax, 0) - dm(Az, 2)) / h, (dm(Ay, 2) - dm(Ax, 1)) / h)


def _velocity(field, shape, h, seed):
    """Face velocities in float64: the vortex, the deformation field, or a seeded random field."""
    nz, ny, nx = shape
    if field == "random":
        return I.random_velocity_torch(shape, h, seed=seed, device=DEV)
    c = lambda n, off: (torch.arange(n, dtype=torch.float64, device=DEV) + off) * h
    if field == "vortex":
        s2 = torch.sin(math.pi * c(nx, 1.0)) ** 2
        return [t + torch.zeros(shape, dtype=torch.float64, device=DEV)
                for t in _curl(None, None, -(s2[None, None, :] * s2[None, :, None]) / math.pi, h)]
    tp = 2.0 * math.pi
    xc, xf = c(nx, 0.5), c(nx, 1.0)
    X, Y, Z = (lambda a: a[None, None, :]), (lambda a: a[None, :, None]), (lambda a: a[:, None, None])
    Ay = X(torch.cos(tp * xf)) * Y(torch.sin(tp * xc)) * Z(torch.sin(math.pi * xf) ** 2) / tp
    Az = -(X(torch.cos(tp * xf)) * Y(torch.sin(math.pi * xf) ** 2) + Y(torch.cos(tp * xf))) * Z(
        torch.sin(tp * xc)) / tp
    return _curl(None, Ay, Az, h)


def _sphere(shape, h, eps, rng, radius=0.15):
    """A tanh sphere (drop in 2D) at a seeded place of the box."""
    nz, ny, nx = shape
    L = (nx * h, ny * h, nz * h)
    R = radius * min(v for v, n in zip(L, (nx, ny, nz)) if n > 1)
    ctr = [0.5 * h if n == 1 else v * float(rng.uniform(0.3, 0.7)) for v, n in zip(L, (nx, ny, nz))]
    return I.spheres_phi_torch(shape, h, [(ctr, R)], eps, device=DEV)


def _box(case, seed):
    """phi, (u, v, w) in the case's dtype, and the step's parameters: gamma = U and eps = dx, on the
    crossover line of Eq. 17."""
    rng = np.random.default_rng(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    h = 1.0 / min(n for n in shape if n > 1)
    t = DTYPE[case["dtype"]]
    vel = [x.to(t).contiguous() for x in _velocity(case.get("field", "random"), shape, h, seed)]
    U = max(float(x.abs().max()) for x in vel)
    phi = _sphere(shape, h, h, rng).to(t)
    cfl = 0.2 if case["kind"] == "rk" else 0.1
    return phi, vel, dict(h=h, U=U, eps=h, gamma=U, dt=cfl * h / U, rng=rng)


def _period(case):
    return {"vortex": 4.0, "deformation": 3.0}.get(case.get("field"), 0.0)


def _batch_boxes(case, seed):
    """(dims, phi, velocities, parameters) of every box of a batch; the edges come from the case alone."""
    dims = np.random.default_rng(case["dims_seed"]).integers(case["nmin"], case["nmax"] + 1, size=(case["nbox"], 3))
    rng = np.random.default_rng(seed)
    t = DTYPE[case["dtype"]]
    out = []
    for nx, ny, nz in dims.tolist():
        shape, h = (nz, ny, nx), 1.0 / min(nx, ny, nz)
        eoh = float(rng.choice([1.0, 1.5]))
        vel = [x.to(t).contiguous() for x in
               I.random_velocity_torch(shape, h, seed=int(rng.integers(1 << 30)), device=DEV)]
        U = max(float(x.abs().max()) for x in vel)
        gamma = U / (2.0 * eoh - 1.0)
        dt = 0.1 * h / U
        out.append((shape, _sphere(shape, h, eoh * h, rng).to(t), vel, dict(h=h, eps=eoh * h, gamma=gamma, dt=dt)))
    return out


def _sweep_boxes(case, seed):
    n, L = case["n"], 2.0
    rng = np.random.default_rng(seed)
    t = DTYPE[case["dtype"]]
    shape, h = (1, n, n), L / n
    c = math.sqrt(2.0) / 2.0
    vel = [torch.full(shape, x, dtype=t, device=DEV) for x in (c, c, 0.0)]
    out = []
    for eoh in np.linspace(0.55, 2.0, case["ne"]):
        for gu in np.linspace(0.3, 3.0, case["ng"]):
            eoh, gu = float(eoh), float(gu)
            out.append((shape, _sphere(shape, h, eoh * h, rng, radius=0.25).to(t), vel,
                        dict(h=h, eps=eoh * h, gamma=gu, dt=euler_dt(eoh, gu, n))))
    return out


def _flat(boxes, t):
    """One buffer for all boxes' states, and each box's view of it (16-byte aligned)."""
    sizes = [math.prod(s) for s, *_ in boxes]
    offs = np.concatenate([[0], np.cumsum([(m + 3) // 4 * 4 for m in sizes])]).tolist()
    buf = torch.zeros(offs[-1], dtype=t, device=DEV)
    return buf, [buf[o:o + m].view(s) for (s, *_), o, m in zip(boxes, offs, sizes)]


def prepare(case, seed):
    kind = case["kind"]
    t = DTYPE[case["dtype"]]
    if kind in ("batch", "sweep"):
        boxes = _batch_boxes(case, seed) if kind == "batch" else _sweep_boxes(case, seed)
        (buf_a, va), (buf_b, vb) = _flat(boxes, t), _flat(boxes, t)
        for x, (_, phi, _, _) in zip(va, boxes):
            x.copy_(phi)
        bt = cdi.Batch([dict(dx=p["h"], dt=p["dt"], eps=p["eps"], gamma=p["gamma"], u=v[0], v=v[1], w=v[2],
                             phi_a=a, phi_b=b) for (_, _, v, p), a, b in zip(boxes, va, vb)])
        if case.get("sharpen", "centre") != "centre":
            bt.set_sharpening(case["sharpen"])
        bt.autotune()
        return dict(case=case, bt=bt, a=buf_a, b=buf_b, phi0=buf_a.clone() if kind == "sweep" else None)
    phi, vel, p = _box(case, seed)
    shape = tuple(phi.shape)
    g = cdi.Grid(shape[2], shape[1], shape[0], p["h"], t)
    g.set_velocity(*vel)
    s = dict(case=case, g=g, vel=vel, args=(p["dt"], p["eps"], p["gamma"]))
    if kind == "host":
        s["out"] = torch.empty(shape, dtype=t, pin_memory=True).numpy()
        s["in"] = torch.empty(shape, dtype=t, pin_memory=True)
        s["in"].copy_(phi)
        s["in"] = s["in"].numpy()
        return s
    s["a"], s["b"] = phi, torch.empty_like(phi)
    if kind == "rk":
        s["w1"], s["w2"] = torch.empty_like(phi), torch.empty_like(phi)
    elif kind == "adjoint":
        s["lam"] = _sphere(shape, p["h"], p["eps"], p["rng"], 0.2).to(t) - phi
        s["grads"] = [torch.zeros_like(phi) for _ in range(3)] if case["vel"] else None
    elif kind == "gradient":
        s["target"] = _sphere(shape, p["h"], p["eps"], p["rng"], 0.2).to(t)
        for x in (phi, *vel):
            x.requires_grad_(True)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        s["bt"].run(case["steps"])
        return s["b"] if s["bt"].info()["parity"] else s["a"]
    if kind == "sweep":  # from the initial state each time: the classification of every point
        s["a"].copy_(s["phi0"])
        s["bt"].reset_run_stats()
        s["bt"].run(case["steps"])
        st = s["bt"].stats()
        return dict(phi=s["a"], **{k: np.array([r[k] for r in st]) for k in ("mass", "min_run", "max_run",
                                                                             "n_tol_run")})
    g, args = s["g"], s["args"]
    if kind == "run":
        out = g.run(s["a"], s["b"], case["steps"], *args, period=_period(case), check=True)
        if out is s["b"]:
            s["a"], s["b"] = s["b"], s["a"]
        return out
    if kind == "rk":
        return g.step_rk(s["a"], s["b"], s["w1"], s["w2"], *args, scheme=case["scheme"])
    if kind == "adjoint":
        lam = g.step_adjoint(s["a"], s["lam"], s["b"], *args, grads=s["grads"])
        return [lam] + (s["grads"] or [])
    if kind == "gradient":
        x = (s["a"], *s["vel"])
        for q in x:
            q.grad = None
        out = rollout(*x, g, case["steps"], *args, ckpt_every=case["ckpt"])
        loss = ((out - s["target"]) ** 2).sum()
        loss.backward()
        return [out, loss] + [q.grad for q in x]
    st = g.step_host(s["in"], s["out"], *args)
    return dict(phi=s["out"], stats={k: st[k] for k in ("mass", "min", "max", "n_tol")})


def work(case):
    """Bytes: phi in, u, v, w in, phi out (2D: no w) once per step, or once per pass where all of it
    stays in L2 between steps; flops: 17 per cell and direction (Section 3.3.3), about twice that for
    an adjoint step."""
    kind, e = case["kind"], ESIZE[case["dtype"]]
    if kind == "batch":
        dims = np.random.default_rng(case["dims_seed"]).integers(case["nmin"], case["nmax"] + 1,
                                                                 size=(case["nbox"], 3))
        cells, axes = int(dims.prod(axis=1).sum()), 3
    elif kind == "sweep":
        cells, axes = case["ne"] * case["ng"] * case["n"] ** 2, 2
    else:
        cells, axes = case["nx"] * case["ny"] * case["nz"], 3 if case["nz"] > 1 else 2
    steps = case.get("steps", 1)
    per = (2 + axes) * e * cells
    reads = steps if per > L2_BYTES else 1
    flops = 17 * axes * cells
    if kind == "rk":  # stage operands read and written besides (RK4: 24 + 32 + 32 + 24 bytes per FP32 cell)
        fields = {"rk2": 11, "rk3": 19, "rk4": 28}[case["scheme"]]
        stages = {"rk2": 2, "rk3": 3, "rk4": 4}[case["scheme"]]
        return dict(bytes=fields * e * cells if per > L2_BYTES else per, flops=stages * flops)
    if kind == "adjoint":
        return dict(bytes=(12 if case["vel"] else 6) * e * cells, flops=2 * flops)
    if kind == "gradient":  # forward, recompute, adjoint with the velocity gradient
        total = (5 * (2 * steps - 1) + 12 * steps) * e * cells
        return dict(bytes=total if per > L2_BYTES else 12 * e * cells, flops=4 * steps * flops)
    if kind == "host":
        return dict(bytes=per, flops=flops)
    return dict(bytes=per * reads, flops=steps * flops)


# ---------------------------------------------------------------------------
# The same results in float64, from the equations

def _p(a, d):
    return torch.roll(a, -1, dims=d)


def _m(a, d):
    return torch.roll(a, 1, dims=d)


def _normal(phi, floor2=0.0):
    g = [_p(phi, d) - _m(phi, d) for d in (2, 1, 0)]
    q = g[0] * g[0] + g[1] * g[1] + g[2] * g[2]
    m = torch.sqrt(q + floor2)
    inv = torch.where(q > 0, 1.0 / torch.where(q > 0, m, torch.ones_like(m)), torch.zeros_like(m))
    return [x * inv for x in g], inv


def _rhs(phi, vel, h, eps, gamma, vs, face=False):
    """d phi / dt of Eq. 1 by central differences on faces (Section 2.2)."""
    n, _ = _normal(phi)
    div = torch.zeros_like(phi)
    for d, u, nd in zip((2, 1, 0), vel, n):
        R = _p(phi, d)
        if face:
            f = 0.5 * (phi + R)
            sh = f * (1 - f) * 0.5 * (nd + _p(nd, d))
        else:
            s = phi * (1 - phi) * nd
            sh = 0.5 * (s + _p(s, d))
        F = vs * u * 0.5 * (phi + R) - gamma * eps * (R - phi) / h + gamma * sh
        div += (F - _m(F, d)) / h
    return -div


def _adjoint(phi, lam, vel, h, dt, eps, gamma, vs, floor, want_vel):
    """lam_k of lam_{k+1} through the step's five parts in reverse; the normal's derivative with |g|
    floored by ``floor``."""
    n, inv = _normal(phi, floor * floor)
    pb = torch.zeros_like(phi)
    sb, gv = [], []
    for d, u in zip((2, 1, 0), vel):
        Fb = (dt / h) * (_p(lam, d) - lam)
        a, c = 0.5 * vs * u, gamma * eps / h
        pb += Fb * (a + c) + _m(Fb * (a - c), d)
        sb.append(0.5 * gamma * (Fb + _m(Fb, d)))
        if want_vel:
            gv.append(Fb * (0.5 * vs) * (phi + _p(phi, d)))
    ns = sum(x * y for x, y in zip(n, sb))
    pb += (1 - 2 * phi) * ns
    for d, nd, s in zip((2, 1, 0), n, sb):
        gb = phi * (1 - phi) * (s - nd * ns) * inv
        pb += _m(gb, d) - _p(gb, d)
    return lam + pb, gv


def exact(case, seed):
    kind = case["kind"]
    d = torch.float64
    if kind in ("batch", "sweep"):
        boxes = _batch_boxes(case, seed) if kind == "batch" else _sweep_boxes(case, seed)
        buf, views = _flat(boxes, d)
        if kind == "batch":
            for x, (_, phi, vel, p) in zip(views, boxes):
                q, vel = phi.to(d), [v.to(d) for v in vel]
                for _ in range(case["steps"]):
                    q = q + p["dt"] * _rhs(q, vel, p["h"], p["eps"], p["gamma"], 1.0)
                x.copy_(q)
            return buf
        # the sweep's boxes are alike: one stack, axis 0 the box (no differences along it: w = 0)
        q = torch.cat([phi.to(d) for _, phi, _, _ in boxes])
        col = lambda k: torch.tensor([p[k] for *_, p in boxes], dtype=d, device=DEV).view(-1, 1, 1)
        h, dt, eps, gamma = boxes[0][3]["h"], col("dt"), col("eps"), col("gamma")
        u = boxes[0][2][0].to(d)
        lo, hi = torch.full_like(dt, math.inf), torch.full_like(dt, -math.inf)
        face = case["sharpen"] == "face"
        for _ in range(case["steps"]):
            g = [_p(q, k) - _m(q, k) for k in (2, 1)]
            r = torch.sqrt(g[0] * g[0] + g[1] * g[1])
            inv = torch.where(r > 0, 1.0 / torch.where(r > 0, r, torch.ones_like(r)), torch.zeros_like(r))
            div = torch.zeros_like(q)
            for k, gd in zip((2, 1), g):
                R, nd = _p(q, k), gd * inv
                if face:
                    f = 0.5 * (q + R)
                    sh = f * (1 - f) * 0.5 * (nd + _p(nd, k))
                else:
                    s = q * (1 - q) * nd
                    sh = 0.5 * (s + _p(s, k))
                F = u * 0.5 * (q + R) - gamma * eps * (R - q) / h + gamma * sh
                div += (F - _m(F, k)) / h
            q = q - dt * div
            lo = torch.minimum(lo, q.amin(dim=(1, 2), keepdim=True))
            hi = torch.maximum(hi, q.amax(dim=(1, 2), keepdim=True))
        for x, y in zip(views, q):
            x.copy_(y.unsqueeze(0))
        # (the face form amplifies rounding in the bulk: its extrema have no value to compare with)
        mass = (q.sum(dim=(1, 2)) * h ** 2).cpu().numpy()
        ext = (None, None) if face else (lo.flatten().cpu().numpy(), hi.flatten().cpu().numpy())
        return dict(phi=buf, mass=mass, min_run=ext[0], max_run=ext[1], n_tol_run=None)
    phi, vel, p = _box(case, seed)
    target_rng = p["rng"]
    q, vel = phi.to(d), [v.to(d) for v in vel]
    a = (p["h"], p["eps"], p["gamma"])
    dt, T = p["dt"], _period(case)
    vs = lambda t: math.cos(math.pi * t / T) if T > 0 else 1.0
    if kind == "run":
        for i in range(case["steps"]):
            q = q + dt * _rhs(q, vel, *a, vs(i * dt))
        return q
    if kind == "host":
        q = q + dt * _rhs(q, vel, *a, 1.0)
        return dict(phi=q, stats=dict(mass=float(q.sum()) * p["h"] ** 3, min=None, max=float(q.max()), n_tol=None))
    if kind == "rk":
        f = lambda y: dt * _rhs(y, vel, *a, 1.0)
        if case["scheme"] == "rk2":
            return q + f(q + 0.5 * f(q))
        if case["scheme"] == "rk3":  # Wray
            k1 = f(q)
            y1 = q + 8 / 15 * k1
            k2 = f(y1)
            y2 = y1 + 5 / 12 * k2 - 17 / 60 * k1
            return y2 + 3 / 4 * f(y2) - 5 / 12 * k2
        k1 = f(q)
        k2 = f(q + 0.5 * k1)
        k3 = f(q + 0.5 * k2)
        return q + (k1 + 2 * k2 + 2 * k3 + f(q + k3)) / 6
    floor = 8 * torch.finfo(DTYPE[case["dtype"]]).eps
    other = _sphere(tuple(phi.shape), p["h"], p["eps"], target_rng, 0.2).to(DTYPE[case["dtype"]])
    if kind == "adjoint":
        lam, gv = _adjoint(q, (other - phi).to(d), vel, p["h"], dt, p["eps"], p["gamma"], 1.0, floor, case["vel"])
        return [lam] + gv
    states = [q]
    for _ in range(case["steps"]):
        states.append(states[-1] + dt * _rhs(states[-1], vel, *a, 1.0))
    out = states.pop()
    r = out - other.to(d)
    lam, grads = 2 * r, [torch.zeros_like(q) for _ in range(3)]
    while states:
        lam, gv = _adjoint(states.pop(), lam, vel, p["h"], dt, p["eps"], p["gamma"], 1.0, floor, True)
        for x, y in zip(grads, gv):
            x += y
    return [out, float((r * r).sum()), lam] + grads
