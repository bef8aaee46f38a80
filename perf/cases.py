"""Measured work of the VIP solver: what a user's program has it do, through its
public entry points, from the smallest node sets to the largest.

Kinds of case
  step    vip_set_state, a few vip_step, vip_get_state on one context: the fractional
          step of Eqs. (12)-(15) from a given field (device buffers in and out).
          Cavities, circular and bumpy cylinders, batches of triangular cavities.
  solve   vip_solve of the Helmholtz or the bordered Poisson system (host arrays).
  apply   vip_apply of the step's operators to a field in device memory.
  build   a new context on a node set (neighbour search, MLS weights, operators,
          multigrid) and the first application of its operators.
  build3d the same for the 3D handle; step3d its fractional step.
  static  vip_bicgstab_static on a device CSR matrix.
  network vip_ws_eval: forward, loss and parameter gradients of the warm-start network.

Solves stop at a relative residual of 1e-12 (as the parity tests do; the default is
1e-8), so that the fields returned are determined by the equations to far
more digits than the stop leaves open.  Fields start from a smooth stream function
drawn from the seed; wall nodes keep the node set's own boundary values.
"""
import ctypes
import math

import numpy as np
import torch

import workloads
from paper_1401_6513_gb300 import vip

DEV = "cuda:0"
PREC = {"fp64": vip.VIP_PREC_FP64, "mixed": vip.VIP_PREC_MIXED, "mg32": vip.VIP_PREC_MG32}
NET = (16, 32, 32, 32, 32, 32, 1)  # channel widths of the warm-start network
LAM = 0.01                         # its loss's default weight


def listed():
    return [
        # the smallest flow in use: a lid-driven cavity for quick studies, where the
        # latency of launches and grid barriers is everything
        {"name": "step_cavity64", "kind": "step", "geom": "cavity", "n": 64, "prec": "fp64", "rtol": 1e-12,
         "steps": 2},
        # the circular cylinder at Re 100 in the form chosen for open channels, with the
        # fitted extrapolation as the Poisson solve's guess
        {"name": "step_cylinder_h32", "kind": "step", "geom": "circle", "n": 32, "prec": "mixed", "rtol": 1e-12,
         "steps": 2, "extrap": 0.9},
        # the headline workload: bumpy cylinder, 2.1M nodes, MIXED, extrapolated guess
        {"name": "step_bumpy_h64", "kind": "step", "geom": "bumpy", "n": 64, "prec": "mixed", "rtol": 1e-12,
         "steps": 2, "extrap": 0.7},
        # a batch of closed triangular cavities in one context, in the form chosen there
        {"name": "step_triangles16", "kind": "step", "geom": "triangles", "n": 256, "count": 16, "prec": "fp64",
         "rtol": 1e-12, "steps": 2},
        # one pressure solve from a zero guess, as a caller with its own stepping asks for
        {"name": "solve_cavity256", "kind": "solve", "n": 256, "which": "POISSON", "prec": "fp64", "rtol": 1e-12},
        # the operators alone, as force probes and diagnostics use them
        {"name": "apply_cylinder_h32", "kind": "apply", "geom": "circle", "n": 32},
        # set-up of a channel at an ordinary resolution (every parity trial pays for it)
        {"name": "build_cylinder_h16", "kind": "build", "geom": "circle", "n": 16},
        # set-up of a jittered walled 3D box and its operators
        {"name": "build3d_box40", "kind": "build3d", "n": 40},
        # the 3D step: ABC flow on the periodic cube, and the lid-driven walled cube
        {"name": "step3d_abc32", "kind": "step3d", "flow": "abc", "n": 32, "rtol": 1e-12, "steps": 2},
        {"name": "step3d_lid30", "kind": "step3d", "flow": "lid", "n": 30, "rtol": 1e-12, "steps": 1},
        # the solve without device allocation, at its largest size
        {"name": "static_512x256", "kind": "static", "nx": 512, "ny": 256, "rtol": 1e-12},
        # one training sample of the warm-start network on the h = 1/32 channel's lattice
        {"name": "network_h32", "kind": "network", "h": 513, "w": 1025},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "solve", "apply", "build", "build3d", "step3d", "step3d",
                       "static", "network"])
    c = {"kind": kind}
    if kind == "step":
        c["geom"] = rng.choice(["cavity", "circle", "bumpy", "triangles"])
        if c["geom"] == "cavity":
            c.update(n=_log_int(rng, 24, 320), prec=rng.choice(["fp64", "mixed", "mg32"]), rtol=1e-12)
        elif c["geom"] == "triangles":
            c.update(n=_log_int(rng, 72, 300), count=rng.randint(2, 20), prec="fp64", rtol=1e-12)
        else:
            lo, hi = (6, 52) if c["geom"] == "circle" else (16, 56)
            c.update(n=_log_int(rng, lo, hi), prec=rng.choice(["mixed", "mixed", "fp64"]), rtol=1e-12,
                     extrap=round(rng.uniform(0.0, 1.0), 2))
        c["steps"] = rng.randint(1, 2)
    elif kind == "solve":
        c.update(n=_log_int(rng, 24, 320), which=rng.choice(["POISSON", "HELM_U"]),
                 prec=rng.choice(["fp64", "mixed"]), rtol=1e-12)
    elif kind in ("apply", "build"):
        c["geom"] = rng.choice(["circle", "cavity"])
        hi = (52 if kind == "apply" else 24) if c["geom"] == "circle" else 400
        c["n"] = _log_int(rng, 6 if c["geom"] == "circle" else 24, hi)
    elif kind == "build3d":
        c["n"] = _log_int(rng, 6, 44)
    elif kind == "step3d":
        c["flow"] = rng.choice(["abc", "lid"])
        c.update(n=_log_int(rng, 8, 44) if c["flow"] == "abc" else _log_int(rng, 6, 30), rtol=1e-12,
                 steps=1 if c["flow"] == "lid" else rng.randint(1, 2))
    elif kind == "static":
        c["nx"] = _log_int(rng, 8, 512)
        c.update(ny=_log_int(rng, 8, min(512, 131072 // c["nx"])), rtol=1e-12)
    else:
        c.update(h=_log_int(rng, 5, 513), w=_log_int(rng, 16, 1025))
    return c


# ---- node sets and fields -----------------------------------------------------
def _nodes2d(c):
    if c["geom"] == "cavity":
        return [workloads.cavity(c["n"], Re=1000.0)]
    if c["geom"] == "circle":
        return [workloads.channel_body(1.0 / c["n"], ("circle", 0.5), Re=100.0)]
    if c["geom"] == "bumpy":
        return [workloads.channel_body(1.0 / c["n"], ("sines", 1.0, [(0.05, 12), (0.02, 31)]), Re=200.0)]
    return workloads.triangle_batch(c["count"], lo=64, hi=c["n"])


def _stream(c, rng):
    """psi(x, y) of the initial field: vortices that vanish with their gradient at the
    walls of closed domains; uniform flow around the body plus wake vortices."""
    a = rng.uniform(-1.0, 1.0, 5)
    if c["geom"] == "cavity":
        def psi(x, y):
            w = np.sin(np.pi * x) * np.sin(np.pi * y)
            return 0.15 * w * w * (a[0] + a[1] * np.cos(np.pi * x) + a[2] * np.cos(np.pi * y)
                                   + a[3] * np.sin(2 * np.pi * x) + a[4] * np.sin(2 * np.pi * y))
    elif c["geom"] == "triangles":
        c30, s30 = math.cos(math.pi / 6), 0.5

        def psi(x, y):
            w = -y * (x * c30 + y * s30) * (-(x - 1.0) * c30 + y * s30)
            return 40.0 * w * w * (a[0] + a[1] * x + a[2] * y + a[3] * x * y + a[4] * x * x)
    else:
        cx, cy = rng.uniform(1.5, 12.0, 5), rng.uniform(-3.0, 3.0, 5)

        def psi(x, y):
            th = np.arctan2(y, x)
            rb = 0.5 if c["geom"] == "circle" else 1.0 + 0.05 * np.sin(12 * th) + 0.02 * np.sin(31 * th)
            d = np.maximum(np.hypot(x, y) - rb, 0.0)
            s = y * (1.0 - np.exp(-4.0 * d * d))
            for k in range(5):
                s = s + 0.15 * a[k] * np.exp(-2.0 * ((x - cx[k]) ** 2 + (y - cy[k]) ** 2))
            return s
    return psi


def _field2d(c, ns, rng):
    psi = _stream(c, rng)
    i = np.nonzero(ns.kind == workloads.KIND_INTERIOR)[0]
    x, y, e = ns.x[i], ns.y[i], 1e-5
    u, v = ns.u0.copy(), ns.v0.copy()
    u[i] = (psi(x, y + e) - psi(x, y - e)) / (2 * e)
    v[i] = -(psi(x + e, y) - psi(x - e, y)) / (2 * e)
    return u, v


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _wave(seed, x, y, z=0.0, k=2.0):
    """A smooth field of unit size with seeded wave numbers near k and phases."""
    a = np.random.default_rng(seed).uniform(0.5, 1.5, 6)
    return (np.sin(k * a[0] * x + a[1]) * np.cos(k * a[2] * y + a[3]) * np.cos(k * a[4] * z + a[5])
            + 0.5 * np.cos(k * (a[5] * x - a[4] * y + a[3] * z)))


# ---- prepare --------------------------------------------------------------------
def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _prepare_step(c, seed):
    nss = _nodes2d(c)
    rng = np.random.default_rng(seed)
    ctx = vip.solver_for(nss, precision=PREC[c["prec"]], rtol=c["rtol"], max_iters=50000, set_state=False)
    if c["geom"] in ("circle", "bumpy"):
        ctx.vip_set_multigrid(1.0, 1.8)
        ctx.vip_ws_extrapolation(c["extrap"])
        ctx.vip_ws_enable(2)
    f = [_field2d(c, ns, rng) for ns in nss]
    u, v = _dev(np.concatenate([a for a, _ in f])), _dev(np.concatenate([b for _, b in f]))
    return {"kind": "step", "ctx": ctx, "in": (u, v, torch.zeros_like(u)), "steps": c["steps"],
            "out": [torch.empty_like(u) for _ in range(4)]}


def _solution(c, n, seed):
    """A field with smooth and rough parts, and mu = 0."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(-1.0, 1.0, 3)
    ns = workloads.cavity(n)
    x = (a[0] * np.cos(np.pi * ns.x) * np.cos(2 * np.pi * ns.y) + a[1] * np.cos(3 * np.pi * ns.x)
         + a[2] * ns.x * ns.y + 0.01 * rng.standard_normal(ns.n))
    if c["which"] != "POISSON":
        return x
    x[np.nonzero(ns.kind == workloads.KIND_INTERIOR)[0][0]] = 0.0  # the row that pins phi
    return np.concatenate([x, [0.0]])


def _prepare_solve(c, seed):
    ctx = vip.solver_for(workloads.cavity(c["n"], Re=1000.0), set_state=False)
    xs = _solution(c, c["n"], seed)
    b = ctx.vip_apply(c["which"], xs)
    return {"kind": "solve", "ctx": ctx, "b": b, "x0": np.zeros_like(b), "which": c["which"],
            "prec": PREC[c["prec"]], "rtol": c["rtol"]}


def _field_for_apply(nss, seed):
    """The field, with a zero for the unknown mu of each closed geometry."""
    f = _wave(seed, np.concatenate([s.x for s in nss]), np.concatenate([s.y for s in nss]))
    closed = sum(1 for s in nss if not (s.kind == workloads.KIND_OUTLET).any())
    return _dev(np.concatenate([f, np.zeros(closed)])), f.size


def _prepare_apply(c, seed):
    nss = _nodes2d(c)
    ctx = vip.solver_for(nss, set_state=False)
    f, n = _field_for_apply(nss, seed)
    return {"kind": "apply", "ctx": ctx, "f": f, "n": n, "out": _apply_buffers(f, n)}


def _apply_buffers(f, n):
    return {k: torch.empty_like(f if k == "POISSON" else f[:n]) for k in ("LAPLACE", "GX", "GY", "POISSON", "HELM_U")}


def _prepare_build(c, seed):
    nss = _nodes2d(c)
    f, n = _field_for_apply(nss, seed)
    return {"kind": "build", "nss": nss, "f": f, "n": n, "out": _apply_buffers(f, n)}


def _box3d(c):
    return workloads.box3d(c["n"], jitter=0.25, seed=13)


def _prepare_build3d(c, seed):
    ns = _box3d(c)
    f = _dev(_wave(seed, ns.x, ns.y, ns.z, k=6.0))
    return {"kind": "build3d", "ns": ns, "f": f,
            "out": {k: torch.empty_like(f) for k in ("LAPLACE", "GX", "GY", "GZ", "NEUMANN")}}


def _prepare_step3d(c, seed):
    rng = np.random.default_rng(seed)
    a = rng.uniform(0.5, 1.0, 3)
    if c["flow"] == "abc":
        ns = workloads.box3d(c["n"], periodic=True, length=2 * np.pi)
        x, y, z = ns.x, ns.y, ns.z
        u = a[0] * np.sin(z) + a[2] * np.cos(y)
        v = a[1] * np.sin(x) + a[0] * np.cos(z)
        w = a[2] * np.sin(y) + a[1] * np.cos(x)
        Re, dt = 10.0, 0.02
    else:
        ns = _box3d(c)
        x, y, z = np.pi * ns.x, np.pi * ns.y, np.pi * ns.z
        s2 = (np.sin(x) * np.sin(y) * np.sin(z)) ** 2
        u, v, w = a[0] * s2 * np.cos(y), -a[1] * s2 * np.cos(x), a[2] * s2 * np.cos(x + y)
        u = np.where(np.isclose(ns.z, 1.0), 1.0, u)
        Re, dt = 100.0, 0.01
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(Re, dt, c["rtol"], 50000)
    return {"kind": "step3d", "ctx": b, "in": [_dev(k) for k in (u, v, w, np.zeros_like(u))], "steps": c["steps"]}


def _static_rows(c):
    """5-point convection-diffusion rows on an nx x ny grid: (offsets, weights)."""
    return ((0, 0), 4.05), ((-1, 0), -1.3), ((1, 0), -0.7), ((0, -1), -1.1), ((0, 1), -0.9)


def _prepare_static(c, seed):
    nx, ny = c["nx"], c["ny"]
    j, i = np.divmod(np.arange(nx * ny), nx)
    xs = np.random.default_rng(seed).standard_normal(nx * ny)
    cols, vals, keep = [], [], []
    for (dx, dy), wgt in sorted(_static_rows(c), key=lambda t: t[0][1] * nx + t[0][0]):
        ok = (i + dx >= 0) & (i + dx < nx) & (j + dy >= 0) & (j + dy < ny)
        cols.append(np.where(ok, (j + dy) * nx + i + dx, 0))
        vals.append(np.full(nx * ny, wgt))
        keep.append(ok)
    cols, vals, keep = (np.stack(t, 1) for t in (cols, vals, keep))
    b = (np.where(keep, vals, 0.0) * xs[cols]).sum(1)
    ptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    return {"kind": "static", "n": nx * ny, "ptr": _dev(ptr), "col": _dev(cols[keep].astype(np.int32)),
            "val": _dev(vals[keep]), "b": _dev(b), "x": torch.empty(nx * ny, dtype=torch.float64, device=DEV),
            "rtol": c["rtol"]}


def _network_data(c, seed):
    rng = np.random.default_rng(seed)
    h, w = c["h"], c["w"]
    flat = []
    for ci, co in zip(NET[:-1], NET[1:]):
        flat += [rng.standard_normal(9 * ci * co) * np.sqrt(2.0 / (9 * ci)), 0.1 * rng.standard_normal(co)]
    g = torch.Generator().manual_seed(int(seed))
    x = torch.zeros(h, w, 16)
    x[..., :6] = torch.randn(h, w, 6, generator=g)  # six input channels, the rest padding
    target = torch.randn(h, w, generator=g)
    mask = (torch.rand(h, w, generator=g) > 0.05).float()
    return np.concatenate(flat).astype(np.float32), x.to(DEV), target.to(DEV), mask.to(DEV)


def _prepare_network(c, seed):
    flat, x, target, mask = _network_data(c, seed)
    ctx = vip.solver_for(workloads.cavity(24, Re=100.0), set_state=False)
    ctx.vip_ws_params(flat)
    return {"kind": "network", "ctx": ctx, "x": x, "target": target, "mask": mask, "h": c["h"], "w": c["w"],
            "y": torch.empty_like(target), "grads": torch.empty(flat.size, device=DEV)}


# ---- run ------------------------------------------------------------------------
def run(state):
    return globals()["_run_" + state["kind"]](state)


def _run_step(s):
    ctx = s["ctx"]
    ctx.vip_set_state(*s["in"])
    ctx.vip_step(s["steps"])
    ctx.vip_get_state(*s["out"])
    return dict(zip(("u", "v", "p", "phi"), s["out"]))


def _run_solve(s):
    x, _, _ = s["ctx"].vip_solve(s["which"], s["b"], s["x0"], precision=s["prec"], rtol=s["rtol"], max_iters=50000)
    return {"x": x}


def _apply_all(ctx, s):
    for k, y in s["out"].items():
        ctx.vip_apply(k, s["f"] if k == "POISSON" else s["f"][:s["n"]], y)
    return s["out"]


def _run_apply(s):
    return _apply_all(s["ctx"], s)


def _run_build(s):
    ctx = vip.solver_for(s["nss"], set_state=False)
    out = _apply_all(ctx, s)
    ctx.close()
    return out


def _run_build3d(s):
    b = vip.build3d_for(s["ns"])
    for k, y in s["out"].items():
        b.vip_3d_apply(k, s["f"], y)
    b.close()
    return s["out"]


def _run_step3d(s):
    b = s["ctx"]
    b.vip_3d_set_state(*s["in"])
    b.vip_3d_step(s["steps"])
    return dict(zip(("u", "v", "w", "p", "phi"), b.vip_3d_get_state()))


def _run_static(s):
    s["x"].zero_()
    st, _, _ = vip.vip_bicgstab_static(0, None, s["n"], s["ptr"], s["col"], s["val"], s["b"], s["x"],
                                       rtol=s["rtol"])
    return {"x": s["x"], "status": st}


def _run_network(s):
    ctx, loss = s["ctx"], ctypes.c_double()
    ctx._check(ctx.L.vip_ws_eval(ctx.h, s["h"], s["w"], s["x"].data_ptr(), s["y"].data_ptr(), s["grads"].data_ptr(),
                                 s["target"].data_ptr(), s["mask"].data_ptr(), ctypes.byref(loss)))
    return {"y": s["y"], "grads": s["grads"], "loss": loss.value}


# ---- work -----------------------------------------------------------------------
def work(case):
    """Bytes: fields read and written once.  Flops: one application of each operator
    the path needs (the number of Krylov iterations is a property of the method)."""
    c = case
    if c["kind"] == "network":
        n = c["h"] * c["w"]
        macs = sum(9 * ci * co for ci, co in zip(NET[:-1], NET[1:]))
        return {"bytes": n * (16 + 1 + 1 + 1) * 4, "flops": n * 2.0 * (3 * macs - 9 * 16 * 32)}
    if c["kind"] == "static":
        n = c["nx"] * c["ny"]
        return {"bytes": n * (5 * 12 + 8 + 16), "flops": n * 10.0}
    if c["kind"] == "solve":
        n = c["n"] ** 2
        return {"bytes": n * 24, "flops": n * 26.0}
    if c["kind"] == "build3d":
        n = (c["n"] + 1) ** 3
        return {"bytes": n * (57 + 6 * 8), "flops": n * 7 * (45 * 110.0 + 600.0)}
    if c["kind"] == "step3d":
        n = c["n"] ** 3 if c["flow"] == "abc" else (c["n"] + 1) ** 3
        return {"bytes": c["steps"] * n * 9 * 8, "flops": c["steps"] * n * 2.0 * 45 * (18 + 12 + 4)}
    if c["geom"] == "cavity":
        n = c["n"] ** 2
    elif c["geom"] == "triangles":
        n = c["count"] * 0.43 * (0.5 * (64 + c["n"])) ** 2
    else:
        n = 512.0 * c["n"] ** 2
    if c["kind"] == "step":
        return {"bytes": c["steps"] * n * 7 * 8, "flops": c["steps"] * n * 2.0 * (190 + 34 + 47 + 3 * 13)}
    if c["kind"] == "apply":
        return {"bytes": n * (2 + 5) * 8, "flops": n * 2.0 * (13 + 18 + 16 + 13 + 13)}
    return {"bytes": n * (41 + 5 * 8), "flops": n * 5 * 2.0 * (13 * 60)}


# ---- exact ----------------------------------------------------------------------
def exact(case, seed):
    c = case
    if c["kind"] == "solve":
        return {"x": _solution(c, c["n"], seed)}
    if c["kind"] == "static":
        return {"x": np.random.default_rng(seed).standard_normal(c["nx"] * c["ny"]), "status": None}
    if c["kind"] in ("apply", "build"):
        return _exact_operators(_nodes2d(c)[0], seed)
    if c["kind"] == "build3d":
        s = _box3d(c)
        f = _dev(_wave(seed, s.x, s.y, s.z, k=6.0))
        xyz, h, nrm = (_dev(np.stack(t, 1)) for t in ((s.x, s.y, s.z), (s.h,), (s.nx, s.ny, s.nz)))
        inside = _dev(s.kind == workloads.KIND_INTERIOR)
        lap, grad, wall = _mls_operators(xyz, h[:, 0], nrm, inside, f)
        return {"LAPLACE": lap, "GX": grad[0], "GY": grad[1], "GZ": grad[2], "NEUMANN": wall}
    if c["kind"] == "network":
        return _exact_network(c, seed)
    return None  # a whole fractional step: minutes in plain numpy


def _exact_operators(s, seed):
    f = _dev(_wave(seed, s.x, s.y))
    xy, h, nrm = (_dev(np.stack(t, 1)) for t in ((s.x, s.y), (s.h,), (s.nx, s.ny)))
    h, kind = h[:, 0], _dev(s.kind)
    inside, outlet = kind == workloads.KIND_INTERIOR, kind == workloads.KIND_OUTLET
    lap, grad, wall = _mls_operators(xy, h, nrm, inside, f)
    scale = -4.0 / (h * h)
    pois = torch.where(inside, lap, scale * torch.where(outlet, f, wall))
    if not bool(outlet.any()):  # closed: the first interior row pins phi, its equation is the last row
        pin = int(torch.nonzero(inside)[0])
        pois = torch.cat([pois, lap[pin:pin + 1]])
        pois[pin] = scale[pin] * f[pin]
    helm = torch.where(inside, f - s.dt / (2.0 * s.Re) * lap, torch.where(kind == workloads.KIND_WALL, f, wall))
    return {"LAPLACE": lap, "GX": grad[0], "GY": grad[1], "POISSON": pois, "HELM_U": helm}


def _mls_operators(x, h, nrm, inside, f):
    """Laplacian at every node, the differences across each pair of points half a
    spacing away (interior) and q - 4/3 q(x - h n) + 1/3 q(x - 2 h n) (boundary)."""
    d = x.shape[1]
    lap = sum(_mls(x, h, x, h, f, [1 + d + a * d - a * (a - 1) // 2 for a in range(d)])) * 2.0
    grad = []
    for a in range(d):
        e = torch.zeros_like(x)
        e[:, a] = 0.5 * h
        lo, hi = (_mls(x, h, (x + sg * e)[inside], h[inside], f, [0])[0] for sg in (-1, 1))
        g = torch.zeros_like(f)
        g[inside] = (hi - lo) / h[inside]
        grad.append(g)
    b, wall = ~inside, torch.zeros_like(f)
    q1, q2 = (_mls(x, h, (x - m * h[:, None] * nrm)[b], h[b], f, [0])[0] for m in (1, 2))
    wall[b] = f[b] - 4.0 / 3.0 * q1 + 1.0 / 3.0 * q2
    return lap, grad, wall


def _mls(x, h, pts, hp, f, which, support=2.2):
    """Moving least squares (quadratic basis, cubic spline weight, dilation support * h)
    of f at pts: for each basis index in `which`, the coefficient in units of the
    points' own coordinates."""
    d, cs = x.shape[1], support * float(h.max()) * (1 + 1e-9)
    lo = x.min(0).values - 2 * cs
    dims = ((x.max(0).values + 3 * cs - lo) / cs).long() + 1
    stride = torch.ones(d, dtype=torch.long, device=x.device)
    for a in range(d - 2, -1, -1):
        stride[a] = stride[a + 1] * dims[a + 1]
    cell = (((x - lo) / cs).long() * stride).sum(1)
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=int(dims.prod()))
    start, cap = torch.cumsum(count, 0) - count, int(count.max())
    steps = (torch.cartesian_prod(*[torch.arange(-1, 2, device=x.device)] * d) * stride).sum(1)
    out = [[] for _ in which]
    for k in range(0, pts.shape[0], 8192):
        p, rho = pts[k:k + 8192], support * hp[k:k + 8192]
        near = (((p - lo) / cs).long() * stride).sum(1)[:, None] + steps
        slot = start[near][..., None] + torch.arange(cap, device=x.device)
        ok = (torch.arange(cap, device=x.device) < count[near][..., None]).flatten(1)
        nb = order[slot.flatten(1).clamp_max(order.numel() - 1)]
        r = (x[nb] - p[:, None]) / rho[:, None, None]
        t = r.square().sum(2).sqrt()
        w = torch.where(t <= 0.5, 2 / 3 - 4 * t ** 2 + 4 * t ** 3, 4 / 3 - 4 * t + 4 * t ** 2 - 4 / 3 * t ** 3)
        w = torch.where(ok & (t < 1.0), w, 0.0)
        basis = torch.stack([torch.ones_like(t)] + [r[..., a] for a in range(d)]
                            + [r[..., a] * r[..., b] for a in range(d) for b in range(a, d)], 2)
        wb = basis * w[..., None]
        coef = torch.linalg.solve(wb.transpose(1, 2) @ basis, (wb * f[nb][..., None]).sum(1)[..., None])[..., 0]
        for o, i in zip(out, which):
            o.append(coef[:, i] / rho ** (0 if i == 0 else 1 if i <= d else 2))
    return [torch.cat(o) for o in out]


def _exact_network(c, seed):
    """The network in 64-bit sums, with the BF16 storage of weights, activations and
    back-propagated gradients that defines it."""
    flat, x, target, mask = _network_data(c, seed)
    bf = lambda t: t.float().bfloat16().double()  # noqa: E731
    lap = torch.tensor([[0., 1, 0], [1, -4, 1], [0, 1, 0]], dtype=torch.float64, device=DEV)[None, None]
    conv, grad = torch.nn.functional.conv2d, torch.nn.grad
    layers, o, n = [], 0, len(NET) - 1
    p = torch.from_numpy(flat).to(DEV)
    for ci, co in zip(NET[:-1], NET[1:]):
        wt = bf(p[o:o + 9 * ci * co]).reshape(3, 3, ci, co).permute(3, 2, 0, 1).contiguous()
        o += 9 * ci * co
        layers.append((wt, p[o:o + co].double()))
        o += co
    acts = [bf(x).permute(2, 0, 1)[None].contiguous()]
    for k, (wt, b) in enumerate(layers):
        z = conv(acts[-1], wt, b, padding=1)
        acts.append(bf(z.clamp_min(0.0)) if k < n - 1 else z)
    y, m, t = acts[-1], mask.double()[None, None], target.double()[None, None]
    cnt = m.sum()
    d = (y.float().double() - t) * m
    r = m * conv(d, lap, padding=1)
    loss = ((r * r).sum() + LAM * (d * d).sum()) / cnt
    gy, grads = bf(2.0 * m * (conv(r, lap, padding=1) + LAM * d) / cnt), []
    for k in range(n - 1, -1, -1):
        wt = layers[k][0]
        gw = grad.conv2d_weight(acts[k], wt.shape, gy, padding=1)
        grads = [gw.permute(2, 3, 1, 0).reshape(-1), gy.sum((0, 2, 3))] + grads
        if k:
            gy = bf(grad.conv2d_input(acts[k].shape, wt, gy, padding=1) * (acts[k] > 0))
    return {"y": y[0, 0], "grads": torch.cat(grads), "loss": float(loss)}
