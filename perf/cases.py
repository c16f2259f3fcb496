"""Performance cases: the sweeps a user of this library runs, through its public entry points.

Three kinds of call are covered.
  * "run":     so2dr.Plan(...).run(host_grid): the sweep on a pinned host grid, out of core (mode 0) under a
               device budget or in core (mode 1).  The whole call counts, host copies included.
  * "adjoint": Plan.adjoint(...): loss and gradients of the variable-coefficient sweep, host to host.
  * "device":  so2dr_run_device_noalloc: the sweep on a grid that already sits on the device.

A case is a dict of plain values: path, kind (star, box, varcoef), r, dtype, n0, ny, nx (ny = 0: a 2D grid of
n0 x nx), T time steps, k_on, k_off (0: the planner's choice), budget (bytes), chunks (least number), mode,
and ckpt (adjoint: steps between checkpoints).
"""
import ctypes
import math

import numpy as np
import torch

from paper_2309_08864_gb300 import so2dr

GIB = 1 << 30
MIB = 1 << 20
TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
SIZE = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}


def _case(name, path, kind, r, dtype, dims, T, k_on=0, k_off=0, budget=0, chunks=1, mode=0, ckpt=0):
    n0, ny, nx = dims if len(dims) == 3 else (dims[0], 0, dims[1])
    c = dict(path=path, kind=kind, r=r, dtype=dtype, n0=n0, ny=ny, nx=nx, T=T, k_on=k_on, k_off=k_off,
             budget=budget, chunks=chunks, mode=mode, ckpt=ckpt)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a short sweep of a small 3D grid that lives on the device (three launches), as in a
        # loop that alternates the sweep with other device work
        _case("device-7pt-f32-small", "device", "star", 1, "f32", (48, 80, 132), 10, k_on=4),
        # a device-resident sweep in double precision, odd sizes: a verification or convergence run
        _case("device-13pt-f64-odd", "device", "star", 2, "f64", (150, 131, 157), 8, k_on=2),
        # 2D 5-point Jacobi in double precision under a 1 MiB budget: the smallest out-of-core run
        _case("ooc-jacobi2d-f64-512", "run", "star", 1, "f64", (512, 512), 16, k_on=4, k_off=8, budget=MIB, chunks=4),
        # the headline: 7-point star, FP32, 1024^3, 64 steps, 1 GiB budget, the planner's own depths
        _case("ooc-7pt-f32-1024", "run", "star", 1, "f32", (1024, 1024, 1024), 64, budget=GIB, chunks=8),
        # the radius-4 star (8th-order Laplacian style), FP32, out of core at the headline's grid-to-budget ratio
        _case("ooc-25pt-f32-768", "run", "star", 4, "f32", (768, 768, 768), 32, budget=512 * MIB),
        # the precision form: BF16 storage with FP32 arithmetic
        _case("ooc-7pt-bf16-768", "run", "star", 1, "bf16", (768, 768, 768), 128, budget=432 * MIB, chunks=8),
        # the differentiation form: gradients with checkpoints every 8 steps
        _case("adjoint-f32-256", "adjoint", "varcoef", 1, "f32", (256, 256, 256), 64, k_on=4, k_off=8,
              budget=64 * MIB, ckpt=8),
        # its forward sweep alone (parameter studies), whole grid on the device, odd sizes
        _case("incore-varcoef-f32-odd", "run", "varcoef", 1, "f32", (243, 251, 262), 32, k_on=4, k_off=32, mode=1),
        # a 7-point sweep whose rows are no multiple of 16 bytes, whole grid on the device
        _case("incore-7pt-f32-odd", "run", "star", 1, "f32", (403, 389, 405), 64, k_on=4, k_off=64, mode=1),
        # a 9-point 2D star (radius 2) of odd size, out of core
        _case("ooc-star2d-f32-odd", "run", "star", 2, "f32", (6001, 5003), 64, k_on=4, k_off=32, budget=64 * MIB,
              chunks=4),
        # the 9-point box on the 12800^2 in-core dataset, 640 steps
        _case("ooc-box9-f32-12800", "run", "box", 1, "f32", (12800, 12800), 640, budget=GIB, chunks=4),
        # the 81-point box, the most arithmetic per cell
        _case("ooc-box81-f32-8192", "run", "box", 4, "f32", (8192, 8192), 96, budget=GIB // 4, chunks=4),
    ]


def _points(c):
    nd = 3 if c["ny"] else 2
    return (2 * c["r"] + 1) ** nd if c["kind"] == "box" else 1 + 2 * nd * c["r"]


def _dims(c):
    return (c["n0"], c["ny"], c["nx"]) if c["ny"] else (c["n0"], c["nx"])


def _cells(c):
    return c["n0"] * max(1, c["ny"]) * c["nx"]


def work(case):
    cells, b, T = _cells(case), SIZE[case["dtype"]], case["T"]
    inner = math.prod(max(0, n - 2 * case["r"]) for n in _dims(case))
    if case["path"] == "adjoint":
        # reads u0, six fields and the target, writes seven gradients; forward, transposed and gradient updates
        return {"bytes": 15 * cells * b, "flops": inner * T * (19 + 19 + 18)}
    if case["kind"] == "varcoef":
        return {"bytes": 8 * cells * b, "flops": inner * T * 19}
    return {"bytes": 2 * cells * b, "flops": inner * T * 2 * _points(case)}


def _cost(c):
    """Bound used by draw(): operations, FP64 ones counted forty-fold (the device's FP64 units are few), halos and
    ragged rows four-fold."""
    w = work(c)["flops"] * (40.0 if c["dtype"] == "f64" else 1.0)
    fast = c["kind"] != "varcoef" and c["nx"] % 8 == 0 and (c["ny"] or c["kind"] == "box")
    return w * (1.0 if fast else 4.0)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    pick = rng.random()
    odd = lambda n: n if rng.random() < 0.5 else max(16, n // 16 * 16)
    if pick < 0.2:      # device-resident sweeps, up to the 32 MiB the entry point's scratch takes
        kind, nd = rng.choice([("star", 3), ("star", 3), ("star", 2), ("box", 2)])
        r = rng.choice([1, 1, 2, 3, 4])
        dtype = rng.choice(["f32", "f32", "f64", "bf16", "f16"])
        cells = _log(rng, 1 << 16, (32 * MIB) // SIZE[dtype])
        if nd == 3:
            n0, ny = _log(rng, 24, 200), _log(rng, 24, 200)
            dims = (n0, ny, odd(min(512, max(24, cells // (n0 * ny)))))
        else:
            n0 = _log(rng, 64, 2000)
            dims = (n0, odd(max(64, cells // n0)))
        k_on = rng.randint(1, {1: 4, 2: 2, 3: 2, 4: 1}[r])
        c = _case(None, "device", kind, r, dtype, dims, _log(rng, 2, 32), k_on=k_on)
        return c if _cells(c) * SIZE[dtype] <= 32 * MIB else None
    if pick < 0.3:      # gradients
        d = [_log(rng, 24, 256) for _ in range(3)]
        C = rng.choice([4, 8])
        dims = (d[0], d[1], odd(d[2]))
        plane = 4 * dims[1] * dims[2]
        return _case(None, "adjoint", "varcoef", 1, "f32", dims, C * rng.randint(1, 8), k_on=2, k_off=C,
                     budget=plane * (28 * C + dims[0]), ckpt=C)
    mode = 1 if rng.random() < 0.4 else 0
    if pick < 0.4:      # variable coefficients, forward
        dtype = rng.choice(["f32", "f32", "f64"])
        d = [_log(rng, 32, 288) for _ in range(3)]
        k_off = rng.choice([4, 8])
        c = _case(None, "run", "varcoef", 1, dtype, (d[0], d[1], odd(d[2])), k_off * rng.randint(1, 8),
                  k_on=rng.choice([1, 2, 4]), k_off=k_off, mode=mode)
        plane = SIZE[dtype] * d[1] * d[2]
        return dict(c, budget=0 if mode else plane * (7 * 4 * k_off + 4 * d[0]))
    if pick < 0.75:     # 3D stars
        kind, r = "star", rng.choice([1, 1, 1, 2, 3, 4])
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f16", "f64"])
        d = [_log(rng, 64, 1024) for _ in range(3)]
        dims = (d[0], d[1], odd(d[2]))
    else:               # 2D boxes and stars
        kind, r = rng.choice(["box", "box", "star"]), rng.choice([1, 2, 3, 4])
        dtype = rng.choice(["f32", "f32", "f32", "bf16", "f64"])
        dims = (_log(rng, 512, 12800), odd(_log(rng, 512, 12800)))
    plane = SIZE[dtype] * math.prod(dims[1:])
    # (16-bit storage rounds at every launch's end: its depth is given, so that results do not hang on the planner)
    k_on = {1: 4, 2: 2, 3: 1, 4: 1}[r] if SIZE[dtype] == 2 else 0
    budget = max(int(plane * dims[0] * rng.uniform(0.2, 0.6)), plane * (8 * r * max(1, 4 * k_on) + 16))
    return _case(None, "run", kind, r, dtype, dims, _log(rng, 4, 160), k_on=k_on, k_off=4 * k_on, budget=budget,
                 chunks=rng.randint(1, 6), mode=mode)


def draw(rng):
    while True:
        c = _draw_once(rng)
        if c and _cells(c) <= 1 << 30 and _cost(c) <= 3e11 and min(_dims(c)) > 2 * c["r"]:
            return c


# ------------------------------------------------------------------ inputs

def _weights(c):
    """The coefficient table; FP32-representable unless the storage is FP64."""
    n = _points(c)
    if c["kind"] == "star" and c["r"] == 1:
        w = np.array([0.2] * 5 if not c["ny"] else [0.4] + [0.1] * 6)
    else:
        w = np.random.RandomState(100 + n).uniform(0.5, 1.5, n)
        w /= w.sum()
    return w if c["dtype"] == "f64" else w.astype(np.float32).astype(np.float64)


def _uniform(shape, dtype, seed, stream, a=0.0, b=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000 + stream)
    u = torch.empty(shape, dtype=dtype if dtype in (torch.float64, torch.float32) else torch.float32, device="cuda")
    u.uniform_(a, b, generator=g)
    return u.to(dtype)


def _fields(c, seed):
    """The case's inputs on the device: the grid; variable coefficients: also the six face fields and the target."""
    dt = TORCH[c["dtype"]]
    u = _uniform(_dims(c), dt, seed, 1)
    if c["kind"] != "varcoef":
        if c["r"] == 1 and not c["ny"] and c["kind"] == "star":  # the Jacobi workload keeps a zero ring
            u[0], u[-1], u[:, 0], u[:, -1] = 0, 0, 0, 0
        return [u]
    f = _uniform((6,) + _dims(c), dt, seed, 2, 0.05, 0.15)
    return [u, f, _uniform(_dims(c), dt, seed, 3)] if c["path"] == "adjoint" else [u, f]


def _pin(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def prepare(case, seed):
    c = case
    if c["path"] == "device":
        u = _fields(c, seed)[0]
        w = _weights(c)
        return {"path": "device", "in": u, "out": torch.empty_like(u), "lib": so2dr.load_library(),
                "args": (len(_dims(c)), (ctypes.c_int64 * len(_dims(c)))(*_dims(c)), c["r"], so2dr.KINDS[c["kind"]],
                         (ctypes.c_double * len(w))(*w), len(w), c["T"], c["k_on"], so2dr.DTYPES[c["dtype"]])}
    host = [_pin(t) for t in _fields(c, seed)]
    plan = so2dr.Plan(_dims(c), c["r"], c["kind"], None if c["kind"] == "varcoef" else _weights(c), c["T"],
                      min_chunks=c["chunks"], k_on=c["k_on"], k_off=c["k_off"], budget_bytes=c["budget"],
                      dtype=c["dtype"])
    plan.bind(in_core=c["mode"])
    s = {"path": c["path"], "plan": plan, "host": host, "mode": c["mode"]}
    if c["path"] == "adjoint":
        s["grads"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in host[:2]]
        s["workspace"] = plan.workspace(c["ckpt"])
        s["ckpt"] = c["ckpt"]
    return s


def run(state):
    if state["path"] == "device":
        rc = state["lib"].so2dr_run_device_noalloc(
            *state["args"], ctypes.c_void_p(state["in"].data_ptr()), ctypes.c_void_p(state["out"].data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != so2dr.OK:
            raise RuntimeError(state["lib"].so2dr_last_error().decode())
        return state["out"]
    if state["path"] == "adjoint":
        u, f, target = state["host"]
        loss, _ = state["plan"].adjoint(u, f, target, state["grads"][0], state["grads"][1], state["workspace"],
                                        state["ckpt"])
        return [loss] + state["grads"]
    state["plan"].run(state["host"][0], state["host"][1] if len(state["host"]) > 1 else None, in_core=state["mode"])
    return state["host"][0]


# ------------------------------------------------------------------ exact values

def _inner(t, r, off=None):
    off = off or (0,) * t.dim()
    return t[tuple(slice(r + o, n - r + o) for n, o in zip(t.shape, off))]


def _offsets(c):
    """Offsets in coefficient-table order."""
    nd, r = (3 if c["ny"] else 2), c["r"]
    if c["kind"] == "box":
        return [(a - r, b - r) for a in range(2 * r + 1) for b in range(2 * r + 1)]
    offs = [] if c["kind"] == "varcoef" else [(0,) * nd]
    for a in range(nd):
        for j in range(1, r + 1):
            for s in (-j, j):
                offs.append(tuple(s if k == a else 0 for k in range(nd)))
    return offs


def exact(case, seed):
    c = case
    if work(c)["flops"] * 12 > 6e13:  # about 15 seconds of FP64 memory traffic
        return None
    fields = [t.double() for t in _fields(c, seed)]
    u, offs, r, T = fields[0], _offsets(c), c["r"], c["T"]
    if c["kind"] != "varcoef":
        w = _weights(c)
        for _ in range(T):
            v = _inner(u, r, offs[0]) * float(w[0])
            for o, k in zip(offs[1:], w[1:]):
                v.add_(_inner(u, r, o), alpha=float(k))
            u = u.clone()
            _inner(u, r).copy_(v)
        return u if c["path"] == "device" else u.cpu()
    f = [_inner(x, 1) for x in fields[1]]
    centre = 1.0 - sum(f)
    step = lambda x: centre * _inner(x, 1) + sum(k * _inner(x, 1, o) for k, o in zip(f, offs))
    states = [u]
    for _ in range(T):
        u = u.clone()
        _inner(u, 1).copy_(step(states[-1]))
        states = states + [u] if c["path"] == "adjoint" else [u]
    if c["path"] == "run":
        return u.cpu()
    lam = u - fields[2]
    loss = 0.5 * float((lam * lam).sum())
    grad = torch.zeros_like(fields[1])
    for t in range(T - 1, -1, -1):
        x, li = states[t], _inner(lam, 1)
        for g, o in zip(grad, offs):
            _inner(g, 1).add_(li * (_inner(x, 1, o) - _inner(x, 1)))
        new = lam.clone()
        _inner(new, 1).copy_(centre * li)
        for k, o in zip(f, offs):
            _inner(new, 1, o).add_(k * li)
        lam = new
    return [loss, lam.cpu(), grad.cpu()]
