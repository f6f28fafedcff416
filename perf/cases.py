"""The work a user has this solver do, as cases that can be timed.

A case is a dict of plain values.  `prepare` makes what a program holds before
the call (speeds on the device, the solver context or the batch, the output
buffers), `run` is one pass through the public entry points, `exact` is the same
result in 64 bits from plain torch (Jacobi iteration of the upwind equations to
their fixed point), and `work` is what a pass cannot do without.

Kinds of case:
  solve   one grid: [new speeds ->] solve -> psi, on the device or from and to
          pinned host memory
  batch   many grids of uneven sizes in one launch, every grid's psi
  train   one pass of the restart-schedule network: forward and gradient
"""
from __future__ import annotations

import math
import random

import torch

import paper_1811_00009_gb300 as eik

BIG = 1e30                 # "not reached" inside the 64-bit iteration


def _solve(name, dims, family, precision="fp32", stride_h=2.0, block=8, sources=1, io="device", new_speed=False,
           window=0.0):
    return {"name": name, "kind": "solve", "nx": dims[0], "ny": dims[1], "nz": dims[2], "family": family,
            "precision": precision, "stride_h": stride_h, "block": block, "sources": sources, "io": io,
            "new_speed": new_speed, "window": window}


def listed():
    """stride_h 0 is the learned schedule (eik_solve(ctx, 0, 0)), the way the benchmark's workload is solved."""
    return [
        # the smallest grid of the batched configuration, alone: launches and latency
        _solve("tiny_32", (32, 32, 32), "grf"),
        # the FP64 verification configuration: 64^3, F = 1, block 16, stride 2h
        _solve("verify_fp64_64", (64, 64, 64), "const", precision="fp64", block=16),
        # an odd, ragged survey box with several sources and speeds that change before every solve
        _solve("ragged_97x61x130", (97, 61, 130), "grf", stride_h=0.0, block=0, sources=3, new_speed=True),
        # the paper's barrier case (shells of F = 0 with holes)
        _solve("barriers_128", (128, 128, 128), "shells"),
        # an inversion or planning service: speeds from host memory, travel times back to it
        _solve("host_io_160", (160, 160, 160), "sines", io="host", new_speed=True),
        # double precision in earnest on a mid-sized random medium
        _solve("fp64_192", (192, 192, 192), "grf", precision="fp64"),
        # the FP32 sines configuration: 256^3, block 16, stride 2h
        _solve("sines_256", (256, 256, 256), "sines", block=16),
        # 32^3 blocks with the stride and window the benchmark gives them
        _solve("block32_320", (320, 320, 320), "grf", stride_h=4.0, block=32, window=4.0),
        # the layered FP32 configuration at full size, learned schedule
        _solve("layers_512", (512, 512, 512), "layers", stride_h=0.0, block=0),
        # the benchmark's workload at full size: 1024^3 random medium, learned schedule
        _solve("grf_1024", (1024, 1024, 1024), "grf", stride_h=0.0, block=0),
        # the batched configuration: 64 grids, edges 32..192, 1-4 sources, the three families
        {"name": "batch_64", "kind": "batch", "grids": 64, "lo": 32, "hi": 192, "step": 16, "layout": 5,
         "precision": "fp32"},
        # training the schedule network: one full-size training batch, forward and gradient
        {"name": "train_32768", "kind": "train", "samples": 32768},
    ]


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["batch", "batch", "train"])
    if kind == "train":
        return {"kind": "train", "samples": int(round(math.exp(rng.uniform(math.log(257), math.log(100000)))))}
    if kind == "batch":
        grids = rng.randint(3, 64)
        lo = rng.randint(17, 48)
        return {"kind": "batch", "grids": grids, "lo": lo, "hi": rng.randint(lo + 16, 192), "step": rng.choice([1, 3, 16]),
                "layout": rng.randrange(1 << 30), "precision": rng.choice(["fp32", "fp32", "fp32", "fp64"])}
    stride, block, window, largest = rng.choice([(0.0, 0, 0.0, 640), (0.0, 0, 0.0, 640), (1.5, 8, 0.0, 640),
                                                 (2.0, 8, 0.0, 560), (3.0, 8, 0.0, 280), (2.0, 16, 0.0, 360),
                                                 (4.0, 32, 4.0, 480)])
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    if precision == "fp64":
        largest = 220
        if block == 32:
            stride, block, window = 2.0, 16, 0.0
    base = math.exp(rng.uniform(math.log(24), math.log(largest)))
    dims = [max(9, int(round(base * math.exp(rng.uniform(-0.4, 0.4))))) for _ in range(3)]
    c = _solve("", dims, rng.choice(["const", "sines", "layers", "grf", "grf", "shells"]), precision, stride, block,
               rng.choice([1, 1, 2, 4]), rng.choice(["device", "device", "device", "host"]), rng.random() < 0.5, window)
    del c["name"]
    return c


# ---- inputs ----

def _spacing(dims):
    return 1.0 / (max(dims) - 1)


def _speed(dims, family, seed, dtype):
    """Speeds of a family on the device, shape (nz, ny, nx): the longest axis spans [0, 1]."""
    nx, ny, nz = dims
    h = _spacing(dims)
    dev = torch.device("cuda")
    rnd = random.Random(seed)
    if family == "const":
        return torch.full((nz, ny, nx), rnd.uniform(0.5, 2.0), dtype=dtype, device=dev)
    if family == "layers":
        vals = torch.tensor([rnd.uniform(0.5, 2.0) for _ in range(16)], dtype=dtype, device=dev)
        layer = (16 * torch.arange(nz, device=dev)) // nz
        return vals[layer][:, None, None].expand(nz, ny, nx).contiguous()
    if family == "grf":
        # exp of a Gaussian random field: white noise smoothed by a periodic Gaussian, std 0.5, length 0.05
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        W = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=gen, device=dev))
        s = 0.05 / math.sqrt(2.0)
        for axis, n in enumerate((nz, ny, nx)):
            f = torch.fft.rfftfreq(n, d=h, device=dev) if axis == 2 else torch.fft.fftfreq(n, d=h, device=dev)
            shape = [1, 1, 1]
            shape[axis] = f.numel()
            W *= torch.exp(-2.0 * (math.pi * s * f) ** 2).reshape(shape)
        g = torch.fft.irfftn(W, s=(nz, ny, nx))
        del W
        g -= g.mean()
        g *= 0.5 / g.std(unbiased=False)
        return g.exp_().to(dtype)
    x, y, z = (torch.arange(n, dtype=torch.float64, device=dev) * h for n in (nx, ny, nz))
    if family == "sines":
        ph = [rnd.uniform(0.0, 1.0) for _ in range(3)]
        sx, sy, sz = (torch.sin(2.0 * math.pi * (c + p)) for c, p in zip((x, y, z), ph))
        return (1.0 + 0.5 * sz[:, None, None] * sy[None, :, None] * sx[None, None, :]).to(dtype)
    # shells: F = c, with four spherical barriers (F = 0) that leave a hole around an axis
    c = [0.5 * (n - 1) * h for n in (nx, ny, nz)]
    X, Y, Z = (x - c[0])[None, None, :], (y - c[1])[None, :, None], (z - c[2])[:, None, None]
    R = torch.sqrt(X * X + Y * Y + Z * Z)
    rad = torch.sqrt(X * X + Y * Y) + 0.0 * Z
    F = torch.full((nz, ny, nx), rnd.uniform(0.5, 2.0), dtype=torch.float64, device=dev)
    for r0, hole, up in ((0.15, 0.05, False), (0.25, 0.10, True), (0.35, 0.10, False), (0.45, 0.10, True)):
        open_ = (rad < hole) & ((Z > 0) if up else (Z < 0))
        F[(R > r0) & (R < r0 + 1.0 / 24.0) & ~open_] = 0.0
    return F.to(dtype)


def _sources(dims, count, seed):
    """count points in the grid's box (one source: near the centre), physical coordinates."""
    h = _spacing(dims)
    rnd = random.Random(seed * 7919 + 11)
    if count == 1:
        return [[(0.5 + rnd.uniform(-0.03, 0.03)) * (n - 1) * h for n in dims]]
    return [[rnd.uniform(0.0, 1.0) * (n - 1) * h for n in dims] for _ in range(count)]


def _batch_layout(case):
    """(dims, family, sources) of every grid; the layout is the case's, the values come from the seed."""
    rnd = random.Random(case["layout"])
    edges = list(range(case["lo"], case["hi"] + 1, case["step"]))
    return [([rnd.choice(edges) for _ in range(3)], rnd.choice(["sines", "layers", "grf"]), rnd.randint(1, 4))
            for _ in range(case["grids"])]


def _dims(case):
    return [case["nx"], case["ny"], case["nz"]]


def _dtype(case):
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def _train_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B = case["samples"]
    w = torch.randn(eik.SCHED_PARAMS, generator=gen, device="cuda") * 0.2
    X = torch.rand((B, eik.SCHED_INPUTS), generator=gen, device="cuda") * 2.0 - 0.5
    act = torch.randint(0, eik.SCHED_ACTIONS, (B,), generator=gen, device="cuda", dtype=torch.int32)
    tgt = torch.randn(B, generator=gen, device="cuda")
    return w, X, act, tgt


def prepare(case, seed):
    if case["kind"] == "train":
        w, X, act, tgt = _train_inputs(case, seed)
        B = case["samples"]
        return {"case": case, "w": w, "X": X, "act": act, "tgt": tgt,
                "Y": torch.empty((B, eik.SCHED_ACTIONS), device="cuda"),
                "grad": torch.empty(eik.SCHED_PARAMS, device="cuda"), "loss": torch.empty(1, device="cuda"),
                "work": torch.empty(eik.eik_mlp_work_floats(B), device="cuda")}
    dt = _dtype(case)
    if case["kind"] == "batch":
        grids, outs = [], []
        for i, (dims, family, count) in enumerate(_batch_layout(case)):
            s = seed * 1000 + i
            grids.append((dims, _spacing(dims), _speed(dims, family, s, dt), _sources(dims, count, s)))
            outs.append(torch.empty(dims[::-1], dtype=dt, device="cuda"))
        return {"case": case, "batch": eik.Batch(grids, case["precision"]), "outs": outs}
    dims = _dims(case)
    F = _speed(dims, case["family"], seed, dt)
    out = torch.empty_like(F)
    if case["io"] == "host":
        F, out = F.cpu().pin_memory(), torch.empty(F.shape, dtype=dt, pin_memory=True)
    S = eik.Solver(dims, _spacing(dims), F, case["precision"])
    S.add_sources(_sources(dims, case["sources"], seed))
    return {"case": case, "solver": S, "out": out, "F": F if case["new_speed"] else None}


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        eik.eik_mlp_forward(state["w"], state["X"], state["Y"])
        eik.eik_mlp_grad(state["w"], state["X"], state["act"], state["tgt"], state["grad"], state["loss"],
                         state["work"])
        return [state["Y"], state["grad"], state["loss"]]
    if case["kind"] == "batch":
        B = state["batch"]
        B.solve()
        return [B.result(i, out) for i, out in enumerate(state["outs"])]
    S = state["solver"]
    if state["F"] is not None:
        eik.eik_set_speed(S.ctx, state["F"], case["precision"])
    S.solve(case["stride_h"] * S.h, block_dim=case["block"], window=case["window"])
    return S.result(state["out"])


def work(case):
    """Speeds read once and psi written once; one upwind solve per node (about 30 operations)."""
    if case["kind"] == "train":
        B, n_in, hid, act = case["samples"], eik.SCHED_INPUTS, eik.SCHED_HIDDEN, eik.SCHED_ACTIONS
        macs = n_in * hid + hid * hid + act * hid
        return {"bytes": 4 * (2 * B * n_in + B * act + 2 * B + 3 * eik.SCHED_PARAMS), "flops": 2 * B * (4 * macs)}
    size = 4 if case["precision"] == "fp32" else 8
    if case["kind"] == "batch":
        nodes = sum(d[0] * d[1] * d[2] for d, _, _ in _batch_layout(case))
    else:
        nodes = case["nx"] * case["ny"] * case["nz"]
    return {"bytes": 2 * size * nodes, "flops": 30 * nodes}


# ---- the same results in 64 bits ----

def _cell(t, n):
    """Nodes of the cell that holds coordinate t (in cells): one if t is a node, else two."""
    if abs(t - round(t)) <= 1e-9:
        return [min(max(int(round(t)), 0), n - 1)]
    i = min(max(int(math.floor(t)), 0), max(n - 2, 0))
    return sorted({i, min(i + 1, n - 1)})


def _exact_psi(F, h, sources):
    """Greatest fixed point of the upwind equations, from Jacobi sweeps in float64."""
    nz, ny, nx = F.shape
    F = F.double()
    r = torch.where(F > 0, h / F, torch.full_like(F, BIG))
    P = torch.full((nz + 2, ny + 2, nx + 2), BIG, dtype=torch.float64, device=F.device)
    psi = P[1:-1, 1:-1, 1:-1]
    for s in sources:
        for k in _cell(s[2] / h, nz):
            for j in _cell(s[1] / h, ny):
                for i in _cell(s[0] / h, nx):
                    f = float(F[k, j, i])
                    d = math.sqrt((i * h - s[0]) ** 2 + (j * h - s[1]) ** 2 + (k * h - s[2]) ** 2)
                    if f > 0 or d == 0.0:
                        psi[k, j, i] = min(float(psi[k, j, i]), d / f if d > 0 else 0.0)
                        r[k, j, i] = BIG
    del F
    r2 = r * r
    for it in range(8 * (nx + ny + nz)):
        mx = torch.minimum(P[1:-1, 1:-1, :-2], P[1:-1, 1:-1, 2:])
        my = torch.minimum(P[1:-1, :-2, 1:-1], P[1:-1, 2:, 1:-1])
        mz = torch.minimum(P[:-2, 1:-1, 1:-1], P[2:, 1:-1, 1:-1])
        lo, hi = torch.minimum(mx, my), torch.maximum(mx, my)
        a, t = torch.minimum(lo, mz), torch.maximum(lo, mz)
        b, c = torch.minimum(hi, t), torch.maximum(hi, t)
        d, e = b - a, c - a
        x = a + r
        x2 = a + 0.5 * (d + (2.0 * r2 - d * d).clamp_(min=0.0).sqrt_())
        x = torch.where(x > b, x2, x)
        x3 = a + (d + e + (3.0 * r2 - (d * d + e * e + (c - b) ** 2)).clamp_(min=0.0).sqrt_()) / 3.0
        x = torch.minimum(torch.where(x > c, x3, x), psi)
        done = it % 16 == 15 and bool((psi - x <= 1e-15 * psi).all())
        psi.copy_(x)
        if done:
            break
    return torch.where(psi < 0.5 * BIG, psi, torch.full_like(psi, math.inf))


def _sweeps(dims):
    return dims[0] * dims[1] * dims[2] * (dims[0] + dims[1] + dims[2])


def exact(case, seed):
    if case["kind"] == "train":
        w, X, act, tgt = _train_inputs(case, seed)
        n_in, hid, n_act = eik.SCHED_INPUTS, eik.SCHED_HIDDEN, eik.SCHED_ACTIONS
        w = w.double().requires_grad_(True)
        sizes = [hid * n_in, hid, hid * hid, hid, n_act * hid, n_act]
        W1, b1, W2, b2, W3, b3 = torch.split(w, sizes)
        y = torch.tanh(X.double() @ W1.view(hid, n_in).T + b1)
        y = torch.tanh(y @ W2.view(hid, hid).T + b2)
        y = y @ W3.view(n_act, hid).T + b3
        loss = (y.gather(1, act.long()[:, None])[:, 0] - tgt.double()).square().mean()
        loss.backward()
        return [y.detach(), w.grad, loss.detach().reshape(1)]
    dt = _dtype(case)
    if case["kind"] == "batch":
        layout = _batch_layout(case)
        if sum(_sweeps(d) for d, _, _ in layout) > 4.5e10:
            return None
        out = []
        for i, (dims, family, count) in enumerate(layout):
            s = seed * 1000 + i
            out.append(_exact_psi(_speed(dims, family, s, dt), _spacing(dims), _sources(dims, count, s)))
        return out
    dims = _dims(case)
    if _sweeps(dims) > 4.5e10:
        return None
    psi = _exact_psi(_speed(dims, case["family"], seed, dt), _spacing(dims), _sources(dims, case["sources"], seed))
    return psi.cpu() if case["io"] == "host" else psi
