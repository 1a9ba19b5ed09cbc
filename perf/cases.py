"""What this framework is timed on: passes through its public entry points.

A solver pass starts a lattice (from a signed-distance field, or from its six
macroscopic fields), advances it and reads the six fields back, as a program that
runs one simulation does.  The surrogate passes are one convolution layer with its
adjoints, the gradients of a whole training batch, and one network hop.

The starting states are interfaces (circular drops and bubbles, or a flat layer)
carried by a smooth flow, so that every field is well above the rounding of the
populations it is a moment of.  Everything is drawn from the seed; `exact` restates
the method in plain 64-bit torch from the equations.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

from paper_2402_15752_gb300 import Batch, Simulation
from paper_2402_15752_gb300 import surrogate as sg

FIELDS6 = ("phi", "ux", "uy", "p", "c1", "c2")


# ------------------------------------------------------------------- cases --
def _solver(name=None, **kw):
    c = dict(kind="solver", nx=64, ny=64, precision="fp32", q=5, walls="none", visc=0, physics="drops",
             start="macros", where="device", steps=64, conserved=False, scalar_model=0, grad_scheme=0)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the droplet configuration: the smallest lattice, where each step is a launch
        _solver("droplet64_fp32", nx=64, ny=64, steps=256),
        # the layered channel of the paper (15 x 150, y walls, viscosity by
        # concentration), run in FP64 to steady state: the smallest FP64 lattice
        _solver("channel15x150_fp64", nx=15, ny=150, precision="fp64", walls="y", visc=1, physics="layer", steps=128),
        # the planar configuration: a long channel of 8 rows between walls in x
        _solver("planar1024x8_fp32", nx=1024, ny=8, walls="x", physics="layer", steps=128),
        # an ordinary ragged box: odd sides, D2Q9 scalars, body forces
        _solver("ragged333x257_q9_fp32", nx=333, ny=257, q=9, walls="y", visc=1, physics="layer", steps=64),
        # the benchmark's rising bubble end to end: the distance field in from
        # page-locked host memory, 20 steps, six FP32 fields back into it
        _solver("bubble1024x2048_fp32_host", nx=1024, ny=2048, walls="xy", visc=2, physics="bubble", start="sdf",
                where="host", steps=20),
        # the same bubble with 16-bit population storage, on the device
        _solver("bubble1024x2048_bf16", nx=1024, ny=2048, precision="bf16", walls="xy", visc=2, physics="bubble",
                steps=20),
        # a half-size bubble in FP64, the precision a result is checked in, with the
        # conserved sums that such a run is watched with
        _solver("bubble512x1024_fp64", nx=512, ny=1024, precision="fp64", walls="xy", visc=2, physics="bubble",
                steps=10, conserved=True),
        # the largest configuration: droplets in an 8192 x 8192 periodic box
        _solver("droplets8192_fp32", nx=8192, ny=8192, steps=6),
        # many lattices of uneven sizes at once (the batched configuration's sides)
        dict(name="batched64_fp32", kind="batched", cases=64, lo=64, hi=512, step=32, q=5, steps=32),
        # one hidden layer of the surrogate, forward and both adjoints, at the
        # training batch (16 samples of 256 x 256)
        dict(name="conv_layer_b16_256", kind="conv", batch=16, h=256, w=256, dilation=4),
        # the gradients of a training batch of the whole network
        dict(name="net_grads_b16_256", kind="grads", batch=16, h=256, w=256),
        # one 16-step hop of the network for 64 lattices, from fields to fields
        dict(name="net_hop_b64_256", kind="hop", batch=64, h=256, w=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solver",) * 6 + ("batched", "conv", "grads", "hop"))
    if kind == "solver":
        precision = rng.choice(("fp32", "fp32", "fp32", "fp64", "bf16", "fp16"))
        nodes = _log(rng, 2e3, 2.5e5 if precision == "fp64" else 6e6)
        aspect = math.exp(rng.uniform(math.log(0.25), math.log(4.0)))
        nx = max(15, int(math.sqrt(nodes * aspect)))
        ny = max(8, nodes // nx)
        physics = rng.choice(("drops", "layer", "bubble"))
        variant = precision in ("fp32", "fp64") and physics == "drops" and rng.random() < 0.3
        return _solver(
            nx=nx, ny=ny, precision=precision, q=rng.choice((5, 5, 9)),
            walls={"drops": "none", "layer": rng.choice(("x", "y")), "bubble": "xy"}[physics],
            visc={"drops": 0, "layer": 1, "bubble": 2}[physics], physics=physics,
            steps=max(5, min(200, int(2.0e7 / (nx * ny) / (8 if precision == "fp64" else 1)))),
            conserved=precision == "fp64" and rng.random() < 0.5, scalar_model=int(variant and rng.random() < 0.5), grad_scheme=int(variant))
    if kind == "batched":
        lo = 16 * rng.randint(2, 10)
        return dict(kind="batched", cases=rng.randint(3, 96), lo=lo, hi=lo + 16 * rng.randint(1, 22),
                    step=rng.choice((16, 17, 32)), q=rng.choice((5, 5, 9)), steps=rng.randint(5, 40))
    h = 8 * rng.randint(4, 40)
    w = 128 * rng.randint(1, 3)
    b = max(1, min(_log(rng, 1, 48), (1 << 20) // (h * w)))
    if kind == "conv":
        return dict(kind="conv", batch=b, h=h, w=w, dilation=rng.choice((1, 2, 4, 8)))
    return dict(kind=kind, batch=b, h=h, w=w)


# ------------------------------------------------------------------ inputs --
def _params(case, r):
    """Lattice-unit parameters of a solver case (the ranges of the seeded
    configurations: density ratio up to 100 for drops, 10 for the layered channel,
    1000 for the bubble)."""
    p = dict(nx=case["nx"], ny=case["ny"], wall_x=int("x" in case["walls"]), wall_y=int("y" in case["walls"]),
             scalar_q=case["q"], W=4.0, M=0.01, sigma=0.01, A=0.1, visc_model=case["visc"], visc_beta=0.0,
             gx=0.0, gy=0.0, g_rho_ref=0.0, Fx=0.0, Fy=0.0, scalar_model=case["scalar_model"],
             grad_scheme=case["grad_scheme"])
    if case["physics"] == "drops":
        ratio = r.uniform(1.0, 100.0)
        p.update(rho1=1.0, rho2=1.0 / ratio, mu1=0.1, mu2=0.1 / ratio, D1=0.1, D2=0.1 / r.uniform(1.0, 100.0),
                 Keq=r.uniform(0.5, 5.0))
    elif case["physics"] == "layer":
        p.update(rho1=r.uniform(2.0, 10.0), rho2=1.0, mu1=1.0, mu2=0.1, D1=0.5, D2=r.uniform(0.1, 0.5), Keq=1.0,
                 Fx=1e-6, Fy=-1e-6)
    else:
        p.update(rho1=1.0, rho2=1e-3, mu1=0.1, mu2=1e-3, D1=0.01, D2=0.05, Keq=1.0 / 33.0, gy=-1e-6, g_rho_ref=1.0,
                 visc_beta=r.uniform(0.1, 2.0))
    return p


def _grid(nx, ny):
    y = torch.arange(ny, dtype=torch.float64, device="cuda").view(ny, 1)
    x = torch.arange(nx, dtype=torch.float64, device="cuda").view(1, nx)
    return x, y


def _sdf(physics, walls, nx, ny, r):
    """Signed distance of the initial interface: phase 1 where it is positive."""
    x, y = _grid(nx, ny)
    if physics == "layer":  # a flat layer across the walled direction, slightly wavy
        s = r.uniform(0.35, 0.65)
        amp = r.uniform(0.5, 1.5)
        if walls == "x":
            return s * nx - x + amp * torch.cos(2 * math.pi * (y / ny + r.random()))
        return s * ny - y + amp * torch.cos(2 * math.pi * (x / nx + r.random()))
    side = min(nx, ny)
    if physics == "bubble":
        return torch.hypot(x - nx * r.uniform(0.45, 0.55), y - ny * r.uniform(0.25, 0.4)) - side * r.uniform(0.12, 0.2)
    out = None
    for _ in range(r.randint(1, 4)):  # periodic drops
        dx, dy = x - nx * r.random(), y - ny * r.random()
        dx, dy = dx - nx * torch.round(dx / nx), dy - ny * torch.round(dy / ny)
        l = side * r.uniform(0.1, 0.2) - torch.hypot(dx, dy)
        out = l if out is None else torch.maximum(out, l)
    return out


def _modes(nx, ny, r, walls):
    """Wave numbers and phases of a smooth field: sines that vanish at walls, else
    periodic waves, no longer than four times the short side."""
    side = 4 * min(nx, ny)
    out = []
    for n, wall in ((nx, "x" in walls), (ny, "y" in walls)):
        k = r.choice((1, 2)) * max(1, round(n / side))
        out.append((math.pi * k / n, 0.5) if wall else (2 * math.pi * k / n, r.random() * n))
    return out


def _flow(nx, ny, r, speed, walls):
    """A divergence-free velocity: two cells of stream functions, no flow through walls."""
    x, y = _grid(nx, ny)
    ux = uy = 0.0
    for _ in range(2):
        (kx, x0), (ky, y0) = _modes(nx, ny, r, walls)
        a = speed * r.choice((-1, 1)) * r.uniform(0.5, 1.0) / max(kx, ky)
        ux = ux + a * ky * torch.sin(kx * (x + x0)) * torch.cos(ky * (y + y0))
        uy = uy - a * kx * torch.cos(kx * (x + x0)) * torch.sin(ky * (y + y0))
    return ux, uy


def _wave(nx, ny, r, amp, walls):
    """A smooth scalar field."""
    x, y = _grid(nx, ny)
    (kx, x0), (ky, y0) = _modes(nx, ny, r, walls)
    return amp * r.choice((-1, 1)) * r.uniform(0.5, 1.0) * torch.sin(kx * (x + x0)) * torch.sin(ky * (y + y0))


def _macros(case, p, sdf, r):
    """Six macroscopic fields of the starting state: [6, ny, nx] FP64."""
    nx, ny = p["nx"], p["ny"]
    # speeds a run reaches; the density-ratio-1000 bubble moves slowly
    U = 2e-4 if case["physics"] == "bubble" else 1e-2
    phi = 0.5 + 0.5 * torch.tanh(2.0 * sdf / p["W"])
    ux, uy = _flow(nx, ny, r, U, case["walls"])
    # sound waves strong enough that FP32 resolves the pressure, weak enough to leave
    # the bulk phases where they are
    amp = {"bubble": 0.1 * U * U, "layer": 3e-4, "drops": max(0.1 * U * U, 1e-4 * min(nx, ny) / 8192)}
    pr = _wave(nx, ny, r, amp[case["physics"]], case["walls"])
    a, b = (0.0, 1.0) if case["physics"] == "bubble" else (1.0, 0.2)
    return torch.stack([phi, ux, uy, pr, a * phi, b * (1.0 - phi)]).contiguous()


def _solver_inputs(case, seed):
    r = random.Random(seed)
    p = _params(case, r)
    sdf = _sdf(case["physics"], case["walls"], p["nx"], p["ny"], r).contiguous()
    if case["start"] == "sdf":
        return p, sdf, None
    return p, None, _macros(case, p, sdf, r)


def _batched_inputs(case, seed):
    r = random.Random(seed)
    out = []
    sizes = random.Random(case["cases"] * 1000 + case["lo"])  # the sides belong to the case, not to the seed
    sides = list(range(case["lo"], case["hi"] + 1, case["step"]))
    for _ in range(case["cases"]):
        c = _solver(nx=sizes.choice(sides), ny=sizes.choice(sides), q=case["q"], physics="drops")
        p = _params(c, r)
        out.append((p, _macros(c, p, _sdf("drops", "none", p["nx"], p["ny"], r), r)))
    return out


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _conv_inputs(case, seed):
    """Activations after a ReLU, He-initialised weights, a gradient of mixed sign."""
    g = _gen(seed)
    B, H, W = case["batch"], case["h"], case["w"]
    x = torch.randn((B, H, W, 48), generator=g, device="cuda").clamp_(min=0).to(torch.bfloat16)
    dy = (torch.randn((B, H, W, 48), generator=g, device="cuda") * 1e-3).to(torch.bfloat16)
    w = (torch.randn((48, 9, 48), generator=g, device="cuda") * math.sqrt(2.0 / (9 * 48))).to(torch.bfloat16)
    b = torch.randn(48, generator=g, device="cuda") * 0.1
    return x, dy, w, b


def _net_fields(case, seed):
    """Fields (phi, ux, uy, p, c1, c2) of drops in a flow, [B, 6, H, W] FP32, with
    the spreads the shipped model was normalised by."""
    r = random.Random(seed)
    d = _model()
    H, W = case["h"], case["w"]
    f = torch.empty((case["batch"], 6, H, W), dtype=torch.float32, device="cuda")
    for k in range(case["batch"]):
        sdf = _sdf("drops", "none", W, H, r)
        phi = 0.5 + 0.5 * torch.tanh(0.5 * sdf)
        spread = [1.0 / float(v) for v in d["scale"][:5]]
        rows = [phi] + list(_flow(W, H, r, spread[1], "none")) + [_wave(W, H, r, spread[3], "none")]
        keq = r.uniform(0.5, 5.0)
        den = keq * phi + (1.0 - phi)
        total = phi + 0.05 * _wave(W, H, r, spread[4], "none")
        rows += [total * keq * phi / den, total * (1.0 - phi) / den]
        f[k] = torch.stack(rows).to(torch.float32)
    return f


def _model():
    return np.load(sg.MODEL_FLOW256)


# ----------------------------------------------------------------- prepare --
def prepare(case, seed):
    kind = case["kind"]
    if kind == "solver":
        p, sdf, macros = _solver_inputs(case, seed)
        sim = Simulation(p, precision=case["precision"])
        s = dict(case=case, sim=sim, macros=macros, c=(0.0, 1.0) if case["physics"] == "bubble" else (1.0, 0.0))
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        s["dtype"] = "f64" if case["precision"] == "fp64" else "f32"
        if case["where"] == "host":  # page-locked buffers, as a program that calls often keeps them
            s["sdf"] = sdf.cpu().pin_memory()
            s["out"] = torch.zeros((6, p["ny"], p["nx"]), dtype=dt).pin_memory()
        else:
            s["sdf"] = sdf
            s["out"] = torch.zeros((6, p["ny"], p["nx"]), dtype=dt, device="cuda")
        return s
    if kind == "batched":
        inp = _batched_inputs(case, seed)
        sims = [Simulation(p, precision="fp32") for p, _ in inp]
        batch = Batch(sims)
        macros = torch.cat([m.reshape(-1) for _, m in inp])
        return dict(case=case, sims=sims, batch=batch, macros=macros,
                    out=torch.zeros(macros.numel(), dtype=torch.float32, device="cuda"))
    if kind == "conv":
        x, dy, w, b = _conv_inputs(case, seed)
        L = sg.nn_lib()
        nb = L.lbm_nn_wgrad_partial_bytes(48, 48, case["batch"], case["h"], case["w"], case["dilation"])
        wt = torch.empty_like(w)
        stream = torch.cuda.current_stream()
        sg._ck(L.lbm_nn_flip_weights(sg._p(w), 48, 48, sg._p(wt), ctypes.c_void_p(stream.cuda_stream)), "flip")
        return dict(case=case, x=x, dy=dy, w=w, wt=wt, b=b, y=torch.empty_like(x), dx=torch.empty_like(x), nb=nb,
                    dw=torch.empty((48, 9, 48), device="cuda"), db=torch.empty(48, device="cuda"),
                    part=torch.empty(nb // 4 + 1, device="cuda"), bpart=torch.empty(1024 * 48, device="cuda"),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"), stream=stream)
    sur = sg.Surrogate.load(sg.MODEL_FLOW256, "cuda")
    B, H, W = case["batch"], case["h"], case["w"]
    ws = sg.Workspace(B, H, W, "cuda", train=kind == "grads", dilations=sur.net.dil)
    s = dict(case=case, sur=sur, ws=ws, fields=_net_fields(case, seed))
    if kind == "grads":  # the target: the input's fields moved on by a little
        s["target"] = torch.roll(s["fields"], shifts=(1, 1), dims=(2, 3)).contiguous()
        s["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    else:
        s["out"] = torch.empty((B, 5, H, W), dtype=torch.float32, device="cuda")
    return s


# --------------------------------------------------------------------- run --
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solver":
        sim, out = state["sim"], state["out"]
        if case["start"] == "sdf":
            sim.init(state["sdf"], *state["c"])
        else:
            sim.init_macros(*state["macros"].unbind(0))
        sim.step(case["steps"])
        if case["where"] == "host":
            sim.fields(names=FIELDS6, dtype=state["dtype"], out=out.numpy())
        else:
            sim.fields(names=FIELDS6, dtype=state["dtype"], device=True, out=out)
        res = {n: out[i] for i, n in enumerate(FIELDS6)}
        if case["conserved"]:
            res["sums"] = sim.conserved()
        return res
    if kind == "batched":
        b = state["batch"]
        b.init_macros(state["macros"])
        b.step(case["steps"])
        b.fields(FIELDS6, state["out"])
        return state["out"]
    if kind == "conv":
        L, p = sg.nn_lib(), sg._p
        s = ctypes.c_void_p(state["stream"].cuda_stream)
        B, H, W, d = case["batch"], case["h"], case["w"], case["dilation"]
        x, dy, st = state["x"], state["dy"], state["status"]
        sg._ck(L.lbm_nn_conv3x3(p(x), 48, p(state["w"]), p(state["b"]), 48, sg.RELU, None, None, p(state["y"]),
                                B, H, W, d, p(st), s), "conv")
        sg._ck(L.lbm_nn_conv3x3_wgrad(p(x), 48, p(dy), 48, p(state["dw"]), p(state["part"]), state["nb"],
                                      B, H, W, d, p(st), s), "wgrad")
        sg._ck(L.lbm_nn_bias_grad(p(dy), 48, B * H * W, p(state["db"]), p(state["bpart"]), s), "bgrad")
        sg._ck(L.lbm_nn_conv3x3(p(dy), 48, p(state["wt"]), None, 48, sg.MASK, None, p(x), p(state["dx"]),
                                B, H, W, d, p(st), s), "dgrad")
        return {k: state[k] for k in ("y", "dx", "dw", "db")}
    sur, ws = state["sur"], state["ws"]
    sur.pack(state["fields"], ws, ws.x32, ws.x16)
    if kind == "hop":
        sur.hop(ws)
        sur.unpack(ws.y32, ws, state["out"])
        return state["out"]
    net, L, p = sur.net, sg.nn_lib(), sg._p
    sur.pack(state["target"], ws, ws.t32)
    net.forward(ws.x32, ws.x16, ws.y32, ws.acts, ws.B, ws.H, ws.W)
    sg._ck(L.lbm_nn_mse(p(ws.y32), p(ws.t32), sg.USED, ws.P, p(ws.dz16), p(ws.loss_part), p(state["loss"]), net.s), "mse")
    net.backward(ws.x16, ws.acts, ws.dz16, ws.dbuf, ws.scratch, ws.B, ws.H, ws.W)
    return {"loss": state["loss"], "gw": list(net.gw), "gb": list(net.gb)}


# -------------------------------------------------------------------- work --
def work(case):
    """Bytes and operations a pass cannot do without.  A solver step reads and
    writes each node's populations and its five previous-step macros once; the
    operations are those of the collision as written in `_Lattice.step`."""
    kind = case["kind"]
    if kind in ("solver", "batched"):
        q = case["q"]
        if kind == "solver":
            nodes, precision = case["nx"] * case["ny"], case["precision"]
        else:
            sizes = random.Random(case["cases"] * 1000 + case["lo"])
            sides = list(range(case["lo"], case["hi"] + 1, case["step"]))
            nodes, precision = sum(sizes.choice(sides) * sizes.choice(sides) for _ in range(case["cases"])), "fp32"
        size = {"fp64": 8, "fp32": 4}.get(precision, 2)
        macro = 8 if precision == "fp64" else 4
        one = (18 + 2 * q) * size + 5 * macro + (12 if size == 2 else 0)  # 16-bit: the writers' bases too
        given = 8 if kind == "solver" and case["start"] == "sdf" else 48
        fields = (18 + 2 * q) * size + 6 * macro
        return {"bytes": nodes * (given + one + 2 * one * case["steps"] + fields),
                "flops": nodes * case["steps"] * (420 + 28 * q)}
    P = case["batch"] * case["h"] * case["w"]
    if kind == "conv":  # x, dy in; y, dx out
        return {"bytes": 4 * P * 96 + 3 * 9 * 48 * 48 * 2, "flops": 3 * 2 * 9 * 48 * 48 * P}
    macs = 9 * sum(ci * co for ci, co in sg.LAYERS)
    if kind == "hop":  # the fields in, five out; each layer's activations written and read once
        return {"bytes": P * (24 + 20 + 2 * 64 + 2 * 5 * 96), "flops": 2 * macs * P}
    # forward activations written once and read by the next layer, the weight
    # gradient and the mask; each layer's gradient written once and read twice
    return {"bytes": P * (48 + 3 * 64 + 5 * 4 * 96 + 5 * 3 * 96), "flops": (3 * 2 * macs - 2 * 9 * 16 * 48) * P}


# ------------------------------------------------------------------- exact --
_C = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_W5 = (1 / 3,) + (1 / 6,) * 4


class _Lattice:
    """The coupled scheme in 64-bit torch, one array operation at a time."""

    def __init__(self, p, macros):
        self.p = p
        self.wq = _W5 if p["scalar_q"] == 5 else _W9
        ny, nx = macros.shape[1:]
        dev = macros.device
        ix, iy = torch.arange(nx, device=dev), torch.arange(ny, device=dev)
        wrap = lambda i, n, wall: i.clamp(0, n - 1) if wall else i % n  # noqa: E731
        self.nx, self.ny = nx, ny
        self.sx = {d: wrap(ix + d, nx, p["wall_x"]) for d in (-1, 1)}
        self.sy = {d: wrap(iy + d, ny, p["wall_y"]) for d in (-1, 1)}
        phi, ux, uy, pr, c1, c2 = macros
        rho = p["rho2"] + (p["rho1"] - p["rho2"]) * phi.clamp(0, 1)
        S = self._source(phi, c1, c2)
        cu = [c[0] * ux + c[1] * uy for c in _C]
        uu = ux * ux + uy * uy
        self.f = [_W9[i] * phi * (1 + 3 * cu[i]) for i in range(9)]
        self.g = [3 * pr * (_W9[i] - (i == 0)) + rho * self._s(i, cu[i], uu) for i in range(9)]
        self.h1 = [w * (c1 * (1 + 3 * cu[i]) - 0.5 * S) for i, w in enumerate(self.wq)]
        self.h2 = [w * (c2 * (1 + 3 * cu[i]) + 0.5 * S) for i, w in enumerate(self.wq)]
        self.prev = (phi, ux, uy, c1, c2)

    def _s(self, i, cu, uu):
        return _W9[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)

    def _dm(self, phi):
        den = self.p["Keq"] * self.p["D1"] * (1 - phi) + self.p["D2"] * phi
        return torch.where(den > 0, self.p["D1"] * self.p["D2"] / torch.where(den > 0, den, torch.ones_like(den)),
                           torch.zeros_like(den))

    def _source(self, phi, c1, c2):
        return self.p["A"] * self._dm(phi) * (self.p["Keq"] * c2 * phi - c1 * (1 - phi))

    def _at(self, a, dx, dy):
        if dx:
            a = a.index_select(1, self.sx[dx])
        return a.index_select(0, self.sy[dy]) if dy else a

    def _grad(self, a):
        gx = gy = 0.0
        for i in range(1, 9):
            n = self._at(a, *_C[i])
            if _C[i][0]:
                gx = gx + 3 * _W9[i] * _C[i][0] * n
            if _C[i][1]:
                gy = gy + 3 * _W9[i] * _C[i][1] * n
        return gx, gy

    def _lap(self, a):
        return sum(6 * _W9[i] * (self._at(a, *_C[i]) - a) for i in range(1, 9))

    def macros(self):
        p = self.p
        phi = sum(self.f)
        P1, P2 = sum(self.h1), sum(self.h2)
        a = 0.5 * p["A"] * self._dm(phi)
        a1, a2 = a * (1 - phi), a * p["Keq"] * phi
        c1 = (P1 + a2 * (P1 + P2)) / (1 + a1 + a2)
        c2 = (P2 + a1 * (P1 + P2)) / (1 + a1 + a2)
        px, py = self._grad(phi)
        pc = phi.clamp(0, 1)
        drho = p["rho1"] - p["rho2"]
        rho = p["rho2"] + drho * pc
        mu_phi = 48 * p["sigma"] / p["W"] * phi * (phi - 1) * (phi - 0.5) - 1.5 * p["sigma"] * p["W"] * self._lap(phi)
        Fx = mu_phi * px + (rho - p["g_rho_ref"]) * p["gx"] + p["Fx"]
        Fy = mu_phi * py + (rho - p["g_rho_ref"]) * p["gy"] + p["Fy"]
        ux = (sum(_C[i][0] * self.g[i] for i in range(1, 9) if _C[i][0]) + 0.5 * Fx) / rho
        uy = (sum(_C[i][1] * self.g[i] for i in range(1, 9) if _C[i][1]) + 0.5 * Fy) / rho
        uu = ux * ux + uy * uy
        pr = 0.6 * (sum(self.g[1:]) + 0.5 * drho * (ux * px + uy * py) - 2 / 3 * rho * uu)
        mu = p["mu2"] + (p["mu1"] - p["mu2"]) * pc
        if p["visc_model"] == 1:
            mu = torch.exp(c1 * math.log(p["mu1"]) + c2 * math.log(p["mu2"]))
        elif p["visc_model"] == 2:
            mu = mu * torch.exp(-p["visc_beta"] * (c1 + c2))
        return phi, ux, uy, pr, c1, c2, rho, mu, px, py, Fx, Fy, P1, P2

    def step(self):
        p = self.p
        phi, ux, uy, pr, c1, c2, rho, mu, px, py, Fx, Fy, P1, P2 = self.macros()
        q0, vx, vy, d1, d2 = self.prev
        wf = 1 / (3 * p["M"] + 0.5)
        w1, w2 = 1 / (3 * p["D1"] + 0.5), 1 / (3 * p["D2"] + 0.5)
        wg = 1 / (3 * mu / rho + 0.5)
        norm = torch.sqrt(px * px + py * py) + 1e-4
        nx, ny = px / norm, py / norm
        uu, drho = ux * ux + uy * uy, p["rho1"] - p["rho2"]
        t = 4 / p["W"] * phi * (1 - phi)
        t1, t2 = 4 / p["W"] * (1 - phi) * c1, 4 / p["W"] * phi * c2
        # forcing vectors of the phase field and of the two scalars
        Ax, Ay = 3 * (phi * ux - q0 * vx) + t * nx, 3 * (phi * uy - q0 * vy) + t * ny
        E1x, E1y = 3 * (c1 * ux - d1 * vx) + t1 * nx, 3 * (c1 * uy - d1 * vy) + t1 * ny
        E2x, E2y = 3 * (c2 * ux - d2 * vx) - t2 * nx, 3 * (c2 * uy - d2 * vy) - t2 * ny
        S = self._source(phi, c1, c2)
        g1x, g1y = self._grad(c1)
        g2x, g2y = self._grad(c2)
        Ht = self._dm(phi) * (px * (g1x + p["Keq"] * g2x) + py * (g1y + p["Keq"] * g2y))
        f, g, h1, h2 = [], [], [], []
        for i, (cx, cy) in enumerate(_C):
            w, cu = _W9[i], cx * ux + cy * uy
            feq = w * phi * (1 + 3 * cu)
            f.append(self.f[i] - wf * (self.f[i] - feq) + (1 - 0.5 * wf) * w * (cx * Ax + cy * Ay))
            geq = 3 * pr * (w - (i == 0)) + rho * self._s(i, cu, uu)
            G = w * (3 * (cx * Fx + cy * Fy) + 3 * drho * cu * (cx * px + cy * py))
            g.append(self.g[i] - wg * (self.g[i] - geq) + (1 - 0.5 * wg) * G)
            if i < len(self.wq):
                w = self.wq[i]
                h1.append(self.h1[i] - w1 * (self.h1[i] - w * c1 * (1 + 3 * cu)) +
                          (1 - 0.5 * w1) * w * (S + cx * E1x + cy * E1y) - w * Ht)
                h2.append(self.h2[i] - w2 * (self.h2[i] - w * c2 * (1 + 3 * cu)) +
                          (1 - 0.5 * w2) * w * (-S + cx * E2x + cy * E2y) + w * Ht)
        self.f, self.g, self.h1, self.h2 = map(self._stream, (f, g, h1, h2))
        self.prev = (phi, ux, uy, c1, c2)

    def _stream(self, a):
        out = []
        for i in range(len(a)):
            cx, cy = _C[i]
            b = torch.roll(a[i], shifts=(cy, cx), dims=(0, 1))
            # half-way bounce-back where the upstream node is behind a wall
            if cx and self.p["wall_x"]:
                k = 0 if cx > 0 else self.nx - 1
                b[:, k] = a[_OPP[i]][:, k]
            if cy and self.p["wall_y"]:
                k = 0 if cy > 0 else self.ny - 1
                b[k, :] = a[_OPP[i]][k, :]
            out.append(b)
        return out


def _solve(p, macros, steps):
    s = _Lattice(p, macros)
    for _ in range(steps):
        s.step()
    return torch.stack(s.macros()[:6])


def _conv64(x, w, d):
    """Periodic dilated 3x3 convolution, x [B, H, W, ci], w [co, 9, ci], in FP64."""
    out = 0.0
    for t in range(9):
        s = torch.roll(x, shifts=(-(t // 3 - 1) * d, -(t % 3 - 1) * d), dims=(1, 2))
        out = out + s @ w[:, t].T
    return out


def _adjoints64(x, dy, w, d):
    """(dx, dw) of sum(dy * conv(x, w))."""
    dx, dw = 0.0, []
    for t in range(9):
        oy, ox = (t // 3 - 1) * d, (t % 3 - 1) * d
        dx = dx + torch.roll(dy @ w[:, t], shifts=(oy, ox), dims=(1, 2))
        s = torch.roll(x, shifts=(-oy, -ox), dims=(1, 2))
        dw.append(dy.flatten(0, 2).T @ s.flatten(0, 2))
    return dx, torch.stack(dw, 1)


def _state64(fields, d):
    """Normalised 16-channel state of the network (5 used)."""
    shift, scale = (torch.from_numpy(np.asarray(d[k], np.float64)).cuda() for k in ("shift", "scale"))
    f = fields.double()
    v = torch.stack([f[:, 0], f[:, 1], f[:, 2], f[:, 3], f[:, 4] + f[:, 5]], -1)
    v = (v - shift[:5]) * scale[:5]
    return torch.cat([v, torch.zeros(v.shape[:-1] + (11,), dtype=v.dtype, device=v.device)], -1)


def _weights64(d):
    w = [torch.from_numpy(np.asarray(d["w%d" % l], np.float32)).cuda().to(torch.bfloat16).double() for l in range(6)]
    b = [torch.from_numpy(np.asarray(d["b%d" % l], np.float32)).cuda().double() for l in range(6)]
    return w, b, [int(v) for v in d["dilations"]]


def _net64(x, w, b, dil):
    acts = [x]
    for l in range(5):
        acts.append(torch.relu(_conv64(acts[-1], w[l], dil[l]) + b[l]))
    return x + _conv64(acts[-1], w[5], dil[5]) + b[5], acts


def exact(case, seed):
    kind = case["kind"]
    if kind == "solver":
        if case["scalar_model"] or case["grad_scheme"]:
            return None  # the paper's variants are held to the bound of their type
        p, sdf, macros = _solver_inputs(case, seed)
        if macros is None:
            c1, c2 = (0.0, 1.0) if case["physics"] == "bubble" else (1.0, 0.0)
            phi = 0.5 + 0.5 * torch.tanh(2.0 * sdf / p["W"])
            z = torch.zeros_like(phi)
            macros = torch.stack([phi, z, z, z, c1 * phi, c2 * (1.0 - phi)])
        out = _solve(p, macros, case["steps"])
        res = {n: out[i] for i, n in enumerate(FIELDS6)}
        if case["precision"] in ("bf16", "fp16"):  # 16-bit populations: the flow may be below their rounding at the start
            res["ux"] = res["uy"] = res["p"] = None
        if case["conserved"]:
            res["sums"] = torch.stack([out[0].sum(), (out[4] + out[5]).sum()])
        return res
    if kind == "batched":
        return torch.cat([_solve(p, m, case["steps"]).reshape(-1) for p, m in _batched_inputs(case, seed)])
    if kind == "conv":
        x, dy, w, b = _conv_inputs(case, seed)
        xd, dyd, wd, d = x.double(), dy.double(), w.double(), case["dilation"]
        dx, dw = _adjoints64(xd, dyd, wd, d)
        return {"y": torch.relu(_conv64(xd, wd, d) + b.double()), "dx": dx * (xd > 0), "dw": dw,
                "db": dyd.sum((0, 1, 2))}
    d = _model()
    w, b, dil = _weights64(d)
    fields = _net_fields(case, seed)
    x = _state64(fields, d)
    if kind == "hop":
        shift, scale = (torch.from_numpy(np.asarray(d[k], np.float64)).cuda()[:5] for k in ("shift", "scale"))
        out = torch.cat([_net64(x[k:k + 1], w, b, dil)[0][..., :5] / scale + shift for k in range(case["batch"])])
        return out.permute(0, 3, 1, 2).contiguous()
    t = _state64(torch.roll(fields, shifts=(1, 1), dims=(2, 3)), d)
    y, acts = _net64(x, w, b, dil)
    diff = (y - t)[..., :5]
    dz = torch.zeros_like(y)
    dz[..., :5] = 2.0 / diff.numel() * diff
    gw, gb = [None] * 6, [None] * 6
    for l in range(5, -1, -1):
        gb[l] = dz.sum((0, 1, 2))
        dx, gw[l] = _adjoints64(acts[l], dz, w[l], dil[l])
        dz = dx * (acts[l] > 0)
    return {"loss": (diff * diff).mean().reshape(1), "gw": gw, "gb": gb}
