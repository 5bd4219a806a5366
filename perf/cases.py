"""Timing cases of the wave-tank library: what a user of it runs, through its
public calls, over the range of sizes, dimensions and precisions it is used at.

Tanks are stepped the way a control loop does it: a few time steps under one
sequence of PTO forces, the step records, then the fields (sigma, velocities,
pressure), which the library hands out as host arrays.  Fields are read once per
several steps, as a program that writes snapshots does.  The solver cases are one
pressure solve, the network cases one inference and one gradient.

The single-precision-stencil tanks (WEC_PREC_MIXED) are not among the tanks: they
round the state to 32 bits in every step, so outputs after several steps say how
32-bit roundings fell and not how accurate a step is.  Their solver is the one of
the MIXED pressure solves, their stencils the ones of the other tanks.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2206_07732_gb300 import synth, wec

PREC = {"fp64": wec.PREC_FP64, "mixed": wec.PREC_MIXED, "mixed_mg": wec.PREC_MIXED_MG, "mixed_df": wec.PREC_MIXED_DF}


def listed():
    return [
        # The small regular-wave tank (4 m x 2 m, heaving box), plain method: launches and latency decide.
        dict(name="tank2 128x64 fp64", kind="tank2", nx=128, ny=64, sea="regular", prec="fp64", sweeps=2, restart=20,
             steps=20),
        # The 16 m x 4 m JONSWAP tank under a PTO force, plain method at its default solver options.
        dict(name="tank2 1024x256 fp64", kind="tank2", nx=1024, ny=256, sea="jonswap", prec="fp64", sweeps=2,
             restart=20, steps=20),
        # A shorter, deeper tank of the same sea, FP32 multigrid inside FP64 refinement at the options its tuning
        # picks (four sweeps); a size that is no power of two.
        dict(name="tank2 640x288 mixed_mg", kind="tank2", nx=640, ny=288, sea="jonswap", prec="mixed_mg", sweeps=4,
             restart=20, steps=20),
        # Twelve uneven tanks, each with its own wave and box, in one graph launch per step (a parameter study).
        dict(name="batch 12 mixed_mg", kind="batch", tanks=12, layout=0, prec="mixed_mg", steps=20),
        # The 3D tank of a closed control loop on a coarse grid: many steps, each of short kernels.
        dict(name="tank3 64x32x32 mixed_df", kind="tank3", nx=64, ny=32, nz=32, prec="mixed_df", sweeps=2, restart=20,
             steps=20),
        # A middle-sized 3D tank, plain method at its default options (the figures others are compared with).
        dict(name="tank3 256x128x128 fp64", kind="tank3", nx=256, ny=128, nz=128, prec="fp64", sweeps=2, restart=20,
             steps=4),
        # A 3D tank with a narrow basin and sizes that are no powers of two, at its tuned options.
        dict(name="tank3 224x80x112 mixed_df", kind="tank3", nx=224, ny=80, nz=112, prec="mixed_df", sweeps=3,
             restart=5, steps=8),
        # The production 3D tank (33.5 million cells) in the precision it is run at, tuned options.
        dict(name="tank3 512x256x256 mixed_df", kind="tank3", nx=512, ny=256, nz=256, prec="mixed_df", sweeps=3,
             restart=5, steps=4),
        # One 2D pressure solve on a caller's coefficients (a training sample of the learned warm start).
        dict(name="solve2 512x256 mixed", kind="solve2", nx=512, ny=256, prec="mixed", sweeps=2, restart=20),
        # One 3D pressure solve on a caller's coefficients, larger than the caches.
        dict(name="solve3 384x192x192 mixed", kind="solve3", nx=384, ny=192, nz=192, prec="mixed", sweeps=3,
             restart=5),
        # Inference of the learned warm start for the 1024x256 tank.
        dict(name="net forward 256x1024", kind="net", H=256, W=1024, batch=1),
        # One gradient of its training: batch 4 of 512x256 samples.
        dict(name="net gradient 4x256x512", kind="net_grad", H=256, W=512, batch=4),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _coarsenable(rng, lo, hi, coarse, most):
    """A size lo..hi that halves to an odd or even number of at most `most` cells, and the halvings."""
    c = rng.choice(coarse)
    k = max(0, round(math.log2(_loguniform(rng, lo, hi) / c)))
    while c << k > hi:
        k -= 1
    while c << k < lo or c << k > most << k:
        k += 1
    return c << k, k


def draw(rng):
    kind = rng.choice(["tank2", "tank2", "batch", "tank3", "tank3", "solve2", "solve3", "net", "net_grad"])
    if kind == "net":
        return dict(kind=kind, H=8 * round(_loguniform(rng, 64, 256) / 8), W=8 * round(_loguniform(rng, 128, 1024) / 8),
                    batch=rng.choice([1, 1, 2]))
    if kind == "net_grad":
        return dict(kind=kind, H=8 * round(_loguniform(rng, 64, 256) / 8), W=8 * round(_loguniform(rng, 128, 512) / 8),
                    batch=rng.choice([1, 2, 4]))
    if kind == "batch":
        return dict(kind=kind, tanks=rng.randint(3, 12), layout=rng.randint(1, 10**6), prec=rng.choice(["fp64", "mixed_mg"]), steps=rng.randint(8, 20))
    sweeps, restart = rng.choice([(2, 20), (2, 8), (3, 8), (4, 8), (4, 20), (3, 5)])
    if kind in ("tank2", "solve2"):
        nx, k = _coarsenable(rng, 128, 1024, [16, 18, 20, 22, 24, 26, 28], 28)
        cy = rng.randint(4, 12)
        ny = max(48, cy << k)
        while ny > nx // 2 and ny % 4 == 0 and ny // 2 >= 48:
            ny //= 2
        if kind == "solve2":
            return dict(kind=kind, nx=nx, ny=ny, prec=rng.choice(["fp64", "mixed"]), sweeps=sweeps, restart=restart)
        return dict(kind=kind, nx=nx, ny=ny, sea=rng.choice(["regular", "jonswap"]), prec=rng.choice(["fp64", "mixed_mg"]),
                    sweeps=sweeps, restart=restart, steps=rng.randint(8, 20))
    nx, k = _coarsenable(rng, 64, 288, [8, 10, 12, 14], 14)
    q = 1 << k
    ny = q * rng.randint(3, 5)
    nz = q * max(4, round(nx / q * rng.uniform(0.42, 0.55)))
    if kind == "solve3":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=rng.choice(["fp64", "mixed", "mixed_df"]), sweeps=sweeps,
                    restart=restart)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=rng.choice(["fp64", "mixed_df", "mixed_df"]), sweeps=sweeps,
                restart=restart, steps=rng.randint(2, 4))


# ------------------------------------------------------------------ inputs ----

def _options(cfg, case):
    cfg["solver"].update(mg_pre=case["sweeps"], mg_post=case["sweeps"], restart=case["restart"])
    return cfg


def _tank2(case, seed):
    """The JONSWAP or regular-wave tank with a heaving box, its lengths in proportion to the water column."""
    nx, ny = case["nx"], case["ny"]
    if case["sea"] == "regular" and nx == 2 * ny:
        return _options(synth.tank_small(seed=seed, nx=nx, ny=ny), case)
    c = synth.tank_large(seed=seed)
    h = 1.0 / 64.0
    lx, ly = nx * h, ny * h
    depth = 0.625 * ly
    c.update(nx=nx, ny=ny, lx=lx, ly=ly, depth=depth, damp_len=0.25 * lx, damp_x0=0.75 * lx, probe_x=0.1 * lx,
             name="tank %dx%d" % (nx, ny))
    c["body"] = synth.box_body(0.4 * lx, 0.25 * ly, 0.2 * ly, 0.1 * ly, depth, c["rho_w"])
    rng = np.random.default_rng(seed)
    scale = ly / 4.0
    if case["sea"] == "regular":
        c["wave"] = synth.regular_wave(0.05 * scale, 1.6 * math.sqrt(scale), rng)
    else:
        c["wave"] = synth.irregular_wave(0.15 * scale, 1.6 * math.sqrt(scale), 3.3, 64, rng)
    return _options(c, case)


def _batch(case, seed):
    """Uneven tanks (sizes, wave heights and periods, boxes) as the case lays them out; wave phases from the seed."""
    cfgs = synth.batch_tanks(case["tanks"], case["layout"])
    for c, phase in zip(cfgs, np.random.default_rng(seed).uniform(0, 2 * math.pi, len(cfgs))):
        c["wave"]["phase"] = float(phase)
    return cfgs


def _tank3(case, seed):
    return _options(synth.tank3d(seed=seed, nx=case["nx"], ny=case["ny"], nz=case["nz"]), case)


def _problem(case, seed):
    """Face coefficients and right-hand side of a tank's pressure equation: water below a wavy surface, air
    above, the coefficient blended over one cell, a body at its Brinkman value; walls and bed closed.  3D
    layouts (1 cell along y for a 2D problem); right-hand side standard normal."""
    nx, nz = case["nx"], case.get("nz", case["ny"])
    ny = case["ny"] if "nz" in case else 1
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = np.random.default_rng(seed)
    lx = 8.0
    h = lx / nx
    depth = 0.5 * nz * h
    k, ph = 2 * math.pi * r.uniform(0.2, 2.0, 32), r.uniform(0, 2 * math.pi, 32)
    a = r.rayleigh(1.0, 32)
    a *= 0.2 / (4 * math.sqrt(0.5 * np.sum(a * a)))
    ctr = lambda n: (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h  # noqa: E731
    face = lambda n: torch.arange(n + 1, device="cuda", dtype=torch.float64) * h  # noqa: E731
    kk, pp, aa = (torch.from_numpy(v).cuda() for v in (k, ph, a))

    def field(z, y, x):
        eta = depth + (aa * torch.cos(kk * x[:, None] + pp)).sum(1)
        s = (0.5 + (z[:, None, None] - eta) / h).clamp(0, 1).expand(len(z), len(y), len(x))
        beta = (1 - s) * synth.BETA3_WATER + s * synth.BETA3_AIR
        near = (x - 0.5 * lx).abs()[None, :] if ny == 1 else torch.hypot(x[None, :] - 0.5 * lx, y[:, None] - 0.5 * ny * h)
        body = (near < 0.5)[None] & ((z - depth).abs() < 0.4)[:, None, None]
        return torch.where(body, synth.BETA3_BODY, beta).contiguous()

    bx, by, bz = field(ctr(nz), ctr(ny), face(nx)), field(ctr(nz), face(ny), ctr(nx)), field(face(nz), ctr(ny), ctr(nx))
    bx[:, :, 0] = bx[:, :, nx] = 0
    by[:, 0] = by[:, ny] = 0
    bz[0] = 0
    return bx, by, bz, torch.randn(nz, ny, nx, device="cuda", dtype=torch.float64, generator=g)


def _samples(case, seed):
    """Features and targets as the tank's pressure problems give them: right-hand side over its rms, log density
    by region (water 0, air, the body), target of order one; and the weights."""
    B, H, W = case["batch"], case["H"], case["W"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(B, H, W, 2, device="cuda", generator=g)
    y = (torch.arange(H, device="cuda") + 0.5)[None, :, None] / H
    wave = torch.rand(B, 1, 1, device="cuda", generator=g) * 6.283 + torch.arange(W, device="cuda")[None, None] * 0.05
    x[..., 1] = torch.where(y > 0.6 + 0.05 * torch.sin(wave), math.log(1025.0 / 1.225) / 4.0, 0.0)
    x[:, H // 2:H // 2 + H // 5, W // 3:W // 3 + W // 8, 1] = math.log(1025.0 * 1e-8 / 5e-4) / 4.0
    t = torch.randn(B, H // 8, W // 8, device="cuda", generator=g)
    t = F.interpolate(t[:, None], size=(H, W), mode="bilinear")[:, 0].contiguous()
    return x, t, synth.unet_weights(wec.net_param_shapes(), seed)


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed + 1)
    if kind == "tank2":
        cfg = _tank2(case, seed)
        return dict(kind=kind, tank=wec.Tank(cfg, precision=PREC[case["prec"]]), steps=case["steps"], dt=cfg["dt"],
                    pto=rng.uniform(-50, 50, case["steps"]))
    if kind == "batch":
        cfgs = _batch(case, seed)
        return dict(kind=kind, batch=wec.Batch(cfgs, precision=PREC[case["prec"]]), steps=case["steps"],
                    dt=np.array([c["dt"] for c in cfgs]), pto=rng.uniform(-20, 20, (case["steps"], case["tanks"])))
    if kind == "tank3":
        cfg = _tank3(case, seed)
        return dict(kind=kind, tank=wec.Tank3(cfg, precision=PREC[case["prec"]]), steps=case["steps"], dt=cfg["dt"],
                    pto=rng.uniform(-200, 200, case["steps"]))
    if kind in ("solve2", "solve3"):
        bx, by, bz, b = _problem(case, seed)
        opt = dict(precision=PREC[case["prec"]], restart=case["restart"], mg_pre=case["sweeps"], mg_post=case["sweeps"])
        if kind == "solve2":
            P = wec.Poisson(case["nx"], case["ny"], **opt)
            P.set_coefficients(bx.contiguous(), bz.contiguous())
        else:
            P = wec.Poisson3(case["nx"], case["ny"], case["nz"], **opt)
            P.set_coefficients(bx, by, bz)
        return dict(kind=kind, P=P, b=b, x=torch.empty_like(b))
    x, t, w = _samples(case, seed)
    net = wec.Net(case["H"], case["W"], case["batch"])
    net.set_params(w)
    return dict(kind=kind, net=net, x=x, t=t, out=torch.empty_like(t))


# -------------------------------------------------------------------- passes ----

def _records(recs):
    return {k: np.array([r[k] for r in recs]) for k in ("t", "z", "zdot", "f_hydro", "eta_probe")}


def run(state):
    kind = state["kind"]
    if kind == "tank2":
        tank = state["tank"]
        recs = tank.step_n(state["steps"], state["dt"], state["pto"])
        return {"records": _records(recs), "fields": [tank.get(f) for f in ("sigma", "u", "v", "p")]}
    if kind == "batch":
        batch = state["batch"]
        recs = batch.step_n(state["steps"], state["dt"], state["pto"])
        return {"records": _records(recs), "fields": [[t.get(f) for f in ("sigma", "u", "v", "p")] for t in batch.tanks]}
    if kind == "tank3":
        tank = state["tank"]
        recs = [tank.step(state["dt"], f) for f in state["pto"]]
        return {"records": _records(recs), "fields": [tank.get(f) for f in (wec.F3_SIGMA, wec.F3_U, wec.F3_V, wec.F3_W,
                                                                              wec.F3_P)]}
    if kind in ("solve2", "solve3"):
        state["x"].zero_()
        state["P"].solve(state["b"], state["x"])
        return state["x"]
    net = state["net"]
    if kind == "net":
        net.forward(state["x"], state["out"])
        return state["out"]
    return {"loss": net.loss_grad(state["x"], state["t"]), "grads": net.grads()}


def work(case):
    """Tanks: the state (level set, velocities, pressure) read and written once per step, in FP64.  Solves: the
    coefficients and the right-hand side read, the solution written.  Networks: inputs, weights and outputs, and
    the multiply-adds of the convolutions (three times those of a forward pass for a gradient)."""
    kind = case["kind"]
    if kind in ("net", "net_grad"):
        px = case["batch"] * case["H"] * case["W"]
        n = sum(int(np.prod(s)) for s in wec.net_param_shapes())
        fl = sum(wec.net_layer_flops(case["H"], case["W"], case["batch"]))
        if kind == "net":
            return {"bytes": 12.0 * px + 4.0 * n, "flops": fl}
        return {"bytes": 12.0 * px + 8.0 * n, "flops": 3.0 * fl}
    if kind == "batch":
        cells = float(sum(c["nx"] * c["ny"] for c in _batch(case, 0)))
    else:
        cells = float(case["nx"] * case["ny"] * case.get("nz", 1))
    if kind in ("solve2", "solve3"):
        return {"bytes": 8.0 * cells * (4 if kind == "solve2" else 5), "flops": 0.0}
    return {"bytes": 16.0 * cells * (5 if kind == "tank3" else 4) * case["steps"], "flops": 0.0}


# ------------------------------------------------------- 64-bit values ----

def _solution(case, seed):
    """The pressure equation solved by Jacobi-preconditioned conjugate gradients to rounding."""
    bx, by, bz, b = _problem(case, seed)
    top = bz[-1]

    def apply(p):
        fx, fz = bx[:, :, 1:-1] * (p[:, :, 1:] - p[:, :, :-1]), bz[1:-1] * (p[1:] - p[:-1])
        y = torch.zeros_like(p)
        y[:, :, :-1] -= fx
        y[:, :, 1:] += fx
        y[:-1] -= fz
        y[1:] += fz
        if p.shape[1] > 1:
            fy = by[:, 1:-1] * (p[:, 1:] - p[:, :-1])
            y[:, :-1] -= fy
            y[:, 1:] += fy
        y[-1] += 2 * top * p[-1]
        return y

    d = bx[:, :, 1:] + bx[:, :, :-1] + by[:, 1:] + by[:, :-1] + bz[1:] + bz[:-1]
    d[-1] += top
    if b.shape[1] == 1:
        d -= by[:, 1:] + by[:, :-1]
    x, r = torch.zeros_like(b), b.clone()
    z = r / d
    p, rz = z.clone(), (r * z).sum()
    stop = 1e-14 * b.norm().item()
    for i in range(20000):
        q = apply(p)
        alpha = rz / (p * q).sum()
        x += alpha * p
        if i % 500 == 499:
            r = b - apply(x)
        else:
            r -= alpha * q
        if i % 50 == 49 and r.norm().item() <= stop:
            break
        z = r / d
        rz, old = (r * z).sum(), rz
        p = z + (rz / old) * p
    return x


def _network(w, x):
    """The network in 64 bits on parameters w (weights and bias in turn, [kh, kw, cin, cout]): its output."""
    def conv(h, k, stride=1, pad=1):
        return F.relu(F.conv2d(h, w[k].permute(3, 2, 0, 1), w[k + 1], stride=stride, padding=pad))

    h, skips, k = x.permute(0, 3, 1, 2), [], 0
    for level in range(4):
        if level:
            h = conv(h, k, 2, 0)
            k += 2
        h = conv(conv(h, k), k + 2)
        k += 4
        skips.append(h)
    for level in (2, 1, 0):
        h = conv(F.interpolate(h, scale_factor=2, mode="nearest"), k)
        h = conv(conv(torch.cat([h, skips[level]], 1), k + 2), k + 4)
        k += 6
    return (h.permute(0, 2, 3, 1) @ w[k])[..., 0] + w[k + 1]


def exact(case, seed):
    """Solves and networks in plain torch.  The tanks have none: their step is a whole two-phase flow solver, not
    an expression of torch or numpy."""
    kind = case["kind"]
    if kind in ("solve2", "solve3"):
        return _solution(case, seed)
    if kind not in ("net", "net_grad"):
        return None
    x, t, flat = _samples(case, seed)
    x, t, flat = x.double(), t.double(), torch.from_numpy(flat).cuda().double()
    shapes = wec.net_param_shapes()
    w = [v.reshape(s) for v, s in zip(torch.split(flat, [int(np.prod(s)) for s in shapes]), shapes)]
    if kind == "net":
        with torch.no_grad():
            return _network(w, x)
    w = [v.clone().requires_grad_() for v in w]
    loss = ((_network(w, x) - t) ** 2).mean()
    return {"loss": float(loss), "grads": torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, w)])}
