"""The work that programs hand to this framework, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the
call (channels with their fields set, or a network with its weights and a batch),
``run`` is one pass through the public entry points, and ``exact`` computes the same
results in float64 with plain torch, written from the method's equations and sharing
no code with the library.

Kinds:
  channel  one nematic channel advanced by some LB steps, then its fields read
  batch    many uneven channels advanced together, then their fields read
  relax    director-only relaxation of a batch of cells with the convergence check
  forward  the warm-start network's prediction
  train    one optimiser step of the warm-start network
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_06610_gb300 import inputs, nh, warmstart

# the velocity of a run on 16-bit populations carries 16 bits of them; BF16 holds the paper's 1e-7
_VELOCITY = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.bfloat16, "bf16s": torch.bfloat16}


# ------------------------------------------------------------------ the cases

def _channel(name, nx, ny, nz, **kw):
    c = dict(name=name, kind="channel", nx=nx, ny=ny, nz=nz, precision="fp32", storage="f32", regime="chiral",
             walls=True, anchoring="homeotropic", dt_fd=16, steps=32, tubes=1, radius=12.0, pitch=32.0, gx=1e-5,
             diagnostics=False, tuned=False)
    c.update(kw)
    return c


def listed():
    return [
        # the tiny nematic channel of the accuracy checks: launches and latency decide
        _channel("tiny fp32", 32, 32, 16, regime="nematic", dt_fd=1, steps=20, gx=1e-6),
        # the paper's own regime (Table I viscosities, free plates, its loop order)
        _channel("table1 fp32", 64, 64, 16, regime="table1", anchoring="none", dt_fd=10, steps=100, radius=7.0,
                 pitch=14.0, gx=2e-9),
        # one skyrmion tube, director updated every step: the accurate end of the dt_FD sweep
        _channel("tube fp32 dt1", 96, 96, 32, dt_fd=1, steps=20),
        # the FP64 reference run of the same tube, which every precision sweep needs
        _channel("tube fp64 dt4", 96, 96, 32, precision="fp64", storage="f64", dt_fd=4, steps=16),
        # odd sizes, periodic in z
        _channel("ragged fp32", 151, 117, 45, walls=False, dt_fd=5, steps=40, gx=1e-8),
        # 16-bit populations on a channel whose rows are not a multiple of 128 sites
        _channel("mid bf16s", 180, 140, 50, storage="bf16s", dt_fd=8, steps=48, tubes=3),
        # the multi-tube production channel, tuned and watched as the benchmark does
        _channel("multitube fp32", 256, 256, 64, tubes=8, radius=20.0, pitch=64.0, diagnostics=True, tuned=True),
        _channel("multitube f16s", 256, 256, 64, storage="f16s", tubes=8, radius=20.0, pitch=64.0, diagnostics=True,
                 tuned=True),
        # a parameter sweep: 64 uneven channels in one batched call
        dict(name="sweep of 64", kind="batch", count=64, dt_fd=16, steps=64, most=96),
        # generating warm-start targets: relax a batch of cells, check convergence
        dict(name="relax 32 cells", kind="relax", count=32, nx=64, ny=64, nz=32, steps=100),
        # the warm start's prediction, and its training step
        dict(name="predict 8 cells", kind="forward", batch=8, nx=64, ny=64, nz=32),
        dict(name="train 8 cells", kind="train", batch=8, nx=64, ny=64, nz=32),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel"] * 6 + ["batch", "relax", "forward", "train"])
    if kind == "channel":
        regime = rng.choice(["nematic", "table1", "chiral", "chiral", "chiral"])
        storage = rng.choice(["f32", "f32", "f32", "f64", "f16s", "bf16s"])
        most = 64 * 64 * 16 * 8 if regime != "chiral" else (3e5 if storage == "f64" else 256 * 256 * 64)
        while True:
            nx, ny, nz = _spread(rng, 24, 300), _spread(rng, 24, 300), _spread(rng, 8, 90)
            if rng.random() < 0.5:
                nx = max(32, nx // 32 * 32)
            if 32 * 32 * 16 <= nx * ny * nz <= most:
                break
        sites = nx * ny * nz
        dt = rng.choice({"table1": [1, 2, 3, 5, 10, 50], "nematic": [1, 2, 4], "chiral": [1, 2, 4, 5, 7, 8, 16, 16]}[regime])
        blocks = rng.randint(2, 8)
        steps = max(dt, min(dt * blocks, int(1.3e8 / sites) // dt * dt, 16 if storage == "f64" else 200))
        steps += rng.choice([0, 0, 0, 1, 3])
        radius = 7.0 if regime == "table1" else float(rng.randint(8, 12))
        c = _channel("", nx, ny, nz, regime=regime, storage=storage, precision="fp64" if storage == "f64" else "fp32",
                     dt_fd=dt, steps=steps, radius=radius, gx=1e-6)
        if regime == "table1":
            c.update(anchoring="none", pitch=14.0, gx=2e-9)
        elif regime == "chiral":
            c.update(walls=rng.random() < 0.8, anchoring=rng.choice(["homeotropic", "homeotropic", "none"]),
                     pitch=float(rng.randint(24, 64)), tuned=rng.random() < 0.3,
                     tubes=rng.randint(1, 4) if min(nx, ny) > 120 else 1)
            c["gx"] = 10 ** rng.uniform(-7, -5) if c["walls"] else 1e-8
            c["diagnostics"] = c["walls"] and dt % 2 == 0 and rng.random() < 0.5
    elif kind == "batch":
        c = dict(kind=kind, count=rng.randint(3, 64), dt_fd=rng.choice([1, 4, 8, 16]), steps=rng.choice([16, 32, 48]),
                 most=rng.choice([48, 64, 96]))
    elif kind == "relax":
        side = 8 * rng.randint(4, 9)
        c = dict(kind=kind, count=rng.randint(1, 24), nx=side, ny=side, nz=8 * rng.randint(2, 4),
                 steps=rng.randint(20, 100))
    else:
        while True:  # the coarsest level holds a multiple of 16 voxels
            c = dict(kind=kind, batch=rng.randint(1, 8), nx=8 * rng.randint(2, 8), ny=8 * rng.randint(2, 8),
                     nz=8 * rng.randint(1, 4))
            if c["batch"] * c["nx"] * c["ny"] * c["nz"] % (16 * 512) == 0:
                break
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _smooth(rng, nx, ny, nz, walls, dev):
    """A smooth random vector field of unit size, zero at the plates."""
    z = torch.arange(nz, device=dev, dtype=torch.float64)[:, None, None]
    y = torch.arange(ny, device=dev, dtype=torch.float64)[None, :, None] * (2 * math.pi / ny)
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, None, :] * (2 * math.pi / nx)
    prof = torch.sin(math.pi * (z + 0.5) / nz) if walls else 1.0 + 0.3 * torch.sin(2 * math.pi * z / nz)
    out = []
    for _ in range(3):
        a = torch.zeros((nz, ny, nx), device=dev, dtype=torch.float64)
        for _ in range(3):
            kx, ky = int(rng.integers(0, 3)), int(rng.integers(0, 3))
            a += float(rng.uniform(0.2, 0.5)) * torch.cos(kx * x + ky * y + float(rng.uniform(0, 6.3)))
        out.append(a * prof)
    return torch.stack(out)


def _tubes(nx, ny, nz, centres, radius, dev):
    """The extruded skyrmion ansatz (radial pi-twist) about each centre."""
    y = torch.arange(ny, device=dev, dtype=torch.float64)[:, None]
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, :]
    best = torch.full((ny, nx), math.inf, device=dev, dtype=torch.float64)
    bx, by = torch.zeros_like(best), torch.zeros_like(best)
    for cx, cy in centres:
        dx = torch.remainder(x - cx + 0.5 * nx, nx) - 0.5 * nx + 0 * y
        dy = torch.remainder(y - cy + 0.5 * ny, ny) - 0.5 * ny + 0 * x
        r = torch.hypot(dx, dy)
        near = r < best
        best, bx, by = torch.where(near, r, best), torch.where(near, dx, bx), torch.where(near, dy, by)
    th = torch.where(best < radius, math.pi * (1 - best / radius), torch.zeros_like(best))
    ph = torch.atan2(by, bx)
    n = torch.stack([-torch.sin(th) * torch.sin(ph), torch.sin(th) * torch.cos(ph), torch.cos(th)])
    return n[:, None].expand(3, nz, ny, nx)


def _fields(c, seed, dev):
    """(n, u, tube centres) of a channel: its texture with a small seeded disturbance, and a developing flow."""
    rng = _gen(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    flow = 0.03 * c["gx"] / 2e-9 * 1e-6 if c["regime"] == "table1" else 2e-3
    u = flow * _smooth(rng, nx, ny, nz, c["walls"], dev)
    if c["regime"] == "nematic":
        tilt = torch.from_numpy(rng.uniform(-0.05, 0.05, (2, nz, ny, nx))).to(dev)
        n, centres = torch.cat([tilt, torch.ones((1, nz, ny, nx), device=dev, dtype=torch.float64)]), []
    else:
        apart = [(float(rng.uniform(0, nx)), float(rng.uniform(0, ny)))]
        for _ in range(10000):  # tubes that do not overlap
            if len(apart) == c["tubes"]:
                break
            p = (float(rng.uniform(0, nx)), float(rng.uniform(0, ny)))
            if all(math.hypot((p[0] - q[0] + nx / 2) % nx - nx / 2, (p[1] - q[1] + ny / 2) % ny - ny / 2)
                   >= 2 * c["radius"] for q in apart):
                apart.append(p)
        n, centres = _tubes(nx, ny, nz, apart, c["radius"], dev), apart
        n = n + 0.05 * _smooth(rng, nx, ny, nz, False, dev)
    n = n / torch.linalg.vector_norm(n, dim=0, keepdim=True)
    return n.reshape(3, -1).contiguous(), u.reshape(3, -1).contiguous(), centres


def _params(c):
    if c["regime"] == "table1":
        p, _ = inputs.table1_regime(nx=c["nx"], ny=c["ny"], nz=c["nz"], dt_fd=c["dt_fd"])
    else:
        nematic = c["regime"] == "nematic"
        p = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], shifted=True, tau=1.0, K=0.04 if nematic else 0.005,
                 q0=0.0 if nematic else 2 * math.pi / c["pitch"], W0=0.0, dt_fd=c["dt_fd"], **inputs.LESLIE_ALIGN_09)
    p.update(walls_z=c["walls"], anchoring=c["anchoring"], g=(c["gx"], 0.0, 0.0), precision=c["precision"],
             storage=c["storage"])
    return p


def _batch_params(c, seed):
    """Uneven channels as in the batched sweep: sizes by place, forces and pitches by seed."""
    sizes, rng, out = _gen(0), _gen(seed), []
    for _ in range(c["count"]):
        side = int(sizes.choice([s for s in (32, 48, 64, 96) if s <= c["most"]]))
        nz = int(sizes.choice([16, 24, 32]))
        out.append(_channel("", side, side, nz, dt_fd=c["dt_fd"], steps=c["steps"], radius=0.25 * side,
                            pitch=float(rng.uniform(nz, 2 * nz)), gx=float(10 ** rng.uniform(-7, -5))))
    return out


def _relax_params(c, seed):
    out = []
    for p, _ in inputs.warmstart_samples(c["count"], seed=seed, nx=16, ny=16, lz_choices=(8,)):
        out.append(dict(p, nx=c["nx"], ny=c["ny"], nz=c["nz"], precision="fp32", storage="f32"))
    return out


def _relax_start(c, seed, k, dev):
    rng = _gen((seed, k))
    n = _tubes(c["nx"], c["ny"], c["nz"], [(c["nx"] // 2, c["ny"] // 2)], float(rng.uniform(7, 14)), dev)
    n = n + 0.05 * _smooth(rng, c["nx"], c["ny"], c["nz"], False, dev)
    return (n / torch.linalg.vector_norm(n, dim=0, keepdim=True)).reshape(3, -1).contiguous()


def _cells(c, seed, dev):
    """A batch for the network: ansatz and target directors (FP32), scalars (q0, Lz, W0)."""
    rng = _gen(seed)
    shape = (c["nx"], c["ny"], c["nz"])
    ans, tgt, sc = [], [], []
    for k in range(c["batch"]):
        pitch = float(rng.uniform(20, 40))
        q0 = 2 * math.pi / pitch
        r = pitch * float(rng.uniform(0.3, 0.5))
        mid = [(c["nx"] // 2, c["ny"] // 2)]
        ans.append(_tubes(*shape, mid, r, dev).reshape(3, -1))
        t = _tubes(*shape, mid, 0.8 * r, dev) + 0.1 * _smooth(rng, *shape, False, dev)
        tgt.append((t / torch.linalg.vector_norm(t, dim=0, keepdim=True)).reshape(3, -1))
        sc.append([q0, float(c["nz"]), float(rng.uniform(3.0, 3.8)) * 0.005 * q0 * q0])
    return (torch.stack(ans).float().contiguous(), torch.stack(tgt).float().contiguous(),
            torch.tensor(sc, device=dev, dtype=torch.float32))


def _weights(seed):
    """Weights and Adam moments of a network in the middle of its training."""
    w = inputs.unet_init_params(seed=seed % 1000)
    rng = _gen(seed)
    return w, 1e-4 * rng.normal(size=w.size), (1e-3 * rng.uniform(0.5, 1.5, size=w.size)) ** 2


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "channel":
        ch = nh.Channel(_params(case))
        n, u, centres = _fields(case, seed, dev)
        ch.set_fields(n, u)
        if case["diagnostics"]:
            ch.set_tubes(centres)
        if case["tuned"]:
            ch.autotune()
        out = [torch.empty(k, ch.N, device=dev, dtype=torch.float64) for k in (3, 3, 1)]
        return dict(case=case, channel=ch, out=out)
    if kind == "batch":
        chans, total = [], 0
        for k, c in enumerate(_batch_params(case, seed)):
            ch = nh.Channel(_params(c))
            n, u, _ = _fields(c, seed + 7919 * (k + 1), dev)
            ch.set_fields(n, u)
            chans.append(ch)
            total += ch.N
        nh.batch_autotune(chans)
        return dict(case=case, channels=chans, out=torch.empty(7 * total, device=dev, dtype=torch.float64))
    if kind == "relax":
        chans = []
        for k, p in enumerate(_relax_params(case, seed)):
            ch = nh.Channel(p)
            ch.set_fields(_relax_start(case, seed, k, dev))
            ch.director_change()
            chans.append(ch)
        return dict(case=case, channels=chans,
                    out=torch.empty(len(chans), 3, chans[0].N, device=dev, dtype=torch.float64))
    ans, tgt, sc = _cells(case, seed, dev)
    dims = (case["nx"], case["ny"], case["nz"])
    w, m, v = _weights(seed)
    net = warmstart.WarmStartNet()
    net.params.copy_(torch.from_numpy(w))
    net.m.copy_(torch.from_numpy(m))
    net.v.copy_(torch.from_numpy(v))
    net.steps = 1000
    return dict(case=case, net=net, ansatz=ans, target=tgt, scalars=sc, dims=dims)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "channel":
        ch, out = state["channel"], state["out"]
        extra = []
        if case["diagnostics"]:
            left = case["steps"]
            while left > 0:
                ch.step(min(left, case["dt_fd"]))
                ch.diagnostics_enqueue()
                left -= case["dt_fd"]
            d = ch.diagnostics_read()
            extra = [np.array([d["mass"], d["energy"], d["max_u"], d["min_norm"], d["max_norm"]], dtype=np.float32),
                     d["centroids"].astype(np.float32)]
        else:
            ch.step(case["steps"])
        nh.nh_get_fields(ch.ctx, *out, on_device=True)
        if case["precision"] == "fp64":
            return out + extra
        return [out[0].float(), out[1].to(_VELOCITY[case["storage"]]), out[2].float()] + extra
    if kind == "batch":
        nh.batch_step(state["channels"], case["steps"])
        out, at = state["out"], 0
        for ch in state["channels"]:
            N = ch.N
            nh.nh_get_fields(ch.ctx, out[at:at + 3 * N], out[at + 3 * N:at + 6 * N], out[at + 6 * N:at + 7 * N],
                             on_device=True)
            at += 7 * N
        return [out.float()]
    if kind == "relax":
        nh.batch_relax(state["channels"], case["steps"])
        change = [ch.director_change() for ch in state["channels"]]
        for ch, o in zip(state["channels"], state["out"]):
            nh.nh_get_fields(ch.ctx, o, on_device=True)
        # the largest changes: small differences of FP32 directors
        return [state["out"].float(), np.array(change, dtype=np.float16)]
    net = state["net"]
    if kind == "forward":
        return [net.predict(state["ansatz"], state["scalars"], state["dims"])]
    loss = net.train_step(state["ansatz"], state["scalars"], state["target"], state["dims"])
    return [loss, net.params, net.m, net.v]


# ------------------------------------------------------------------ work

def work(case):
    """Bytes: the state a pass starts from and the state and fields it leaves, once each; operations: all steps."""
    kind = case["kind"]
    if kind == "channel":
        sites = case["nx"] * case["ny"] * case["nz"]
        return _step_work(sites, case["steps"], case["dt_fd"], case["storage"])
    if kind == "batch":
        sites = sum(c["nx"] * c["ny"] * c["nz"] for c in _batch_params(case, 0))
        return _step_work(sites, case["steps"], case["dt_fd"], "f32")
    if kind == "relax":
        sites = case["count"] * case["nx"] * case["ny"] * case["nz"]
        return {"bytes": sites * (12 + 12 + 12 + 12), "flops": sites * case["steps"] * 2 * 75}
    vox = case["batch"] * case["nx"] * case["ny"] * case["nz"]
    level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0]
    flops = sum(2 * 27 * ci * co * vox / 8 ** lv for (_, ci, co), lv in zip(inputs.UNET_CONV_LAYERS, level))
    weights = 4 * nh.UNet.param_count()
    if kind == "forward":
        return {"bytes": vox * 24 + weights, "flops": flops}
    return {"bytes": vox * 24 + 8 * weights, "flops": 3 * flops}


def _step_work(sites, steps, dt_fd, storage):
    store, real = {"f64": (8, 8), "f32": (4, 4), "f16s": (2, 4), "bf16s": (2, 4)}[storage]
    state = 2 * 19 * store + 2 * (3 + 3) * real + 4 * real  # populations, director and force; u and rho written
    return {"bytes": sites * (state + 7 * 8), "flops": sites * (250.0 * steps + 750.0 * (steps // dt_fd))}


# ------------------------------------------------------------------ the same in float64, from the equations

_E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1)]


def _lattice(dev):
    w = torch.tensor([(1 / 3, 1 / 18, 1 / 36)[sum(abs(v) for v in e)] for e in _E], device=dev, dtype=torch.float64)
    return torch.tensor(_E, device=dev, dtype=torch.float64), w.reshape(19, 1, 1, 1)


def _equilibrium(rho, u):
    """Deviation of the equilibrium from the weights."""
    E, w = _lattice(u.device)
    eu = torch.tensordot(E, u, 1)
    return w * (rho * (3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)) + (rho - 1))


def _lb(f, force, force_u, p):
    """One LB step of the shifted populations; force_u shifts the velocity."""
    E, w = _lattice(f.device)
    nz = f.shape[1]
    g = torch.empty_like(f)
    for i, e in enumerate(_E):
        g[i] = torch.roll(f[i], (e[2], e[1], e[0]), (0, 1, 2))
        if p["walls_z"] and e[2]:  # half-way bounce-back
            k = 0 if e[2] > 0 else nz - 1
            g[i, k] = f[_E.index(tuple(-v for v in e)), k]
    rho = 1 + g.sum(0)
    acc = torch.tensor(p["g"], dtype=f.dtype, device=f.device).reshape(3, 1, 1, 1)
    F, H = force + rho * acc, force_u + rho * acc
    u = (torch.tensordot(E.T, g, 1) + 0.5 * H) / rho
    om = 1 / p["tau"]
    eu, eF = torch.tensordot(E, u, 1), torch.tensordot(E, F, 1)
    src = w * (3 * eF + 9 * eu * eF - 3 * (u * F).sum(0))
    return g - om * (g - _equilibrium(rho, u)) + (1 - 0.5 * om) * src, u, rho


def _shift(a, b, s, p, ghost):
    """a(x + s e_b); beyond the plates the ghost: 'copy', 'zero' or 'zhat'."""
    dim = a.dim() - 1 - b
    out = torch.roll(a, -s, dim)
    if b == 2 and p["walls_z"]:
        k = a.shape[1] - 1 if s > 0 else 0
        if ghost == "copy":
            out[:, k] = a[:, k]
        else:
            out[:, k] = 0
            if ghost == "zhat":
                out[2, k] = 1
    return out


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _gradients(n, u, p):
    """Molecular field, G[b] = d_b n and U[a] = d_a u (None at rest)."""
    ghost = "zhat" if p["anchoring"] == "homeotropic" else "copy"
    lap, G, U = -6 * n, [], []
    for b in range(3):
        hi, lo = _shift(n, b, 1, p, ghost), _shift(n, b, -1, p, ghost)
        lap = lap + hi + lo
        G.append(0.5 * (hi - lo))
        if u is not None:
            U.append(0.5 * (_shift(u, b, 1, p, "zero") - _shift(u, b, -1, p, "zero")))
    curl = torch.stack([G[1][2] - G[2][1], G[2][0] - G[0][2], G[0][1] - G[1][0]])
    h = p["K"] * lap - 2 * p["K"] * p["q0"] * curl
    h[2] += p["W0"] * n[2]
    if p["walls_z"] and ghost == "copy":  # links to free plates carry no energy
        for k, side in ((0, -1), (n.shape[1] - 1, 1)):
            h[0, k] -= side * p["K"] * p["q0"] * n[1, k]
            h[1, k] += side * p["K"] * p["q0"] * n[0, k]
    return h, G, U


def _rate(n, u, p):
    h, G, U = _gradients(n, u, p)
    r = h / p["gamma1"]
    if u is not None:
        lam = p["gamma2"] / p["gamma1"]
        for m in range(3):
            for a in range(3):
                D, W = 0.5 * (U[a][m] + U[m][a]), 0.5 * (U[a][m] - U[m][a])
                r[m] += (W - lam * D) * n[a] - u[a] * G[a][m]
    return r


def _director_step(n, u, p):
    dt = p["dt_fd"]
    r = _rate(n, u, p)
    n = n + 0.5 * dt * (r + _rate(n + dt * r, u, p))
    return n / torch.linalg.vector_norm(n, dim=0, keepdim=True)


def _lc_force(n, u, p):
    h, G, U = _gradients(n, u, p)
    D = [[0.5 * (U[a][b] + U[b][a]) for b in range(3)] for a in range(3)]
    Dn = torch.stack([sum(D[a][b] * n[b] for b in range(3)) for a in range(3)])
    nDn, hn = (n * Dn).sum(0), (n * h).sum(0)
    N = ((h - hn * n) - p["gamma2"] * (Dn - nDn * n)) / p["gamma1"]
    F = torch.zeros_like(n)
    for a in range(3):
        X = _cross(G[a], n)
        for b in range(3):
            s = (p["alpha1"] * nDn * n[a] * n[b] + p["alpha2"] * n[b] * N[a] + p["alpha3"] * n[a] * N[b]
                 + p["alpha4p"] * D[a][b] + p["alpha5"] * n[b] * Dn[a] + p["alpha6"] * n[a] * Dn[b]
                 - p["K"] * (G[a] * G[b]).sum(0) - p["K"] * p["q0"] * X[b])[None]
            F[a] += 0.5 * (_shift(s, b, 1, p, "zero") - _shift(s, b, -1, p, "zero"))[0]
    return F


def _advance(p, n, u, steps):
    """n, u, rho after steps of the hybrid loop from (n, u) at rho = 1."""
    shape = (p["nz"], p["ny"], p["nx"])
    n, u = n.reshape(3, *shape), u.reshape(3, *shape)
    f = _equilibrium(torch.ones(shape, device=n.device, dtype=n.dtype), u)
    F = _lc_force(n, u, p)
    rho = None
    for s in range(1, steps + 1):
        fd = s % p["dt_fd"] == 0
        g, u, rho = _lb(f, F, F, p)
        if fd:
            old = F
            n = _director_step(n, u, p)
            F = _lc_force(n, u, p)
            if p.get("paper_order"):  # the collision of this step takes the new force
                g, _, _ = _lb(f, F, old, p)
        f = g
    return n.reshape(3, -1), u.reshape(3, -1), rho.reshape(1, -1), f


def _conv(x, w, b):
    """3x3x3 cross-correlation of [B][Z][Y][X][C], periodic in x and y, zero beyond z; w [27][cout][cin]."""
    out = b
    for t in range(27):
        dz, dy, dx = t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1
        s = torch.roll(x, (-dy, -dx), (2, 3))
        if dz:
            pad = torch.zeros_like(s[:, :1])
            s = torch.cat([s[:, 1:], pad], 1) if dz > 0 else torch.cat([pad, s[:, :-1]], 1)
        out = out + s @ w[t].T
    return torch.relu(out)


def _pool(x):
    B, Z, Y, X, C = x.shape
    return x.reshape(B, Z // 2, 2, Y // 2, 2, X // 2, 2, C).mean((2, 4, 6))


def _up(x):
    return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)


def _unet(flat, ans, sc, dims):
    nx, ny, nz = dims
    B = ans.shape[0]
    layer, at = {}, 0
    for name, ci, co in inputs.UNET_CONV_LAYERS:
        w = flat[at:at + 27 * ci * co].reshape(27, co, ci)
        layer[name] = (w, flat[at + 27 * ci * co:at + 27 * ci * co + co])
        at += 27 * ci * co + co
    head, bias = flat[at:at + 48].reshape(3, 16), flat[at + 48:at + 51]
    a = ans.reshape(B, 3, nz, ny, nx).permute(0, 2, 3, 4, 1)
    x = torch.zeros((B, nz, ny, nx, 16), device=ans.device, dtype=ans.dtype)
    x[..., :3] = a
    for k, v in enumerate((sc[:, 0] * sc[:, 1] / (2 * math.pi), sc[:, 1] / 32, sc[:, 2] / 1e-3)):
        x[..., 3 + k] = v.reshape(B, 1, 1, 1)

    def two(x, name):
        return _conv(_conv(x, *layer[name + "a"]), *layer[name + "b"])

    e1 = two(x, "enc1")
    e2 = two(_pool(e1), "enc2")
    e3 = two(_pool(e2), "enc3")
    d = two(_pool(e3), "bot")
    for name, e in (("dec3", e3), ("dec2", e2), ("dec1", e1)):
        d = two(torch.cat([_up(d), e], -1), name)
    v = a + d @ head.T + bias
    v = v / torch.linalg.vector_norm(v, dim=-1, keepdim=True)
    return v.permute(0, 4, 1, 2, 3).reshape(B, 3, -1)


def _energy(n, p):
    """Lattice Frank energy: nearest-neighbour links (to plates with anchoring too) and sites."""
    K, q0, N = p["K"], p["q0"], n[0].numel()
    e = torch.zeros((), device=n.device, dtype=n.dtype)
    eps = [[1, 2], [2, 0], [0, 1]]

    def link(a, c, b):  # eps_abc n_a(x) n_c(x + e_b)
        i, k = eps[b][1], eps[b][0]  # (a, b, c) = (i, b, k) is a positive permutation
        return (0.5 * K * ((c - a) ** 2).sum(0) + K * q0 * (a[i] * c[k] - a[k] * c[i])).sum()

    for b in range(3):
        if b == 2 and p["walls_z"]:
            e = e + link(n[:, :-1], n[:, 1:], b)
            if p["anchoring"] == "homeotropic":
                zh = torch.zeros_like(n[:, :1])
                zh[2] = 1
                e = e + link(n[:, -1:], zh, b) + link(zh, n[:, :1], b)
        else:
            e = e + link(n, torch.roll(n, -1, 3 - b), b)
    return float(e + 0.5 * K * q0 * q0 * N - 0.5 * p["W0"] * (n[2] ** 2).sum())


def exact(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "channel":
        n, u, _ = _fields(case, seed, dev)
        p = _params(case)
        n, u, rho, f = _advance(p, n, u, case["steps"])
        out = [n, u, rho]
        if case["diagnostics"]:
            norm = torch.linalg.vector_norm(n, dim=0)
            shape = (3, p["nz"], p["ny"], p["nx"])
            out += [np.array([float(f.sum()) + n[0].numel(), _energy(n.reshape(shape), p),
                              float(torch.linalg.vector_norm(u, dim=0).max()), float(norm.min()), float(norm.max())]),
                    None]  # the centroids follow the earlier ones
        return out
    if kind == "batch":
        parts = []
        for k, c in enumerate(_batch_params(case, seed)):
            n, u, _ = _fields(c, seed + 7919 * (k + 1), dev)
            parts += [v.reshape(-1) for v in _advance(_params(c), n, u, case["steps"])[:3]]
        return [torch.cat(parts)]
    if kind == "relax":
        out = []
        for k, p in enumerate(_relax_params(case, seed)):
            n = _relax_start(case, seed, k, dev).reshape(3, p["nz"], p["ny"], p["nx"])
            for _ in range(case["steps"]):
                n = _director_step(n, None, p)
            out.append(n.reshape(3, -1))
        return [torch.stack(out), None]
    ans, tgt, sc = (t.double() for t in _cells(case, seed, dev))
    w, m, v = (torch.from_numpy(a).to(dev) for a in _weights(seed))
    dims = (case["nx"], case["ny"], case["nz"])
    if kind == "forward":
        with torch.no_grad():
            return [_unet(w, ans, sc, dims)]
    w.requires_grad_(True)
    pred = _unet(w, ans, sc, dims)
    loss = ((pred - tgt) ** 2).sum(1).mean()
    (g,) = torch.autograd.grad(loss, w)
    with torch.no_grad():
        m, v, t = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g, 1001
        new = w - 1e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        return [loss.detach().reshape(1), new, m, v]
