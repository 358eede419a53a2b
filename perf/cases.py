"""Performance cases of the differentiable lattice Boltzmann library.

What a program does with this library, through its public entry points: gradient evaluations of an
inversion (forward sweep, loss, checkpointed reverse sweep) on one lattice or on a batch of lattices,
plain time stepping, the cylinder wake with a loss over a time window, the observation calls on a
finished state, and the learned initialiser's training and inference passes.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges, ``prepare`` makes a
case's inputs and handles from a seed, ``run`` is one pass, ``work`` the bytes and operations the pass
cannot do without and ``exact`` the same outputs in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_00810_gb300 import lbm
from paper_2310_00810_gb300 import unet as N
from paper_2310_00810_gb300 import workloads as W

DEV = "cuda"
RHO_OUT = 1.0


# ------------------------------------------------------------------ cases

def _lattice(name, kind, q, nx, ny, nz, real, steps, inlet, porosity, radius, layout="auto", loss="vec", roi=False):
    c = dict(kind=kind, q=q, nx=nx, ny=ny, nz=nz, real=real, steps=steps, inlet=inlet, porosity=porosity,
             radius=radius, layout=layout, loss=loss, roi=roi, tau=0.8)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem of the configurations: a 64 x 32 FP64 channel, T = 1000, gradient of the inlet
        # density; every launch is latency
        _lattice("channel_64x32_fp64", "gradient", 9, 64, 32, 1, 8, 1000, "const", 1.0, 0),
        # the headline inversion's lattice: disks, porosity 0.6, a 256-entry inlet profile (a tenth of its T)
        _lattice("disks_512x256", "gradient", 9, 512, 256, 1, 4, 2000, "profile", 0.6, 9),
        # a user's own image: odd sizes (no vector or TMA alignment), the norm loss over an outlet band
        _lattice("odd_301x149", "gradient", 9, 301, 149, 1, 4, 1000, "profile", 0.7, 6, loss="norm", roi=True),
        # the 3D joint inversion's lattice: spheres, porosity 0.45, constant head and tau
        _lattice("spheres_128x64x64", "gradient", 19, 128, 64, 64, 4, 400, "const", 0.45, 6),
        # 2D packing larger than the caches, gradient evaluation in the default layout
        _lattice("disks_4096x2048", "gradient", 9, 4096, 2048, 1, 4, 20, "profile", 0.6, 9),
        # the largest 2D lattice, plain time stepping in the fluid-only layout
        _lattice("steps_8192x4096", "steps", 9, 8192, 4096, 1, 4, 20, "profile", 0.6, 9, layout="compact"),
        # the largest 3D lattice, gradient evaluation
        _lattice("spheres_512x256x256", "gradient", 19, 512, 256, 256, 4, 10, "const", 0.45, 6),
        # 64 inversions of uneven sizes (128 x 64 .. 1024 x 512) advanced together in the fluid-only layout
        dict(name="batch_64", kind="batch", count=64, lo=4, hi=32, steps=100, layout="compact"),
        # viscosity inversion behind a cylinder: MRT, periodic y, ramped velocity inlet, loss over a time window
        dict(name="wake_400x160", kind="wake", nx=400, ny=160, diameter=10, steps=1000, observed=5),
        # reading out a finished 3D state: velocity and density fields, loss and its seed, permeability
        _lattice("observe_128x64x64", "observe", 19, 128, 64, 64, 4, 1, "const", 0.45, 6),
        # one training pass of the learned initialiser (loss and gradients), its full size
        dict(name="unet_train", kind="unet_train", base=32, height=128, width=256, batch=16),
        # its inference on one observed field
        dict(name="unet_predict", kind="unet_predict", base=32, height=128, width=256, batch=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["2d", "2d", "2d", "3d", "3d", "steps", "batch", "wake", "observe", "unet_train", "unet_predict"])
    if what in ("2d", "steps"):
        nx = _log(rng, 48, 6000)
        ny = max(24, int(nx * rng.uniform(0.3, 0.7)))
        real = 8 if rng.random() < 0.25 else 4
        steps = max(10, min(600, int(2e8 / (nx * ny))))
        porosity = round(rng.uniform(0.5, 0.9), 3)
        # the norm loss wants a flow everywhere it looks: only where the sweep crosses the lattice
        loss = rng.choice(["vec", "vec", "norm"]) if steps >= 3 * nx else "vec"
        return _lattice("", "steps" if what == "steps" else "gradient", 9, nx, ny, 1, real, steps,
                        rng.choice(["const", "profile"]), porosity, rng.randint(5, 10),
                        rng.choice(["auto", "auto", "compact"]), loss, rng.random() < 0.3)
    if what in ("3d", "observe"):
        nx = _log(rng, 24, 400)
        ny, nz = max(12, int(nx * rng.uniform(0.3, 0.7))), max(12, int(nx * rng.uniform(0.3, 0.7)))
        real = 8 if rng.random() < 0.25 else 4
        steps = 1 if what == "observe" else max(10, min(300, int(1e8 / (nx * ny * nz))))
        return _lattice("", "observe" if what == "observe" else "gradient", 19, nx, ny, nz, real, steps,
                        rng.choice(["const", "const", "profile"]), round(rng.uniform(0.4, 0.8), 3),
                        rng.randint(3, 7), "auto", "vec", rng.random() < 0.3)
    if what == "batch":
        hi = rng.randint(6, 32)
        return dict(kind="batch", count=_log(rng, 3, 64), lo=4, hi=hi, steps=rng.randint(20, 100),
                    layout=rng.choice(["compact", "compact", "dense"]))
    if what == "wake":
        nx = _log(rng, 120, 800)
        return dict(kind="wake", nx=nx, ny=max(48, int(nx * rng.uniform(0.35, 0.6))), diameter=rng.randint(8, 14),
                    steps=rng.randint(200, 900), observed=rng.randint(1, 8))
    base = rng.choice([8, 16, 32, 32, 64])
    h, w = 8 * rng.randint(4, 20), 8 * rng.randint(4, 36)
    most = max(1, min(24, int(16 * 32 * 32 * 128 * 256 / (base * base * h * w))))
    return dict(kind=what, base=base, height=h, width=w, batch=rng.randint(1, most))


# ----------------------------------------------------------------- inputs

def _rng(seed):
    return np.random.Generator(np.random.PCG64(int(seed)))


def _grains(case, seed):
    """uint8 mask [nz][ny][nx] on the GPU: grains of the case's radius, eight free columns at both ends.
    2D: one disk per cell of a jittered grid (they do not overlap); 3D: overlapping spheres at random."""
    nx, ny, nz, r = case["nx"], case["ny"], case["nz"], case["radius"]
    mask = torch.zeros(nz * ny * nx, dtype=torch.uint8, device=DEV)
    if r == 0 or case["porosity"] >= 1.0:
        return mask.view(nz, ny, nx)
    por = max(0.35, (case["porosity"] * nx - 16) / (nx - 16))  # of the part between the free columns
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)
    uni = lambda n: torch.rand(n, generator=g, device=DEV)
    if case["q"] == 9:
        cell = max(2.0 * r + 1.0, r * math.sqrt(math.pi / (1.0 - por)))
        gx, gy = int((nx - 16) / cell) + 1, int(ny / cell) + 1
        k = torch.arange(gx * gy, device=DEV)
        rad = torch.clamp(r * (0.8 + 0.4 * uni(gx * gy)), max=(cell - 1.0) / 2)
        slack = torch.clamp(cell - 2.0 * rad - 1.0, min=0.0)
        cx = 8.0 + (k % gx) * cell + rad + 0.5 + slack * uni(gx * gy)
        cy = (k // gx) * cell + rad + 0.5 + slack * uni(gx * gy)
        cz = torch.zeros_like(cx)
    else:
        pad = 2 * r  # centres outside the walls too, so that the packing is even up to them
        n = max(1, int(-math.log(por) * nx * (ny + pad) * (nz + pad) / (4.0 / 3.0 * math.pi * r ** 3)))
        cx, cy, cz, rad = uni(n) * nx, uni(n) * (ny + pad) - r, uni(n) * (nz + pad) - r, torch.full((n,), float(r), device=DEV)
    reach = int(math.ceil(1.2 * r)) + 1
    o = torch.arange(-reach, reach + 1, device=DEV)
    oz = o if case["q"] == 19 else o[:1] * 0
    for dz in oz.tolist():
        z = torch.floor(cz) + dz
        for dy in o.tolist():
            y = torch.floor(cy) + dy
            x = torch.floor(cx)[:, None] + o[None, :]
            d2 = (x - cx[:, None]) ** 2 + ((y - cy) ** 2 + (z - cz) ** 2 * (case["q"] == 19))[:, None]
            ok = (d2 <= (rad * rad)[:, None]) & (x >= 8) & (x < nx - 8)
            ok &= ((y >= 0) & (y < ny) & (z >= 0) & (z < nz))[:, None]
            at = (z[:, None] * ny + y[:, None]) * float(nx)
            mask[(at.to(torch.int64) + x.to(torch.int64))[ok]] = 1
    return mask.view(nz, ny, nx)


def _shape(case):
    return (case["ny"], case["nx"]) if case["q"] == 9 else (case["nz"], case["ny"], case["nx"])


def _waves(shape, seed, scale, parts):
    """float64 [parts, *shape]: smooth fields, products of sines with seeded phases and wave numbers."""
    r = _rng(seed)
    out = torch.empty((parts, *shape), dtype=torch.float64, device=DEV)
    for p in range(parts):
        v = torch.full((1,) * len(shape), scale * float(r.uniform(0.5, 1.0)), dtype=torch.float64, device=DEV)
        for a, n in enumerate(shape):
            t = torch.arange(n, dtype=torch.float64, device=DEV) / n
            t = torch.sin(2 * math.pi * (float(r.integers(1, 6)) * t + float(r.uniform())))
            v = v * (1.0 + 0.5 * t).view([-1 if b == a else 1 for b in range(len(shape))])
        out[p] = v
    return out


def _inlet(case, seed):
    n = case["ny"] * case["nz"]
    if case["inlet"] == "const":
        return torch.tensor([1.0 + 1e-3 * float(_rng(seed).uniform(0.5, 1.5))], dtype=torch.float64, device=DEV)
    return torch.as_tensor(1.0 + W.inlet_profile(n, seed), dtype=torch.float64, device=DEV)


def _lattice_inputs(case, seed):
    d, shape = 2 if case["q"] == 9 else 3, _shape(case)
    target = _waves(shape, seed + 3, 2e-4, d)
    target[1:] *= 0.2
    roi = None
    if case["roi"]:
        roi = torch.zeros(shape, dtype=torch.uint8, device=DEV)
        roi[..., (2 * case["nx"]) // 3:] = 1
    return dict(mask=_grains(case, seed), rho_in=_inlet(case, seed + 1), target=target, roi=roi,
                tau=torch.tensor([case["tau"]], dtype=torch.float64, device=DEV))


def _state_inputs(case, seed, mask):
    """A developed-looking state: a pressure gradient, a smooth flow and a little of every other mode."""
    dtype = torch.float32 if case["real"] == 4 else torch.float64
    shape = _shape(case)
    c, w, _ = _velocities(case["q"])
    m = _waves(shape, seed + 5, 1e-3, c.shape[1] + 1)
    fluid = (mask.view(shape) == 0).to(torch.float64)
    f = torch.empty((case["q"], *shape), dtype=dtype, device=DEV)
    for i in range(case["q"]):
        v = m[0] * (1.0 + 0.01 * i)
        for a in range(c.shape[1]):
            if c[i, a]:
                v = v + 0.3 * float(c[i, a]) * m[a + 1]
        f[i] = (float(w[i]) * v * fluid).to(dtype)
    return f


def _wake_inputs(case, seed):
    nx, ny, r = case["nx"], case["ny"], _rng(seed)
    yy, xx = torch.meshgrid(torch.arange(ny, device=DEV), torch.arange(nx, device=DEV), indexing="ij")
    cx, cy = nx * 0.2 + float(r.uniform(-2, 2)), ny * 0.5 + float(r.uniform(1, 2))
    mask = ((xx - cx) ** 2 + (yy - cy) ** 2 <= (case["diameter"] / 2) ** 2).to(torch.uint8)
    k, T = case["observed"], case["steps"]
    roi = torch.zeros((ny, nx), dtype=torch.uint8, device=DEV)
    roi[ny // 4:(3 * ny) // 4, nx // 4:nx // 2] = 1
    targets = torch.stack([_waves((ny, nx), seed + 11 + j, 0.1, 2) for j in range(k)])
    targets[:, 1] *= 0.1
    return dict(mask=mask, roi=roi, targets=targets, steps=[T - (k - 1 - j) * max(1, T // (4 * k)) for j in range(k)],
                rho_in=torch.ones(1, dtype=torch.float64, device=DEV), u_in=(0.1 + 0.1 * float(r.uniform()), 0.0),
                tau=torch.tensor([0.56 + 0.1 * float(r.uniform())], dtype=torch.float64, device=DEV), ramp=T // 2,
                rates=(1.1, 1.1, 1.2))


def _network_inputs(case, seed):
    """Observed fields and masks as the network's input, profile targets, FP32 master parameters."""
    b, h, w = case["batch"], case["height"], case["width"]
    x = torch.zeros((b, h, w, N.IN_CHANNELS), dtype=torch.float32, device=DEV)
    for j in range(b):
        m = _grains(dict(q=9, nx=w, ny=h, nz=1, radius=6, porosity=0.6), seed + 31 * j)[0].float()
        v = _waves((h, w), seed + 31 * j + 1, 0.3, 2).float() * (1.0 - m)
        x[j, :, :, 0], x[j, :, :, 1], x[j, :, :, 2] = v[0], 0.3 * v[1], m
    target = np.stack([W.inlet_profile(h, seed + j) / 1e-3 for j in range(b)]).astype(np.float32)
    r = _rng(seed + 2)
    parts = []
    for s in N.param_shapes(case["base"]):
        scale = 0.05 if len(s) == 1 else math.sqrt(2.0 / ((s[0] * s[1] if s[0] == 3 else 1) * s[2]))
        parts.append(r.normal(0.0, scale, int(np.prod(s))).astype(np.float32))
    return x.to(torch.bfloat16), torch.as_tensor(target, device=DEV), torch.as_tensor(np.concatenate(parts), device=DEV)


def _batch_sizes(case, seed):
    """Sizes of the batched recipe, nx = 32 U{lo..hi} and ny = nx / 2, the same for every seed."""
    r = _rng(4000 + case["count"] * 131 + case["hi"])
    return [(32 * int(r.integers(case["lo"], case["hi"] + 1)), float(r.uniform(0.5, 0.7))) for _ in range(case["count"])]


# ---------------------------------------------------------------- prepare

def _solver(case, mask):
    s = lbm.Solver(case["q"], case["nx"], case["ny"], case["nz"], precision=case["real"], n_steps=case["steps"],
                   loss_kind=lbm.LBM_LOSS_VEC if case["loss"] == "vec" else lbm.LBM_LOSS_NORM,
                   inlet_kind=lbm.LBM_INLET_PROFILE if case["inlet"] == "profile" else lbm.LBM_INLET_CONST,
                   geometry=mask, layout=case["layout"])
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("gradient", "steps", "observe"):
        p = _lattice_inputs(case, seed)
        p.update(kind=kind, solver=_solver(case, p["mask"]), steps=case["steps"])
        if kind != "gradient":
            p["f0"] = _state_inputs(case, seed, p["mask"])
        return p
    if kind == "wake":
        p = _wake_inputs(case, seed)
        s = lbm.Solver(9, case["nx"], case["ny"], precision=4, n_steps=case["steps"], geometry=p["mask"],
                       periodic_y=True)
        s.set_velocity_inlet(p["u_in"])
        s.set_velocity_ramp(p["ramp"])
        s.set_collision(lbm.LBM_COLLISION_MRT, *p["rates"])
        p.update(kind=kind, solver=s)
        return p
    if kind == "batch":
        sizes = _batch_sizes(case, seed)
        geoms = [dict(kind=lbm.LBM_GEOM_DISKS, seed=seed * 1000 + i, r_min=6, r_max=12, target_porosity=por)
                 for i, (_, por) in enumerate(sizes)]
        b = lbm.Batch(9, [(n, n // 2, 1) for n, _ in sizes], precision=4, n_steps=case["steps"],
                      inlet_kind=lbm.LBM_INLET_PROFILE, geometries=geoms, layout=case["layout"])
        rho_in, target = b.new_inlet(), b.new_velocity()
        for i, (n, _) in enumerate(sizes):
            b.view_inlet(rho_in, i).copy_(torch.as_tensor(1.0 + W.inlet_profile(n // 2, seed + 7 * i)))
            b.view_velocity(target, i).copy_(_waves((n // 2, n), seed + 7 * i + 1, 2e-4, 2))
        tau = torch.full((b.n,), 0.8, dtype=torch.float64, device=DEV)
        return dict(kind=kind, batch=b, rho_in=rho_in, target=target, tau=tau)
    x, target, params = _network_inputs(case, seed)
    net = N.UNet(base=case["base"], height=case["height"], width=case["width"], batch=case["batch"], seed=0)
    net.params.copy_(params)
    return dict(kind=kind, net=net, x=x.view(torch.int16), target=target)


# -------------------------------------------------------------------- run

def _as(f, t):
    """A loss or gradient in the precision of the populations it was formed from (its sums are FP64)."""
    return t.to(f.dtype)


def run(p):
    kind = p["kind"]
    if kind == "gradient":
        s = p["solver"]
        f = s.forward(p["rho_in"], p["tau"], RHO_OUT)
        loss, lam = s.loss_grad(f, p["target"], p["roi"])
        g_in, g_tau = s.adjoint(p["rho_in"], p["tau"], RHO_OUT, lam)
        return dict(f=f, loss=_as(f, loss), lam=lam, grad_rho_in=_as(f, g_in), grad_tau=_as(f, g_tau))
    if kind == "steps":
        return p["solver"].step(p["rho_in"], p["tau"], RHO_OUT, p["f0"], p["steps"])
    if kind == "observe":
        s = p["solver"]
        rho, u = s.macroscopic(p["f0"])
        loss, lam = s.loss_grad(p["f0"], p["target"], p["roi"])
        k, flux = s.darcy(p["f0"], p["rho_in"], p["tau"], RHO_OUT)
        return dict(rho=rho, u=u, loss=loss, lam=lam, k=k, flux=flux)
    if kind == "wake":
        s = p["solver"]
        f = s.forward(p["rho_in"], p["tau"], RHO_OUT)
        loss, _, g_tau = s.adjoint_window(p["rho_in"], p["tau"], RHO_OUT, f, p["steps"], p["targets"], p["roi"])
        return dict(f=f, loss=_as(f, loss), grad_tau=_as(f, g_tau))
    if kind == "batch":
        b = p["batch"]
        f = b.forward(p["rho_in"], p["tau"], RHO_OUT)
        loss, lam = b.loss_grad(f, p["target"])
        g_in, g_tau = b.adjoint(p["rho_in"], p["tau"], RHO_OUT, lam)
        return dict(f=f, loss=_as(f, loss), grad_rho_in=_as(f, g_in), grad_tau=_as(f, g_tau))
    net = p["net"]
    if kind == "unet_train":
        loss = net.loss_and_grad(p["x"], p["target"])
        return dict(loss=loss, out=net.out, grad=net.grad)
    return N.predict(net, p["x"])


# ------------------------------------------------------------------- work

def work(case):
    """A step moves each fluid node's populations in and out; its reverse also reads the state.  About 14
    operations per population forward, 36 in reverse.  The network: its convolutions' products."""
    kind = case["kind"]
    if kind.startswith("unet"):
        c = [case["base"] << l for l in range(4)]
        px = [case["batch"] * case["height"] * case["width"] >> (2 * l) for l in range(4)]
        f, prev = 0, N.IN_CHANNELS
        act = px[0] * N.IN_CHANNELS
        for l in range(4):
            f += 18 * px[l] * (prev * c[l] + c[l] * c[l])
            act += 2 * px[l] * c[l]
            prev = c[l]
        for l in (2, 1, 0):
            f += px[l] * (2 * c[l + 1] * c[l] + 18 * (2 * c[l] * c[l] + c[l] * c[l]))
            act += 3 * px[l] * c[l]
        n = sum(int(np.prod(s)) for s in N.param_shapes(case["base"]))
        if kind == "unet_train":  # activations kept for and read by the reverse pass, FP32 gradients
            return {"bytes": 2 * 2 * act + 2 * px[0] * N.IN_CHANNELS + 8 * n, "flops": 3 * f}
        return {"bytes": 2 * px[0] * N.IN_CHANNELS + 4 * n, "flops": f}
    if kind == "batch":
        nodes = sum(n * (n // 2) * por for n, por in _batch_sizes(case, 0)) * case["steps"]
        return {"bytes": 5 * 9 * 4 * nodes, "flops": 50 * 9 * nodes}
    if kind == "wake":
        nodes = case["nx"] * case["ny"] * case["steps"]
        return {"bytes": 5 * 9 * 4 * nodes, "flops": 100 * 9 * nodes}
    q, s = case["q"], case["real"]
    every = case["nx"] * case["ny"] * case["nz"]
    nodes = every * case["porosity"] * case["steps"]
    if kind == "steps":
        return {"bytes": 2 * q * s * nodes, "flops": 14 * q * nodes}
    if kind == "observe":
        d = 2 if q == 9 else 3
        return {"bytes": (q * s * case["porosity"] + q * s + 8 * (1 + d) + 8 * d * case["porosity"]) * every,
                "flops": 8 * q * every}
    return {"bytes": 5 * q * s * nodes, "flops": 50 * q * nodes}


# ------------------------------------------------------------------ exact

def _velocities(q):
    if q == 9:
        c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        opp, w = [0, 3, 4, 1, 2, 7, 8, 5, 6], [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        c = [(0, 0, 0)]
        for v in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)):
            c += [v, tuple(-a for a in v)]
        opp, w = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)], [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return np.array(c), np.array(w), np.array(opp)


def _mrt(rates, omega):
    """M^-1 S M of the D2Q9 moment matrix (rows rho, e, epsilon, j_x, q_x, j_y, q_y, p_xx, p_xy)."""
    c, _, _ = _velocities(9)
    cx, cy = c[:, 0].astype(float), c[:, 1].astype(float)
    s2 = cx * cx + cy * cy
    m = np.stack([cx * 0 + 1, -4 + 3 * s2, 4 - 10.5 * s2 + 4.5 * s2 * s2, cx, (-5 + 3 * s2) * cx, cy,
                  (-5 + 3 * s2) * cy, cx * cx - cy * cy, cx * cy])
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=DEV)
    zero = omega * 0.0
    s = torch.stack([zero, zero + rates[0], zero + rates[1], zero, zero + rates[2], zero, zero + rates[2], omega, omega])
    return t(np.linalg.inv(m)) @ (s[:, None] * t(m))


class _Exact:
    """One time step of the method on fluid nodes in 64 bits: collide, stream, bounce back, Eq. 6."""

    def __init__(self, q, mask, periodic_y=False, u_in=None, ramp=0, rates=None):
        nz, ny, nx = mask.shape
        self.q, self.shape = q, (q, ny, nx) if q == 9 else (q, nz, ny, nx)
        c, w, opp = _velocities(q)
        self.c = torch.as_tensor(c, dtype=torch.float64, device=DEV)
        self.w = torch.as_tensor(w, dtype=torch.float64, device=DEV)
        self.u_in, self.ramp, self.rates = u_in, ramp, rates
        solid = mask.reshape(-1) != 0
        self.node = torch.nonzero(~solid).view(-1)
        nf = self.node.numel()
        compact = torch.full((nz * ny * nx,), -1, dtype=torch.int64, device=DEV)
        compact[self.node] = torch.arange(nf, device=DEV)
        x, y, z = self.node % nx, (self.node // nx) % ny, self.node // (nx * ny)
        self.take = torch.empty((q, nf), dtype=torch.int64, device=DEV)
        open_, wall = [], []
        me = torch.arange(nf, device=DEV)
        for i in range(q):
            xs, ys = x - int(c[i, 0]), y - int(c[i, 1])
            zs = z - (int(c[i, 2]) if q == 19 else 0)
            if periodic_y:
                ys = ys % ny
            inside = (ys >= 0) & (ys < ny) & (zs >= 0) & (zs < nz)
            plane = (xs < 0) | (xs >= nx)
            at = ((zs * ny + ys) * nx + xs)[inside & ~plane]
            src = torch.full((nf,), -1, dtype=torch.int64, device=DEV)
            src[inside & ~plane] = compact[at]
            self.take[i] = torch.where(src >= 0, i * nf + src, int(opp[i]) * nf + me)
            k = me[inside & plane]
            open_.append(torch.stack([torch.full_like(k, i), k]))
        self.open = torch.cat(open_, 1)
        k = self.open[1]
        self.at_inlet = x[k] == 0
        self.row = (z * ny + y)[k]
        self.flat = self.open[0] * nf + k
        self.sign = torch.ones(q * nf, dtype=torch.float64, device=DEV)
        flip = self.flat if u_in is None else self.flat[~self.at_inlet]
        self.sign[flip] = -1.0
        self.nf = nf

    def moments(self, f):
        rho = 1.0 + f.sum(0)
        return rho, (self.c.t() @ f) / rho

    def step(self, f, rho_in, tau, t):
        rho, u = self.moments(f)
        uu = (u * u).sum(0)
        cu = self.c @ u
        d = f - self.w[:, None] * ((rho - 1.0) + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
        g = f - d / tau if self.rates is None else f - _mrt(self.rates, 1.0 / tau.reshape(())) @ d
        i, k = self.open
        rw = torch.where(self.at_inlet, rho_in[self.row] if rho_in.numel() > 1 else rho_in[0],
                         torch.full((), RHO_OUT, dtype=torch.float64, device=DEV))
        cw = cu[i, k]
        add = 2.0 * self.w[i] * ((rw - 1.0) + rw * (4.5 * cw * cw - 1.5 * uu[k]))
        if self.u_in is not None:
            r = 1.0 if self.ramp <= 0 or t >= self.ramp else math.sin(math.pi * t / (2 * self.ramp)) ** 2
            cin = self.c[i] @ torch.as_tensor(self.u_in, dtype=torch.float64, device=DEV)
            add = torch.where(self.at_inlet, 6.0 * self.w[i] * cin * r, add)
        out = g.reshape(-1)[self.take.view(-1)] * self.sign
        return out.index_add(0, self.flat, add).view(self.q, self.nf)

    def loss(self, f, target, roi, kind):
        d = self.c.shape[1]
        _, u = self.moments(f)
        t = target.reshape(d, -1)[:, self.node]
        if kind == "vec":
            e = ((u - t) ** 2).sum(0)
        else:
            uu = (u * u).sum(0)
            un = torch.where(uu > 0, uu, torch.ones_like(uu)).sqrt() * (uu > 0)
            e = (un - (t * t).sum(0).sqrt()) ** 2
        return e.sum() if roi is None else (e * roi.reshape(-1)[self.node]).sum()

    def dense(self, f):
        out = torch.zeros((f.shape[0], math.prod(self.shape[1:])), dtype=torch.float64, device=DEV)
        out[:, self.node] = f
        return out.view(f.shape[0], *self.shape[1:])

    def sweep(self, rho_in, tau, steps, losses):
        """f^T and the sum of the losses ({step: function of f}), its gradients and lambda^T."""
        every = max(1, int(math.sqrt(steps)))
        kept, f = {}, torch.zeros((self.q, self.nf), dtype=torch.float64, device=DEV)
        with torch.no_grad():
            for t in range(steps):
                if t % every == 0:
                    kept[t] = f
                f = self.step(f, rho_in, tau, t + 1)
        total, lam, first = 0.0, torch.zeros_like(f), None
        g_in, g_tau = torch.zeros_like(rho_in), torch.zeros_like(tau)
        for t0 in sorted(kept, reverse=True):
            seg = [kept.pop(t0)]
            with torch.no_grad():
                while len(seg) < min(every, steps - t0):
                    seg.append(self.step(seg[-1], rho_in, tau, t0 + len(seg)))
            for t in range(t0 + len(seg), t0, -1):
                a = seg.pop().requires_grad_()
                r, s = rho_in.detach().requires_grad_(), tau.detach().requires_grad_()
                b = self.step(a, r, s, t)
                if t in losses:
                    c = b.detach().requires_grad_()
                    v = sum(fn(c) for fn in losses[t])
                    lam = lam + torch.autograd.grad(v, c)[0]
                    total = total + v.detach()
                if first is None:
                    first = lam
                lam, di, dt = torch.autograd.grad(b, (a, r, s), lam, allow_unused=True)
                g_in, g_tau = g_in if di is None else g_in + di, g_tau + dt
        return f, total.reshape(1), first, g_in, g_tau


def _exact_network(case, seed):
    x, target, params = _network_inputs(case, seed)
    p, o = [], 0
    for s in N.param_shapes(case["base"]):
        n = int(np.prod(s))
        p.append(params[o:o + n].double().view(s).requires_grad_(case["kind"] == "unet_train"))
        o += n
    weights = iter(p)
    nn = torch.nn.functional

    def conv(v, w, b):  # v [B, C, H, W]; one matrix product per tap
        B, C, H, Wd = v.shape
        e = nn.pad(v, (1, 1, 1, 1))
        y = b.view(1, -1, 1, 1)
        for dy in range(3):
            for dx in range(3):
                part = e[:, :, dy:dy + H, dx:dx + Wd].reshape(B, C, H * Wd)
                y = y + torch.matmul(w[dy, dx].t(), part).view(B, -1, H, Wd)
        return torch.relu(y)

    def up(v, w, b):
        B, C, H, Wd = v.shape
        y = torch.einsum("bchw,yxco->bohywx", v, w).reshape(B, -1, 2 * H, 2 * Wd)
        return y + b.view(1, -1, 1, 1)

    with torch.set_grad_enabled(case["kind"] == "unet_train"):
        v, skips = x.double().permute(0, 3, 1, 2), []
        for l in range(4):
            v = conv(v, next(weights), next(weights))
            v = conv(v, next(weights), next(weights))
            if l < 3:
                skips.append(v)
                v = nn.max_pool2d(v, 2)
        for l in (2, 1, 0):
            v = torch.cat([up(v, next(weights), next(weights)), skips[l]], 1)
            v = conv(v, next(weights), next(weights))
            v = conv(v, next(weights), next(weights))
        out = (torch.einsum("bchw,c->bhw", v, next(weights)) + next(weights)).mean(2)
        if case["kind"] == "unet_predict":
            return out
        loss = ((out - target.double()) ** 2).mean()
        grad = torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, p)])
    return dict(loss=loss.detach().reshape(1), out=out.detach(), grad=grad)


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("unet"):
        return _exact_network(case, seed)
    if kind == "batch":
        return None  # its packings come from the library's own grain placement
    if kind == "wake":
        p = _wake_inputs(case, seed)
        e = _Exact(9, p["mask"][None], True, p["u_in"], p["ramp"], p["rates"])
        losses = {}
        for t, target in zip(p["steps"], p["targets"]):
            losses.setdefault(t, []).append(lambda f, target=target: e.loss(f, target, p["roi"], "vec"))
        f, loss, _, _, g_tau = e.sweep(p["rho_in"], p["tau"], case["steps"], losses)
        return dict(f=e.dense(f), loss=loss, grad_tau=g_tau)
    p = _lattice_inputs(case, seed)
    e = _Exact(case["q"], p["mask"])
    if kind == "gradient":
        fn = lambda f: e.loss(f, p["target"], p["roi"], case["loss"])
        f, loss, lam, g_in, g_tau = e.sweep(p["rho_in"], p["tau"], case["steps"], {case["steps"]: [fn]})
        return dict(f=e.dense(f), loss=loss, lam=e.dense(lam), grad_rho_in=g_in, grad_tau=g_tau)
    f0 = _state_inputs(case, seed, p["mask"]).double().view(case["q"], -1)[:, e.node]
    if kind == "steps":
        for t in range(case["steps"]):
            f0 = e.step(f0, p["rho_in"], p["tau"], t + 1)
        return e.dense(f0)
    rho, u = e.moments(f0)
    f0.requires_grad_()
    loss = e.loss(f0, p["target"], p["roi"], case["loss"])
    lam = torch.autograd.grad(loss, f0)[0]
    rho_f, u_f = e.dense(rho[None])[0].detach(), e.dense(u).detach()
    xs = case["nx"] // 2
    flux = (rho_f * u_f[0])[..., xs].sum() / (case["ny"] * case["nz"])
    drop = (p["rho_in"].mean() - RHO_OUT) / (3.0 * case["nx"])
    k = (p["tau"] - 0.5) / 3.0 * flux / drop
    return dict(rho=rho_f, u=u_f, loss=loss.detach().reshape(1), lam=e.dense(lam), k=k, flux=flux.reshape(1))
