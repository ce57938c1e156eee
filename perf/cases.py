"""Workloads of this library as its users run it, one pass each through the
public entry points: plain projections from one 128^2 grid to the 16 x 512^2
batch and a 2048^2 grid, ragged and open boxes, whole driver steps, the
adjoint of the fixed-count projection, the networks' forward, hybrid
projection, single convolution, and the training gradient.

``listed`` names the workloads, ``draw`` takes another one of the same ranges,
``prepare`` makes the inputs on the device from a seed, ``run`` is one pass,
``work`` what a pass cannot do without, and ``exact`` the same outputs by plain
torch in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2109_09363_gb300 as hp
from paper_2109_09363_gb300 import autograd as hp_autograd
from paper_2109_09363_gb300 import training as hp_training


def listed():
    return [
        # one solver step of the small plume (driver step, then projection):
        # launches and latency
        dict(name="step_1x128", kind="step", batch=1, ny=128, nx=128, scheme=1,
             threshold=1e-3, max_iters=1000, sweeps=200),
        # many training-size grids at once (hybrid evaluation, data generation)
        dict(name="project_256x128", kind="project", batch=256, ny=128, nx=128, field="training",
             threshold=1e-3, max_iters=5000, fixed=0, open_top=False, sweeps=1300),
        # the benchmark batch: vortex fields with obstacles, E_t 1e-4, cap 5000
        dict(name="project_16x512", kind="project", batch=16, ny=512, nx=512, field="vortex",
             threshold=1e-4, max_iters=5000, fixed=0, open_top=False, sweeps=4800),
        # one grid of the paper's size with an open top and an injecting inlet
        dict(name="project_1x512_open", kind="project", batch=1, ny=512, nx=512, field="vortex",
             threshold=1e-4, max_iters=2000, fixed=0, open_top=True, sweeps=2000),
        # a fixed number of sweeps (targets, rollouts) on rows that allow no
        # vector access
        dict(name="project_6x331x467", kind="project", batch=6, ny=331, nx=467, field="vortex",
             threshold=0.0, max_iters=0, fixed=400, open_top=False, sweeps=400),
        # the large plume box: more cells than one cluster of SMs holds
        dict(name="project_1x2048", kind="project", batch=1, ny=2048, nx=2048, field="training",
             threshold=1e-8, max_iters=400, fixed=0, open_top=False, sweeps=400),
        # forward and backward of one rollout step of 20 sweeps
        dict(name="adjoint_8x256", kind="adjoint", batch=8, ny=256, nx=256, k=20),
        # the network alone on the benchmark batch
        dict(name="cnn_16x512", kind="cnn", arch="multiscale", batch=16, ny=512, nx=512),
        # one hybrid projection of the paper's size: guess, then a few sweeps
        dict(name="hybrid_1x512", kind="hybrid", arch="unet", batch=1, ny=512, nx=512,
             threshold=1e-6, max_iters=60),
        # the networks' dominant layer by itself
        dict(name="conv_8x512", kind="conv", batch=8, ny=512, nx=512, cin=64, cout=64, relu=True),
        # the gradient of one training batch of 64 pairs
        dict(name="train_64x128", kind="train", arch="multiscale", batch=64, ny=128, nx=128),
        # the driver step of the benchmark batch, MacCormack
        dict(name="advect_16x512", kind="advect", batch=16, ny=512, nx=512, scheme=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


ARCHS = ("multiscale", "smallscale", "monoscale", "unet")


def draw(rng):
    kind = rng.choice(("step", "project", "project", "project", "large", "adjoint", "cnn",
                       "hybrid", "conv", "train", "advect"))
    batch, ny, nx = _log(rng, 1, 64), _log(rng, 32, 512), _log(rng, 32, 512)
    if kind in ("project", "large"):
        if kind == "large":
            batch, ny, nx = rng.randint(1, 3), _log(rng, 400, 2048), _log(rng, 520, 2048)
        sweeps = min(_log(rng, 20, 3000), int(4e9 / (batch * ny * nx)) + 10)
        fixed = rng.random() < 0.4
        return dict(kind="project", batch=batch, ny=ny, nx=nx,
                    field=rng.choice(("vortex", "training")), threshold=0.0 if fixed else 1e-8,
                    max_iters=0 if fixed else sweeps, fixed=sweeps if fixed else 0,
                    open_top=not fixed and rng.random() < 0.3, sweeps=sweeps)
    if kind == "step":
        n = _log(rng, 48, 512)
        sweeps = _log(rng, 20, 600)
        return dict(kind="step", batch=rng.randint(1, 8), ny=n, nx=n + rng.randint(0, 9),
                    scheme=rng.randint(0, 1), threshold=1e-8, max_iters=sweeps, sweeps=sweeps)
    if kind == "adjoint":
        return dict(kind="adjoint", batch=min(batch, 16), ny=ny, nx=nx, k=_log(rng, 4, 80))
    if kind == "advect":
        return dict(kind="advect", batch=min(batch, 16), ny=ny, nx=nx, scheme=rng.randint(0, 1))
    if kind == "conv":
        return dict(kind="conv", batch=min(batch, 8), ny=ny, nx=nx, cin=rng.choice((32, 64)),
                    cout=rng.choice((32, 64)), relu=rng.random() < 0.7)
    arch = rng.choice(ARCHS)
    ny, nx = 16 * _log(rng, 2, 32), 16 * _log(rng, 2, 32)
    if kind == "train":
        return dict(kind="train", arch=arch, batch=min(batch, 32), ny=min(ny, 256),
                    nx=min(nx, 256))
    c = dict(kind=kind, arch=arch, batch=min(batch, 8), ny=ny, nx=nx)
    if kind == "hybrid":
        c.update(threshold=1e-8, max_iters=_log(rng, 5, 300))
    return c


# ------------------------------------------------------------------ inputs

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _uniform(g, shape, lo, hi):
    return (torch.rand(shape, generator=g, dtype=torch.float64) * (hi - lo) + lo).to(
        _dev(), torch.float32)


def _faces(ny, nx):
    dev = _dev()
    r = lambda n: torch.arange(n, device=dev, dtype=torch.float32)  # noqa: E731
    return (r(nx + 1)[None, None], (r(ny) + 0.5)[None, :, None],
            (r(nx) + 0.5)[None, None], r(ny + 1)[None, :, None])


def _velocity(g, batch, ny, nx, field):
    """Gaussian vortices on the faces; "training" adds divergence sources."""
    xu, yu, xv, yv = _faces(ny, nx)
    n = max(ny, nx)
    train = field == "training"
    count, w = (max(4, n // 8), (n / 32, n / 8)) if train else (32, (4.0, 32.0))
    u = torch.zeros((batch, ny, nx + 1), device=_dev())
    v = torch.zeros((batch, ny + 1, nx), device=_dev())
    for k in range(count + (max(2, n // 16) if train else 0)):
        vortex = k < count
        cx, cy = _uniform(g, (batch, 1, 1), 0, nx), _uniform(g, (batch, 1, 1), 0, ny)
        a = _uniform(g, (batch, 1, 1), -1.0, 1.0)
        s = _uniform(g, (batch, 1, 1), *w)
        eu = torch.exp(-((xu - cx) ** 2 + (yu - cy) ** 2) / (2 * s * s))
        ev = torch.exp(-((xv - cx) ** 2 + (yv - cy) ** 2) / (2 * s * s))
        if vortex:
            u -= a * (yu - cy) / s * eu
            v += a * (xv - cx) / s * ev
        else:
            u -= a * (xu - cx) / (s * s) * eu
            v -= a * (yv - cy) / (s * s) * ev
    return u, v


def _obstacles(g, batch, ny, nx, few=False):
    """1 to 6 (few: 0 to 4) rectangles or discs per grid, sized to the grid."""
    n = max(ny, nx)
    y = (torch.arange(ny, device=_dev(), dtype=torch.float32) + 0.5)[None, :, None]
    x = (torch.arange(nx, device=_dev(), dtype=torch.float32) + 0.5)[None, None]
    fl = torch.zeros((batch, ny, nx), dtype=torch.bool, device=_dev())
    lo, hi = (0, 4) if few else (1, 6)
    count = torch.randint(lo, hi + 1, (batch, 1, 1), generator=g).to(_dev())
    for k in range(hi):
        cx, cy = _uniform(g, (batch, 1, 1), 0, nx), _uniform(g, (batch, 1, 1), 0, ny)
        w, h = (_uniform(g, (batch, 1, 1), n / 32, n / 5.33) for _ in range(2))
        r = _uniform(g, (batch, 1, 1), n / 64, n / 10.67)
        rect = _uniform(g, (batch, 1, 1), 0, 1) < 0.5
        a = ((x - cx).abs() <= w / 2) & ((y - cy).abs() <= h / 2)
        b = (x - cx) ** 2 + (y - cy) ** 2 <= r * r
        fl |= torch.where(rect, a, b) & (k < count)
    return fl.to(torch.uint8)


def _inlet(nx):
    w = max(1, round(0.29 * nx))
    return nx // 2 - w // 2, nx // 2 - w // 2 + w


U_IN = 0.5  # injection speed of the open box


def _flow(case, seed):
    """u*, v* and flags; an open box carries the injection on its inlet."""
    g = torch.Generator().manual_seed(int(seed))
    B, ny, nx = case["batch"], case["ny"], case["nx"]
    field = case.get("field", "vortex")
    u, v = _velocity(g, B, ny, nx, field)
    fl = _obstacles(g, B, ny, nx, few=field == "training")
    if case.get("open_top"):
        x0, x1 = _inlet(nx)
        v[:, ny, x0:x1] = torch.where(fl[:, ny - 1, x0:x1] == 0, -U_IN, 0.0)
    return g, u, v, fl


def _density(g, B, ny, nx):
    """Ambient density with a plume column above the inlet and noise."""
    rho = 1.0 + 1e-4 * torch.randn((B, ny, nx), generator=g).to(_dev())
    x0, x1 = _inlet(nx)
    rho[:, ny // 3:, x0:x1] += 0.1
    return rho


def _params(case, seed):
    """Initial weights, representable in BF16 (the networks' storage)."""
    p = torch.from_numpy(hp_training.init_params(seed, case["arch"]))
    return p.to(torch.bfloat16).to(torch.float32).numpy()


PLUME = dict(dt=0.5, gravity=-0.5, rho_amb=1.0, rho_in=1.1)
TARGET_SWEEPS = 500
LAMBDA = 0.1


def _project_params(case):
    x = _inlet(case["nx"]) if case.get("open_top") else (0, 0)
    dt = PLUME["dt"] if case["kind"] == "step" else 1.0
    return hp.ProjectParams(threshold=case["threshold"], max_iters=case["max_iters"],
                            fixed_iters=case.get("fixed", 0), dt=dt,
                            open_top=int(bool(case.get("open_top"))), inflow=x)


def _plume_params(case):
    x0, x1 = _inlet(case["nx"])
    return hp.PlumeParams(inlet_x0=x0, inlet_x1=x1, scheme=case["scheme"], **PLUME)


def _conv_inputs(case, seed):
    g = torch.Generator(device=_dev()).manual_seed(int(seed))
    ci, co = case["cin"], case["cout"]
    x = torch.randn((case["batch"], case["ny"], case["nx"], ci), generator=g, device=_dev())
    x = torch.relu(x).to(torch.bfloat16)  # activations of the layer before
    lim = math.sqrt(6.0 / (9 * ci))
    w = (torch.rand((3, 3, co, ci), generator=g, device=_dev()) * 2 - 1) * lim
    b = (torch.rand((co,), generator=g, device=_dev()) * 2 - 1) * 0.1
    return x, w.to(torch.bfloat16), b


def _divergence(u, v, fl):
    o = _open(fl, False)
    return _divergence64(u.double(), v.double(), o, torch.zeros_like(o[0][:, 0])).float()


def _train_inputs(case, seed):
    """Divergence, flags and the pressure that plain sweeps reach from zero."""
    _, u, v, fl = _flow(dict(case, field="training"), seed)
    div = _divergence(u, v, fl)
    target, _, _ = _sweeps64(_open(fl, False), div.double(), torch.zeros_like(div).double(), 0.0,
                             0, TARGET_SWEEPS)
    return div, fl, target.float()


def prepare(case, seed):
    kind, B, ny, nx = case["kind"], case["batch"], case["ny"], case["nx"]
    st = {"case": case}
    if kind == "conv":
        st["x"], st["w"], st["b"] = _conv_inputs(case, seed)
        return st
    if kind == "train":
        st["div"], st["flags"], st["target"] = _train_inputs(case, seed)
        st["cnn"] = hp.CNN(B, ny, nx, params=_params(case, seed), arch=case["arch"])
        st["trainer"] = hp.Trainer(st["cnn"], B, ny, nx)
        return st
    g, u, v, fl = _flow(case, seed)
    st.update(u=u, v=v, flags=fl)
    if kind in ("step", "advect"):
        st["rho"] = _density(g, B, ny, nx)
        st["plume"] = _plume_params(case)
    if kind in ("cnn", "hybrid"):
        st["cnn"] = hp.CNN(B, ny, nx, params=_params(case, seed), arch=case["arch"])
    if kind == "cnn":
        st["div"] = _divergence(u, v, fl)
    if kind in ("step", "project", "adjoint", "hybrid"):
        st["ctx"] = hp.Context(B, ny, nx)
    if kind in ("step", "project", "hybrid"):
        st["prm"] = _project_params(case)
    if kind in ("project", "hybrid"):  # corrected in place: the pass works on a copy
        st["uw"], st["vw"] = torch.empty_like(u), torch.empty_like(v)
    if kind == "adjoint":
        s = lambda *d: torch.randn(d, generator=g).to(_dev())  # noqa: E731
        st.update(phi0=s(B, ny, nx), gu=s(B, ny, nx + 1), gv=s(B, ny + 1, nx), gp=s(B, ny, nx))
    return st


# -------------------------------------------------------------------- pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "conv":
        return hp.hp_conv3x3_bf16(st["x"], st["w"], st["b"], case["relu"])
    if kind == "train":
        grad, loss = st["trainer"].gradient(st["div"], st["flags"], st["target"],
                                            lambda_div=LAMBDA)
        return {"grad": grad, "loss": loss}
    if kind == "cnn":
        phi_hat, s = hp.hp_cnn_forward(st["cnn"], st["div"], st["flags"])
        return {"phi_hat": phi_hat, "s": s}
    if kind == "advect":
        u, v, rho = hp.hp_advect_step(st["u"], st["v"], st["rho"], st["flags"], st["plume"])
        return {"u": u, "v": v, "rho": rho}
    if kind == "step":
        u, v, rho = hp.hp_advect_step(st["u"], st["v"], st["rho"], st["flags"], st["plume"])
        out = hp.hp_project(st["ctx"], u, v, st["flags"], st["prm"])
        return {"u": u, "v": v, "rho": rho, **out}
    if kind == "adjoint":
        leaves = [t.detach().requires_grad_() for t in (st["u"], st["v"], st["phi0"])]
        outs = hp_autograd.project_fixed(*leaves, st["flags"], st["ctx"], case["k"])
        grads = torch.autograd.grad(outs, leaves, (st["gu"], st["gv"], st["gp"]))
        names = ("u", "v", "p", "gu_star", "gv_star", "g_phi0")
        return dict(zip(names, [t.detach() for t in outs] + list(grads)))
    u, v = st["uw"].copy_(st["u"]), st["vw"].copy_(st["v"])
    if kind == "hybrid":
        out = hp.hp_project_hybrid(st["ctx"], st["cnn"], u, v, st["flags"], st["prm"])
    else:
        out = hp.hp_project(st["ctx"], u, v, st["flags"], st["prm"])
    return {"u": u, "v": v, **out}


# -------------------------------------------------------------------- work

def _branches(arch):
    """(scale, cin, cout, kernel size) of every convolution in network order."""
    layers = hp_training.ARCH_LAYERS[arch]
    if arch == "unet":
        scales = [1, 1, 2, 2, 4, 4, 8, 8, 16, 16, 16, 8, 8, 4, 4, 2, 2, 1, 1, 1]
    elif arch == "monoscale":
        scales = [1] * 9
    else:
        scales = [4] * 5 + [2] * 7 + [1] * 7
    return [(s, *(tuple(l) + (3,))[:3]) for s, l in zip(scales, layers)]


def _net_flops(case):
    px = case["batch"] * case["ny"] * case["nx"]
    return sum(2.0 * k * k * ci * co * px / (s * s) for s, ci, co, k in _branches(case["arch"]))


# FP32 operations of one Jacobi update and its residual's share of E_1
SWEEP_FLOPS = 9


def work(case):
    kind = case["kind"]
    cells = float(case["batch"] * case["ny"] * case["nx"])
    if kind == "conv":
        io, w = case["cin"] + case["cout"], 9.0 * case["cin"] * case["cout"]
        return {"bytes": 2.0 * cells * io + 2.0 * w, "flops": 2.0 * w * cells}
    if kind == "cnn":
        return {"bytes": 9.0 * cells, "flops": _net_flops(case)}
    if kind == "train":  # forward, input gradient and weight gradient
        n = sum(k * k * ci * co + co for _, ci, co, k in _branches(case["arch"]))
        return {"bytes": 9.0 * cells + 6.0 * n, "flops": 3.0 * _net_flops(case)}
    if kind == "advect":
        return {"bytes": 25.0 * cells, "flops": (150.0 if case["scheme"] else 60.0) * cells}
    if kind == "adjoint":
        return {"bytes": 58.0 * cells, "flops": (2 * SWEEP_FLOPS * case["k"] + 40.0) * cells}
    sweeps = case["max_iters"] if kind == "hybrid" else case["sweeps"]
    w = {"bytes": 21.0 * cells, "flops": (SWEEP_FLOPS * sweeps + 20.0) * cells}
    if kind == "step":
        w["bytes"] += 13.0 * cells
        w["flops"] += (150.0 if case["scheme"] else 60.0) * cells
    if kind == "hybrid":
        w["flops"] += _net_flops(case)
    return w


# ------------------------------------------------------------ FP64, by torch

def _open(flags, open_top):
    """Open faces of every cell (west, east, north, south) as FP64 0 or 1."""
    fl = (flags == 0).double()
    o = [torch.zeros_like(fl) for _ in range(4)]
    o[0][:, :, 1:] = fl[:, :, 1:] * fl[:, :, :-1]
    o[1][:, :, :-1] = o[0][:, :, 1:]
    o[2][:, 1:] = fl[:, 1:] * fl[:, :-1]
    o[3][:, :-1] = o[2][:, 1:]
    if open_top:
        o[2][:, 0] = fl[:, 0]
    return o


def _divergence64(u, v, o, inflow):
    """inflow: 0 or 1 per column, the bottom faces that keep their velocity."""
    s = o[3].clone()
    s[:, -1] += inflow
    return o[1] * u[:, :, 1:] - o[0] * u[:, :, :-1] + s * v[:, 1:] - o[2] * v[:, :-1]


def _neighbour_sum(o, phi):
    """sum over open faces of (phi_nb - phi); exterior values are zero."""
    p = F.pad(phi, (1, 1, 1, 1))
    return (o[0] * (p[:, 1:-1, :-2] - phi) + o[1] * (p[:, 1:-1, 2:] - phi)
            + o[2] * (p[:, :-2, 1:-1] - phi) + o[3] * (p[:, 2:, 1:-1] - phi))


def _sweeps64(o, div, phi, threshold, cap, fixed):
    """Every grid to its first k with mean |r_k| <= threshold, or the cap."""
    n = o[0] + o[1] + o[2] + o[3]
    inv = torch.where(n > 0, 1.0 / n.clamp(min=1), 0.0)
    o = [t * (n > 0) for t in o]
    B = div.shape[0]
    active = torch.ones((B, 1, 1), dtype=torch.bool, device=div.device)
    iters = torch.zeros(B, dtype=torch.int32, device=div.device)
    for k in range((fixed or cap) + 1):
        r = div - _neighbour_sum(o, phi)
        if not fixed:
            active = active & (r.abs().mean((1, 2), keepdim=True) > threshold)
        if k == (fixed or cap) or (k % 64 == 0 and not bool(active.any())):
            break
        phi = torch.where(active, phi - r * inv, phi)
        iters += active.reshape(-1).to(torch.int32)
    return phi, iters, ~active.reshape(-1)


def _project64(case, u, v, flags, phi=None):
    u, v = u.double(), v.double()
    open_top = bool(case.get("open_top"))
    o = _open(flags, open_top)
    B, ny, nx = flags.shape
    inflow = torch.zeros((B, nx), dtype=torch.float64, device=u.device)
    if open_top:
        x0, x1 = _inlet(nx)
        inflow[:, x0:x1] = (flags[:, -1, x0:x1] == 0).double()
    div = _divergence64(u, v, o, inflow)
    keep = (o[0] + o[1] + o[2] + o[3]) > 0
    phi = torch.zeros_like(div) if phi is None else phi.double() * keep
    fixed = case.get("fixed", 0)
    phi, iters, conv = _sweeps64(o, div, phi, case["threshold"], case["max_iters"], fixed)
    un, vn = torch.zeros_like(u), torch.zeros_like(v)
    un[:, :, 1:-1] = o[0][:, :, 1:] * (u[:, :, 1:-1] - (phi[:, :, 1:] - phi[:, :, :-1]))
    vn[:, 1:-1] = o[2][:, 1:] * (v[:, 1:-1] - (phi[:, 1:] - phi[:, :-1]))
    if open_top:
        vn[:, 0] = o[2][:, 0] * (v[:, 0] - phi[:, 0])
        vn[:, -1] = inflow * v[:, -1]
    d = _divergence64(un, vn, o, inflow).abs()
    dt = PLUME["dt"] if case["kind"] == "step" else 1.0
    return {"u": un, "v": vn, "p": phi / dt, "iters": iters, "e1": d.mean((1, 2)),
            "einf": d.amax((1, 2)), "converged": conv.to(torch.uint8) if not fixed
            else torch.ones_like(conv, dtype=torch.uint8)}


def _sample(q, x, y, ox, oy, corners=False):
    B, my, mx = q.shape
    tx, ty = (x - ox).clamp(0, mx - 1), (y - oy).clamp(0, my - 1)
    i0, j0 = tx.floor().clamp(max=max(mx - 2, 0)), ty.floor().clamp(max=max(my - 2, 0))
    fx, fy = tx - i0, ty - j0
    i0, j0 = i0.long(), j0.long()
    i1, j1 = (i0 + 1).clamp(max=mx - 1), (j0 + 1).clamp(max=my - 1)
    at = lambda j, i: q.reshape(B, -1).gather(1, (j * mx + i).reshape(B, -1)).reshape(x.shape)  # noqa: E731
    c = [at(j0, i0), at(j0, i1), at(j1, i0), at(j1, i1)]
    if corners:
        c = torch.stack(c)
        return c.amin(0), c.amax(0)
    return (c[0] * (1 - fx) + c[1] * fx) * (1 - fy) + (c[2] * (1 - fx) + c[3] * fx) * fy


def _advect64(case, u, v, rho, flags):
    u, v, rho = u.double(), v.double(), rho.double()
    dt = PLUME["dt"]
    B, ny, nx = rho.shape
    x0, x1 = _inlet(nx)
    rho[:, -1, x0:x1] = float(np.float32(PLUME["rho_in"]))
    out = []
    for q, ox, oy in ((rho, 0.5, 0.5), (u, 0.0, 0.5), (v, 0.5, 0.0)):
        x = (torch.arange(q.shape[2], device=q.device).double() + ox)[None, None].expand(q.shape)
        y = (torch.arange(q.shape[1], device=q.device).double() + oy)[None, :, None].expand(q.shape)
        vx, vy = _sample(u, x, y, 0.0, 0.5), _sample(v, x, y, 0.5, 0.0)
        new = _sample(q, x - dt * vx, y - dt * vy, ox, oy)
        if case["scheme"]:
            lo, hi = _sample(q, x - dt * vx, y - dt * vy, ox, oy, corners=True)
            back = _sample(new, x + dt * vx, y + dt * vy, ox, oy)
            new = torch.minimum(torch.maximum(new + 0.5 * (q - back), lo), hi)
        out.append(new)
    rho, u, v = out
    v[:, 1:-1] += dt * PLUME["gravity"] * (0.5 * (rho[:, :-1] + rho[:, 1:]) - PLUME["rho_amb"])
    o = _open(flags, False)
    uz, vz = torch.zeros_like(u), torch.zeros_like(v)
    uz[:, :, 1:-1] = o[0][:, :, 1:] * u[:, :, 1:-1]
    vz[:, 1:-1] = o[2][:, 1:] * v[:, 1:-1]
    return uz, vz, rho


def _adjoint64(case, st):
    leaves = [st[k].double().requires_grad_() for k in ("u", "v", "phi0")]
    u, v, phi = leaves
    o = _open(st["flags"], False)
    n = o[0] + o[1] + o[2] + o[3]
    inv = torch.where(n > 0, 1.0 / n.clamp(min=1), 0.0)
    div = _divergence64(u, v, o, torch.zeros_like(n[:, 0]))
    phi = phi * (n > 0)
    for _ in range(case["k"]):
        phi = phi - (div - _neighbour_sum(o, phi)) * inv
    un = F.pad(o[0][:, :, 1:] * (u[:, :, 1:-1] - (phi[:, :, 1:] - phi[:, :, :-1])), (1, 1))
    vn = F.pad(o[2][:, 1:] * (v[:, 1:-1] - (phi[:, 1:] - phi[:, :-1])), (0, 0, 1, 1))
    outs = (un, vn, phi)
    grads = torch.autograd.grad(outs, leaves, [st[k].double() for k in ("gu", "gv", "gp")])
    names = ("u", "v", "p", "gu_star", "gv_star", "g_phi0")
    return dict(zip(names, [t.detach() for t in outs] + list(grads)))


def _conv64(h, w, b, relu):
    if w.shape[2] == 3:
        h = F.pad(h, (1, 1, 1, 1), mode="replicate")
    y = F.conv2d(h, w, b)
    return torch.relu(y) if relu else y


def _up64(h):
    return F.interpolate(h, scale_factor=2, mode="bilinear", align_corners=False)


def _net64(arch, flat, div, flags):
    """phi_hat (with gradients to `flat`) and s of the FP64 network."""
    layers, off = [], 0
    for s, ci, co, k in _branches(arch):
        w = flat[off:off + k * k * ci * co].reshape(co, ci, k, k)
        off += k * k * ci * co
        layers.append((s, w, flat[off:off + co]))
        off += co
    fluid = flags == 0
    s = (div.abs() * fluid).sum((1, 2)) / fluid.sum((1, 2)).clamp(min=1)
    s = torch.where(s > 0, s, torch.ones_like(s))
    x0 = torch.stack([div / s[:, None, None], (~fluid).double()], 1)
    if arch == "unet":
        it = iter(enumerate(layers))

        def conv(h):
            l, (_, w, b) = next(it)
            return _conv64(h, w, b, l < len(layers) - 2)
        h, skips = x0, []
        for level in range(4):
            h = conv(conv(F.max_pool2d(h, 2) if level else h))
            skips.append(h)
        h = conv(conv(conv(F.max_pool2d(h, 2))))
        for level in (3, 2, 1, 0):
            h = conv(conv(torch.cat([_up64(h), skips[level]], 1)))
        return conv(h)[:, 0], s
    prev = None
    for scale in sorted({l[0] for l in layers}, reverse=True):
        part = [l for l in layers if l[0] == scale]
        h = F.avg_pool2d(x0, scale) if scale > 1 else x0
        if prev is not None:
            h = torch.cat([h, _up64(prev)], 1)
        for l, (_, w, b) in enumerate(part):
            h = _conv64(h, w, b, l < len(part) - 2)
        prev = h
    return prev[:, 0], s


def _train64(case, st, flat):
    flat = flat.requires_grad_()
    div, fl, target = st["div"].double(), st["flags"], st["target"].double()
    B = div.shape[0]
    o = _open(fl, False)
    total = torch.zeros(1, dtype=torch.float64, device=div.device)
    grad = torch.zeros_like(flat)
    for b in range(0, B, 8):  # chunks: the tape of a whole batch is large
        sl = slice(b, b + 8)
        phi, s = _net64(case["arch"], flat, div[sl], fl[sl])
        fluid = (fl[sl] == 0).double()
        cnt = fluid.sum((1, 2), keepdim=True).clamp(min=1)
        t, d = target[sl] / s[:, None, None], div[sl] / s[:, None, None]
        e = phi - t
        var = lambda q: (((q - (q * fluid).sum((1, 2), keepdim=True) / cnt) * fluid) ** 2).sum((1, 2))  # noqa: E731
        vt, d2 = var(t), (d * d).sum((1, 2))
        ob = [q[sl] for q in o]
        r = (d - _neighbour_sum(ob, phi)) * ((ob[0] + ob[1] + ob[2] + ob[3]) > 0)
        loss = torch.where(vt > 0, var(e) / vt.clamp(min=1e-300), 0.0)
        loss = loss + torch.where(d2 > 0, LAMBDA * (r * r).sum((1, 2)) / d2.clamp(min=1e-300), 0.0)
        loss = loss.sum() / B
        grad += torch.autograd.grad(loss, flat)[0]
        total += loss.detach()
    return {"grad": grad, "loss": total}


# FP64 convolutions beyond this many operations take too long
MOST_FP64_FLOPS = 2e12


@torch.no_grad()
def _exact(case, seed):
    kind = case["kind"]
    if kind in ("cnn", "hybrid", "train", "conv") and work(case)["flops"] > MOST_FP64_FLOPS:
        return None
    if kind == "conv":
        x, w, b = _conv_inputs(case, seed)
        y = [_conv64(x[i:i + 1].double().permute(0, 3, 1, 2), w.double().permute(2, 3, 0, 1),
                     b.double(), case["relu"]).permute(0, 2, 3, 1) for i in range(x.shape[0])]
        return torch.cat(y).contiguous()
    if kind == "train":
        div, fl, target = _train_inputs(case, seed)
        flat = torch.from_numpy(_params(case, seed)).to(_dev()).double()
        with torch.enable_grad():
            return _train64(case, dict(div=div, flags=fl, target=target), flat)
    g, u, v, fl = _flow(case, seed)
    B, ny, nx = fl.shape
    if kind in ("step", "advect"):
        rho = _density(g, B, ny, nx)
        u, v, rho = _advect64(case, u, v, rho, fl)
        if kind == "advect":
            return {"u": u, "v": v, "rho": rho}
        return {"rho": rho, **_project64(case, u, v, fl)}
    if kind == "adjoint":
        s = lambda *d: torch.randn(d, generator=g).to(_dev())  # noqa: E731
        st = dict(u=u, v=v, flags=fl, phi0=s(B, ny, nx), gu=s(B, ny, nx + 1),
                  gv=s(B, ny + 1, nx), gp=s(B, ny, nx))
        with torch.enable_grad():
            return _adjoint64(case, st)
    if kind in ("cnn", "hybrid"):
        div = _divergence(u, v, fl).double()
        flat = torch.from_numpy(_params(case, seed)).to(_dev()).double()
        parts = [_net64(case["arch"], flat, div[b:b + 1], fl[b:b + 1]) for b in range(B)]
        phi_hat, s = (torch.cat(t) for t in zip(*parts))
        if kind == "cnn":
            return {"phi_hat": phi_hat, "s": s}
        return _project64(case, u, v, fl, phi=phi_hat * s[:, None, None])
    return _project64(case, u, v, fl)


def exact(case, seed):
    return _exact(case, seed)
