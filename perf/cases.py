"""What a user of this flood model has it do, as measurable passes.

Every case builds its inputs from a seed on the GPU, keeps the handle a program
would keep, and runs through the package's public entry points.  Forward cases
are a run loop: each pass advances the simulation by some steps and reads its
whole state into device tensors.  Calibration cases are one evaluation of a
gauge-misfit loss and its gradient with respect to the Manning field.

``exact`` is the method (local-inertial faces, depth update, Manning boundary
faces, the time-step rule) in 64-bit torch, without the package's code; its
gradient is torch's.
"""
from __future__ import annotations

import ctypes as C
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as TF

import paper_2204_10323_gb300 as F
from paper_2204_10323_gb300.autograd import FloodRun

DEV = "cuda"
G, H_DRY, ALPHA, E = 9.81, 1e-3, 0.7, 16


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest calls: a 128^2 channel reach at 10 m, one CFL epoch a call, as a coupled
        # or interactive program takes it; the launches and the inflow solve are what it waits for
        dict(name="channel_128", kind="step", nx=128, ny=128, dx=10.0, steps=16, dtype="f32", terrain="channel",
             wet=0.0, theta=1.0, friction=0, parts=1),
        # the same reach in double precision, the path that results are checked against
        dict(name="channel_128_f64", kind="step", nx=128, ny=128, dx=10.0, steps=16, dtype="f64", terrain="channel",
             wet=0.0, theta=1.0, friction=0, parts=1),
        # a double-precision run of an ordinary grid of odd size
        dict(name="valley_1001x777_f64", kind="step", nx=1001, ny=777, dx=5.0, steps=16, dtype="f64",
             terrain="fractal", wet=0.3, theta=1.0, friction=0, parts=1),
        # the calibration grid, forward only: small enough to stay in L2
        dict(name="valley_1024", kind="step", nx=1024, ny=1024, dx=5.0, steps=64, dtype="f32", terrain="fractal",
             wet=0.3, theta=1.0, friction=0, parts=1),
        # the ordinary grid: 2048^2 at 5 m
        dict(name="valley_2048", kind="step", nx=2048, ny=2048, dx=5.0, steps=64, dtype="f32", terrain="fractal",
             wet=0.3, theta=1.0, friction=0, parts=1),
        # ragged grid with the vector norm in the friction term
        dict(name="ragged_norm", kind="step", nx=3001, ny=1803, dx=5.0, steps=32, dtype="f32", terrain="fractal",
             wet=0.3, theta=1.0, friction=1, parts=1),
        # theta-weighted faces on a smooth channel reach
        dict(name="reach_theta", kind="step", nx=1500, ny=701, dx=10.0, steps=32, dtype="f32", terrain="channel",
             wet=0.0, theta=0.9, friction=0, parts=1),
        # the 1 m grid, the largest run
        dict(name="valley_16384", kind="step", nx=16384, ny=16384, dx=1.0, steps=16, dtype="f32", terrain="fractal",
             wet=0.3, theta=1.0, friction=0, parts=1),
        # 1 x 4 row strips with a halo exchange every 4 steps (the paper's subgrids)
        dict(name="strips_4096", kind="step", nx=4096, ny=4096, dx=2.0, steps=32, dtype="f32", terrain="fractal",
             wet=0.3, theta=1.0, friction=0, parts=4),
        # a scenario sweep: 20 uneven grids, four steps a launch
        dict(name="ensemble_20", kind="ensemble", members=20, steps=64, shapes=0),
        # calibration: forward with gauges, loss, gradient of the Manning field
        dict(name="calibrate_1024", kind="calibrate", nx=1024, ny=1024, dx=5.0, steps=64, dtype="f32", gauges=16,
             checkpoints=12),
        # the 1 m DEM averaged to 4 m
        dict(name="coarsen_16384", kind="coarsen", nx=16384, ny=16384, factor=4, dtype="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["ensemble", "calibrate", "calibrate", "coarsen"])
    if kind == "step":
        dtype = rng.choice(["f32"] * 5 + ["f64"])
        hi = 12000 if dtype == "f32" else 1200
        nx, ny = _log_int(rng, 64, hi), _log_int(rng, 64, hi)
        option = rng.choice(["", "", "", "norm", "theta"])
        if option == "theta":                        # theta < 1 needs smooth terrain
            nx, ny = min(nx, 3000), min(ny, 3000)
        parts = rng.choice([1, 1, 1, 2, 3, 4]) if dtype == "f32" and not option else 1
        smooth = option == "theta" or max(nx, ny) < 200
        return dict(kind="step", nx=nx, ny=ny, dx=10.0 if smooth else rng.choice([1.0, 2.0, 5.0]),
                    steps=16 * rng.choice([1, 1, 2, 4]) if nx * ny < 1 << 26 else 16, dtype=dtype,
                    terrain="channel" if smooth else "fractal", wet=0.0 if smooth else rng.choice([0.0, 0.1, 0.3, 0.5]),
                    theta=0.9 if option == "theta" else 1.0, friction=1 if option == "norm" else 0, parts=parts)
    if kind == "ensemble":
        return dict(kind="ensemble", members=rng.randint(3, 20), steps=16 * rng.choice([1, 2, 4]),
                    shapes=rng.randint(1, 1000))
    if kind == "calibrate":
        dtype = rng.choice(["f32", "f32", "f64"])
        hi = 1400 if dtype == "f32" else 400
        return dict(kind="calibrate", nx=_log_int(rng, 96, hi), ny=_log_int(rng, 96, hi), dx=5.0,
                    steps=rng.randint(8, 64 if dtype == "f32" else 40), dtype=dtype, gauges=rng.randint(1, 24),
                    checkpoints=rng.choice([4, 12, 40]))
    dtype = rng.choice(["f32", "f32", "f64"])
    hi = 16384 if dtype == "f32" else 8192
    return dict(kind="coarsen", nx=_log_int(rng, 100, hi), ny=_log_int(rng, 100, hi), factor=rng.choice([2, 3, 4, 5, 8]),
                dtype=dtype)


def work(case):
    """The state and the static fields read once, the state written once; about 45 operations a cell and step."""
    kind = case["kind"]
    if kind == "coarsen":
        e = 4 if case["dtype"] == "f32" else 8
        n = case["nx"] * case["ny"]
        m = -(-case["nx"] // case["factor"]) * -(-case["ny"] // case["factor"])
        return {"bytes": (n + m) * e, "flops": n}
    if kind == "ensemble":
        n = sum(nx * ny for nx, ny in _shapes(case))
        return {"bytes": 32 * n, "flops": 45 * n * case["steps"]}
    e = 4 if case["dtype"] == "f32" else 8
    n = case["nx"] * case["ny"]
    if kind == "calibrate":                          # forward, and about three times that in reverse
        return {"bytes": 8 * e * n, "flops": 4 * 45 * n * case["steps"]}
    return {"bytes": 8 * e * n, "flops": 45 * n * case["steps"]}


# --------------------------------------------------------------------------- inputs
def _rand(gen, ny, nx):
    return torch.rand((ny, nx), generator=gen, device=DEV, dtype=torch.float32) * 2.0 - 1.0


def _fractal(nx, ny, relief, gen):
    """Octaves of smooth noise, the amplitude falling by 0.6 per halving of the cell spacing."""
    a = torch.zeros((ny, nx), device=DEV, dtype=torch.float32)
    span, amp = max(nx, ny), 1.0
    while span >= 2:
        my, mx = ny // span + 2, nx // span + 2
        f = _rand(gen, my, mx)[None, None]
        a += amp * TF.interpolate(f, size=(ny, nx), mode="bilinear", align_corners=False)[0, 0]
        del f
        span, amp = span // 2, amp * 0.6
    lo, hi = a.min(), a.max()
    return (a - lo) * (relief / (hi - lo))


def _terrain(case, gen):
    """Bed and roughness in the case's precision, the inflow rows (j0, j1), and the channel's centre rows."""
    nx, ny, dx = case["nx"], case["ny"], case["dx"]
    ic = torch.arange(nx, device=DEV, dtype=torch.float32) + 0.5
    jc = torch.arange(ny, device=DEV, dtype=torch.float32) + 0.5
    if case.get("terrain", "fractal") == "channel":  # tilted plane, sinusoidal channel 3 m deep, +-0.1 m noise
        yc = ny / 2 + ny / 8 * torch.sin(2 * math.pi * ic / nx)
        half = max(1.5, min(4.0, ny / 8))
        chan = (jc[:, None] - yc[None, :]).abs() < half
        z = 100.0 - 1e-3 * (ic * dx)[None, :] - 3.0 * chan + 0.1 * _rand(gen, ny, nx)
        n = torch.full((ny, nx), 0.03, device=DEV) + 0.002 * _rand(gen, ny, nx)
    else:                                            # fractal relief, meandering channel with a falling bed
        z = _fractal(nx, ny, min(40.0, 0.008 * dx * max(nx, ny)), gen)
        yc = ny / 2 + 0.098 * ny * torch.sin(4 * math.pi * ic / nx) + 0.039 * ny * torch.sin(2 * math.pi * ic / (0.17 * nx))
        half = max(1.5, min(60.0 / dx, ny / 16))
        cj = yc.long().clamp(0, ny - 1)
        bed = torch.cummin(z[cj, torch.arange(nx, device=DEV)] - min(4.0, 0.002 * dx * max(nx, ny)), 0).values
        chan = (jc[:, None] - yc[None, :]).abs() < half
        z = torch.where(chan, torch.minimum(z, bed[None, :]), z)
        n = torch.where(chan, 0.035, 0.06).to(torch.float32) + 0.002 * _rand(gen, ny, nx)
    y0 = float(yc[0])
    j0, j1 = max(0, int(y0 - half) - 2), min(ny, int(y0 + half) + 3)
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    return z.to(dt), n.to(dt), (j0, j1), yc


def _depth(case, z):
    """Depth under a gently tilted water surface that wets the fraction `wet` of the cells (0: dry)."""
    if not case.get("wet"):
        return torch.zeros_like(z)
    nx, ny, dx = case["nx"], case["ny"], case["dx"]
    fall = (1e-4 * dx * (torch.arange(nx, device=DEV, dtype=torch.float32) + 0.5)).to(z.dtype)
    key = (z + fall[None, :])[:: max(1, ny // 512), :: max(1, nx // 512)].reshape(-1)
    level = key.kthvalue(max(1, int(case["wet"] * key.numel()))).values
    return (level - fall[None, :] - z).clamp_(min=0.0).to(z.dtype)


def _problem(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    z, n, (j0, j1), yc = _terrain(case, gen)
    nx, ny, dx = case["nx"], case["ny"], case["dx"]
    peak = (2.0 + 2.0 * float(torch.rand((), generator=gen, device=DEV))) * (j1 - j0) * dx * 0.5
    secs = [SimpleNamespace(side=F.XMIN, kind=F.INFLOW, frac_start=j0 / ny, frac_end=j1 / ny, slope=1e-3,
                            t_s=np.array([0.0, 600.0, 1e6]), q_m3s=np.array([0.5 * peak, peak, peak])),
            SimpleNamespace(side=F.XMAX, kind=F.OUTFLOW, frac_start=0.0, frac_end=1.0, slope=1e-3, t_s=None, q_m3s=None)]
    cal = case["kind"] == "calibrate"                # a gradient holds the time steps fixed
    opts = SimpleNamespace(g=G, h_dry=H_DRY, cfl_alpha=ALPHA, dt_cap=0.1 * dx, dt_const=0.02 * dx,
                           dt_mode=1 if cal else 0, epoch_steps=E, bc_form=0, theta=case.get("theta", 1.0),
                           friction=case.get("friction", 0))
    p = SimpleNamespace(name="case", nx=nx, ny=ny, dx=dx, z=z, n=n, sections=secs, opts=opts, h0=None, qx0=None,
                        qy0=None, yc=yc, inflow=(j0, j1))
    return p, _depth(case, z), gen


def _on_host(p):
    """The problem as the handles take it: bed and roughness as host arrays."""
    q = SimpleNamespace(**vars(p))
    q.z, q.n = p.z.cpu().numpy(), p.n.cpu().numpy()
    return q


def _prec(case):
    return F.F32 if case["dtype"] == "f32" else F.F64


_SHAPES = [(256, 256), (512, 512), (1024, 1024), (1536, 1024), (2048, 2048)]


def _shapes(case):
    """The scenarios' grids: the five sizes in turn, or odd ones around them."""
    if not case["shapes"]:
        return [_SHAPES[k % 5] for k in range(case["members"])]
    r = np.random.RandomState(case["shapes"])
    return [tuple(int(v * r.uniform(0.6, 1.0)) for v in _SHAPES[r.randint(0, 5)]) for _ in range(case["members"])]


def _member_case(case, k, shape):
    return dict(kind="step", nx=shape[0], ny=shape[1], dx=5.0, steps=case["steps"], dtype="f32", terrain="fractal",
                wet=0.3, theta=1.0, friction=0)


def _calibration(case, seed):
    """Wet valley, gauges in the channel, the observed depths there, and the roughness to differentiate."""
    p, h, gen = _problem(dict(case, terrain="fractal", wet=0.3), seed)
    k = case["gauges"]
    i = torch.linspace(2, case["nx"] - 3, k, device=DEV).long().cpu().numpy()
    j = p.yc.long().clamp(0, case["ny"] - 1).cpu().numpy()[i]
    gauges = np.stack([i, j], 1).astype(np.int64)
    at = h[torch.from_numpy(j).to(DEV), torch.from_numpy(i).to(DEV)].double()
    obs = at[None, :] * (0.6 + 0.2 * torch.rand((case["steps"], k), generator=gen, device=DEV).double())
    return p, h, gauges, obs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "coarsen":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        z = 40.0 * torch.rand((case["ny"], case["nx"]), generator=gen, device=DEV,
                              dtype=torch.float32 if case["dtype"] == "f32" else torch.float64)
        return dict(kind=kind, z=z, factor=case["factor"])
    if kind == "ensemble":
        probs, depths = [], []
        for k, shape in enumerate(_shapes(case)):
            p, h, _ = _problem(_member_case(case, k, shape), seed * 64 + k)
            probs.append(_on_host(p))
            depths.append(h)
        ens = F.Ensemble(probs)
        ens.set_launch(2, 256, 64)                   # the launch shape the autotuner picks for such mixes
        ens.set_kernel(F.KERNEL_TILED, 4)
        for m, h in zip(ens.members, depths):
            m.write_state(h)
        return dict(kind=kind, ens=ens, steps=case["steps"], out=[_buffers(m.nx, m.ny, h.dtype) for m, h in zip(ens.members, depths)])
    if kind == "calibrate":
        p, h, gauges, obs = _calibration(case, seed)
        sim = F.Sim(_on_host(p), precision=_prec(case))
        return dict(kind=kind, sim=sim, h=h, n=p.n, gauges=gauges, obs=obs, steps=case["steps"],
                    checkpoints=case["checkpoints"])
    p, h, _ = _problem(case, seed)
    if case["parts"] > 1:
        sim = F.Decomp(_on_host(p), case["parts"], 4, precision=_prec(case))
    else:
        sim = F.Sim(_on_host(p), precision=_prec(case))
    sim.write_state(h)
    return dict(kind=kind, sim=sim, steps=case["steps"], parts=case["parts"], out=_buffers(case["nx"], case["ny"], h.dtype))


# --------------------------------------------------------------------------- one pass
def _buffers(nx, ny, dtype):
    return {"h": torch.empty((ny, nx), dtype=dtype, device=DEV), "qx": torch.empty((ny, nx + 1), dtype=dtype, device=DEV),
            "qy": torch.empty((ny + 1, nx), dtype=dtype, device=DEV)}


_FIELDS = (("h", F.FIELD_H), ("qx", F.FIELD_QX), ("qy", F.FIELD_QY))


def _read(handle, out):
    for key, field in _FIELDS:
        t = out[key]
        F.flood_read(handle, field, C.c_void_p(t.data_ptr()), t.numel() * t.element_size(), 1)
    return out


def run(state):
    kind = state["kind"]
    if kind == "coarsen":
        return F.coarsen(state["z"], state["factor"])
    if kind == "ensemble":
        state["ens"].step(state["steps"])
        return [_read(m.h, o) for m, o in zip(state["ens"].members, state["out"])]
    sim = state["sim"]
    if kind == "calibrate":                          # from the same start each time, as an optimiser's iteration
        sim.write_state(state["h"])
        sim.set_clock(0.0, 0, 0.0)
        n = state["n"].detach().requires_grad_(True)
        series = FloodRun.apply(n, sim, state["gauges"], state["steps"], state["checkpoints"])
        ((series - state["obs"]) ** 2).sum().backward()
        return {"depths": series.detach().to(n.dtype), "grad_n": n.grad}
    sim.step(state["steps"])
    if state["parts"] == 1:
        return _read(sim.h, state["out"])
    for key, field in _FIELDS:
        t = state["out"][key]
        F._dec_check(F.lib().flood_decomp_read(sim.h, field, C.c_void_p(t.data_ptr()), t.numel() * t.element_size(), 1), sim.h)
    return state["out"]


# --------------------------------------------------------------------------- the same in 64 bits
def _inflow(p, sec, times, z, n):
    """Unit-width inflow of every section cell at each of the times: the level W at which the cells'
    Manning discharges sum to Q, by bisection, then each cell's share (n may carry a gradient)."""
    j0, j1 = p.inflow
    zc, nc = z[j0:j1, 0], n[j0:j1, 0]
    Q = torch.from_numpy(np.interp(times, sec.t_s, sec.q_m3s)).to(DEV)[:, None]
    s = math.sqrt(sec.slope)

    def cells(W, nn):
        d = (W - zc[None, :]).clamp(min=0.0)
        return p.dx * d ** (5.0 / 3.0) * s / nn[None, :]

    with torch.no_grad():
        lo = zc.min().expand(Q.shape).clone()
        top = 1.0
        while bool((cells(lo + top, nc).sum(1, keepdim=True) < Q).any()):
            top *= 2.0
        hi = lo + top
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            less = cells(mid, nc).sum(1, keepdim=True) < Q
            lo, hi = torch.where(less, mid, lo), torch.where(less, hi, mid)
        W = hi
        slope = (p.dx * (5.0 / 3.0) * (W - zc[None, :]).clamp(min=0.0) ** (2.0 / 3.0) * s / nc[None, :]).sum(1, keepdim=True)
    if n.requires_grad:                              # one Newton step carries dW/dn
        W = W - (cells(W, nc).sum(1, keepdim=True) - Q) / slope
    w = cells(W, nc)
    return w * (Q / w.sum(1, keepdim=True)) / p.dx


def _faces(q, qn, qm, hL, zL, nL, hR, zR, nR, dt, dx):
    eL, eR = hL + zL, hR + zR
    hf = torch.where(eL >= eR, eL, eR) - torch.maximum(zL, zR)
    wet = hf > H_DRY
    hf = torch.where(wet, hf, 1.0)
    num = qn - (G * dt / dx) * hf * (eR - eL)
    nf = 0.5 * (nL + nR)
    return torch.where(wet, num / (1.0 + (G * dt) * nf * nf * qm * hf ** (-7.0 / 3.0)), 0.0)


def _step(p, h, qx, qy, z, n, dt, qin):
    o, dx = p.opts, p.dx
    x, y = qx[:, 1:-1], qy[1:-1, :]
    xn, yn = x, y
    if o.theta != 1.0:
        w = 0.5 * (1.0 - o.theta)
        xn = o.theta * x + w * (qx[:, :-2] + qx[:, 2:])
        yn = o.theta * y + w * (qy[:-2, :] + qy[2:, :])
    xm, ym = x.abs(), y.abs()
    if o.friction:
        xo = 0.25 * ((qy[:-1, :-1] + qy[:-1, 1:]) + (qy[1:, :-1] + qy[1:, 1:]))
        yo = 0.25 * ((qx[:-1, :-1] + qx[:-1, 1:]) + (qx[1:, :-1] + qx[1:, 1:]))
        xm, ym = torch.sqrt(x * x + xo * xo), torch.sqrt(y * y + yo * yo)
    fx = _faces(x, xn, xm, h[:, :-1], z[:, :-1], n[:, :-1], h[:, 1:], z[:, 1:], n[:, 1:], dt, dx)
    fy = _faces(y, yn, ym, h[:-1], z[:-1], n[:-1], h[1:], z[1:], n[1:], dt, dx)
    j0, j1 = p.inflow
    west = TF.pad(qin, (j0, p.ny - j1))[:, None]
    hl = h[:, -1:]
    wet = hl > H_DRY
    east = torch.where(wet, torch.where(wet, hl, 1.0) ** (5.0 / 3.0) * math.sqrt(p.sections[1].slope) / n[:, -1:], 0.0)
    qx2 = torch.cat([west, fx, east], 1)
    qy2 = TF.pad(fy, (0, 0, 1, 1))
    del fx, fy
    hn = h + (dt / dx) * ((qx2[:, :-1] - qx2[:, 1:]) + (qy2[:-1] - qy2[1:]))
    return hn.clamp(min=0.0), qx2, qy2


def _advance(p, h, z, n, steps, gauges=None):
    """`steps` steps from depth h at rest at t = 0; with gauges, the depths there after every step."""
    qx = torch.zeros((p.ny, p.nx + 1), device=DEV, dtype=torch.float64)
    qy = torch.zeros((p.ny + 1, p.nx), device=DEV, dtype=torch.float64)
    t, series = 0.0, []
    for k in range(steps):
        if k % E == 0:
            top = float(h.detach().max())
            dt = p.opts.dt_const if p.opts.dt_mode else min(p.opts.dt_cap, ALPHA * p.dx / math.sqrt(G * top)) if top > 0 else p.opts.dt_cap
            times = [t]
            for _ in range(E):
                times.append(times[-1] + dt)
            qin = _inflow(p, p.sections[0], np.array(times[:E]), z, n)
        h, qx, qy = _step(p, h, qx, qy, z, n, dt, qin[k % E])
        t = times[k % E + 1]
        if gauges is not None:
            series.append(h[gauges[:, 1], gauges[:, 0]])
    return (h, qx, qy) if gauges is None else torch.stack(series)


def exact(case, seed):
    kind = case["kind"]
    if kind == "coarsen":
        z, f = prepare(case, seed)["z"].double(), case["factor"]
        py, px = -z.shape[0] % f, -z.shape[1] % f
        ones = TF.pad(torch.ones_like(z), (0, px, 0, py)) if px or py else None
        z = TF.pad(z, (0, px, 0, py))
        my, mx = z.shape[0] // f, z.shape[1] // f
        total = z.view(my, f, mx, f).sum((1, 3))
        return total / (f * f if ones is None else ones.view(my, f, mx, f).sum((1, 3)))
    if kind == "ensemble":
        out = []
        for k, shape in enumerate(_shapes(case)):
            p, h, _ = _problem(_member_case(case, k, shape), seed * 64 + k)
            out.append(dict(zip(("h", "qx", "qy"), _advance(p, h.double(), p.z.double(), p.n.double(), case["steps"]))))
        return out
    if kind == "calibrate":
        if case["nx"] * case["ny"] * case["steps"] > 1 << 27:
            return None                              # torch's graph of every step would not fit
        p, h, gauges, obs = _calibration(case, seed)
        n = p.n.double().requires_grad_(True)
        at = torch.from_numpy(gauges).to(DEV)
        series = _advance(p, h.double(), p.z.double(), n, case["steps"], at)
        ((series - obs) ** 2).sum().backward()
        return {"depths": series.detach(), "grad_n": n.grad}
    p, h, _ = _problem(case, seed)
    z, n = p.z.double(), p.n.double()
    p.z = p.n = None
    return dict(zip(("h", "qx", "qy"), _advance(p, h.double(), z, n, case["steps"])))
