"""Performance cases of the red-black Gauss-Seidel framework: what its users call it for.

A case is one call sequence through the public entry points, over inputs made on the GPU:

  sweep    a fixed number of sweeps of one 2D problem in a kept solver: load the problem,
           sweep, take the residual, read the solution (the paper's experiment: fixed
           iteration counts); fma selects the bit-exact or the fused FP64 update
  solve    rbgs_solve on one 2D problem with the residual checked at intervals, FP64 or the
           FP32 + FP64 refinement, stopped by its sweep limit
  batched  rbgs_solve_batched over independent problems of uneven sizes
  sweep3d  the 7-point variant: create the solver for a problem, sweep, residual, solution
  train    forward, loss and backward of one U-Net training batch (gradients out)
  guess    the learned initial guess of one problem at full resolution

Sizes are those of the repository's own workloads: 255^2 is the small configuration, 511^2
the time-to-residual comparison, 1023^2 and 4095^2 the learned-guess grids, 8192^2 the
mixed-precision workload, 16384^2 the headline, 511^3 the 3D workload; batches mix sizes up
to 255^2; the network trains on 255^2 problems.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2607_01735_gb300 as rb
from paper_2607_01735_gb300 import unet as ru

DEV = "cuda"
MAX_LUP = 100 * 16384 ** 2  # lattice updates of the largest listed case


def listed():
    return [
        # the smallest regular call: a short run on a tiny grid, all launch latency
        {"name": "sweep-127", "kind": "sweep", "n": 127, "sweeps": 100, "fma": 0},
        # the small configuration: 1000 sweeps with the residual every 100 (ten host checks)
        {"name": "solve-255", "kind": "solve", "n": 255, "sweeps": 1000, "check": 100, "refine": 0},
        # default FP64 sweeps on a middle grid, the learned-guess evaluation's size
        {"name": "sweep-1023", "kind": "sweep", "n": 1023, "sweeps": 200, "fma": 0},
        # default FP64 sweeps on a large grid, the paper's 100 iterations
        {"name": "sweep-4095", "kind": "sweep", "n": 4095, "sweeps": 100, "fma": 0},
        # fused FP64 update on a middle grid of no special size
        {"name": "fused-1500", "kind": "sweep", "n": 1500, "sweeps": 200, "fma": 1},
        # the headline: fused FP64 update at 16384^2, the paper's 100 iterations
        {"name": "fused-16384", "kind": "sweep", "n": 16384, "sweeps": 100, "fma": 1},
        # refinement on the time-to-residual grid
        {"name": "refine-511", "kind": "solve", "n": 511, "sweeps": 1000, "check": 100, "refine": 1},
        # the mixed-precision workload: two corrections of 100 FP32 sweeps
        {"name": "refine-8192", "kind": "solve", "n": 8192, "sweeps": 200, "check": 100, "refine": 1},
        # many small problems at once, three sizes
        {"name": "batched-255", "kind": "batched", "count": 240, "n": 255, "sweeps": 400, "refine": 0},
        # the 3D workload
        {"name": "sweep3d-511", "kind": "sweep3d", "n": 511, "sweeps": 20},
        # one training batch of the learned guess (255^2 problems, batch 16)
        {"name": "train-255", "kind": "train", "n": 255, "batch": 16},
        # one full-resolution initial guess
        {"name": "guess-1023", "kind": "guess", "n": 1023},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("sweep", "sweep", "sweep", "solve", "solve", "batched", "sweep3d", "train", "guess"))
    if kind == "sweep":
        fma = rng.randint(0, 1)
        n = _log(rng, 48, 16000)
        return {"kind": kind, "n": n, "fma": fma,
                "sweeps": max(1, min(_log(rng, 20, 400), int((0.5 + 0.5 * fma) * MAX_LUP) // n ** 2))}
    if kind == "solve":
        n = _log(rng, 48, 8192)
        check = rng.choice((50, 100, 200))
        sweeps = check * rng.randint(2, 8)
        return {"kind": kind, "n": n, "sweeps": min(sweeps, check * max(1, MAX_LUP // 4 // n ** 2 // check)),
                "check": check, "refine": rng.randint(0, 1)}
    if kind == "batched":
        return {"kind": kind, "count": _log(rng, 16, 400), "n": _log(rng, 63, 300), "sweeps": 100 * rng.randint(1, 5),
                "refine": rng.randint(0, 1)}
    if kind == "sweep3d":
        return {"kind": kind, "n": _log(rng, 24, 500), "sweeps": rng.randint(10, 20)}
    if kind == "train":
        return {"kind": kind, "n": rng.randint(60, 255), "batch": rng.randint(2, 16)}
    return {"kind": kind, "n": _log(rng, 120, 1500)}


# ------------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(shape, g):
    return torch.rand(shape, generator=g, dtype=torch.float64, device=DEV) * 2.0 - 1.0


def _field(n, g):
    """A smooth random field with power spectrum |k|^-3 and unit RMS."""
    z = torch.randn((n, n), generator=g, dtype=torch.float64, device=DEV)
    k = torch.fft.fftfreq(n, device=DEV).to(torch.float64)[:, None] * n
    l = torch.fft.rfftfreq(n, device=DEV).to(torch.float64)[None, :] * n
    k2 = k * k + l * l
    k2[0, 0] = 1.0
    a = torch.fft.rfft2(z) * k2 ** -0.75
    a[0, 0] = 0.0
    f = torch.fft.irfft2(a, s=(n, n))
    return (f / f.square().mean().sqrt()).contiguous()


def _h2(n):
    h = 1.0 / (n + 1)
    return h * h


def _coords(n):
    return torch.arange(n + 2, dtype=torch.float64, device=DEV) / (n + 1)


def _ring(n, values):
    """(n+2)^2 grid: `values` on the ring, zero inside (the usual start)."""
    u = torch.zeros((n + 2, n + 2), dtype=torch.float64, device=DEV)
    u[0], u[-1], u[:, 0], u[:, -1] = values[0], values[-1], values[:, 0], values[:, -1]
    return u


def _quadratic_ring(n, g):
    a = float(_uniform((1,), g))
    x = _coords(n)
    return _ring(n, (1.0 + 0.25 * a) * (x[:, None] ** 2 - x[None, :] ** 2))


def _linear_ring(n, g):
    a, b, c = _uniform((3,), g).tolist()
    x = _coords(n)
    return _ring(n, a + b * x[:, None] + c * x[None, :])


def _poisson_correction(f):
    """The solution of the 5-point problem for f with a zero ring, by sine transforms: what a
    training set holds as converged solutions, less the boundary interpolation."""
    n = f.shape[-1]
    m = 2 * (n + 1)

    def dst(a):  # sine sum over the last axis
        e = torch.zeros(a.shape[:-1] + (m,), dtype=torch.float64, device=DEV)
        e[..., 1:n + 1] = a
        e[..., n + 2:] = -a.flip(-1)
        return -0.5 * torch.fft.rfft(e).imag[..., 1:n + 1]

    h = 1.0 / (n + 1)
    lam = (2.0 - 2.0 * torch.cos(torch.arange(1, n + 1, dtype=torch.float64, device=DEV) * math.pi * h)) / (h * h)
    t = dst(dst(f).transpose(-1, -2)) / (lam[:, None] + lam[None, :])
    return dst(dst(t).transpose(-1, -2)) * (2.0 * h) ** 2


def _sizes(case):
    """Problem sizes of a batch: three uneven sizes in turn."""
    n = case["n"]
    return [max(1, (n + 1) // (1 << (p % 3)) - 1) for p in range(case["count"])]


def prepare(case, seed):
    g = _gen(seed)
    kind, n = case["kind"], case["n"]
    st = {"case": case}
    if kind in ("sweep", "solve"):
        refine = kind == "solve" and case["refine"]
        st["f"] = _field(n, g) if refine else _uniform((n, n), g)
        st["u0"] = _quadratic_ring(n, g)
        st["out"] = torch.empty_like(st["u0"])
        if kind == "sweep":
            kw = {"fma": case["fma"]}
        else:
            kw = {"check_every": case["check"], "inner_sweeps": case["check"], "max_sweeps": case["sweeps"],
                  "precision": rb.RBGS_FP32_REFINE if refine else rb.RBGS_FP64}
        st["solver"] = rb.Solver(n, _h2(n), st["f"], st["u0"], **kw)
    elif kind == "batched":
        sizes = _sizes(case)
        st["probs"] = []
        for m in sizes:
            c = float(_uniform((1,), g))
            u = _ring(m, torch.full((m + 2, m + 2), c, dtype=torch.float64, device=DEV))
            st["probs"].append((m, _h2(m), _uniform((m, m), g), u))
        st["out"] = torch.empty(sum((m + 2) ** 2 for m in sizes), dtype=torch.float64, device=DEV)
        st["views"] = [v.view(m + 2, m + 2) for v, m in zip(st["out"].split([(m + 2) ** 2 for m in sizes]), sizes)]
        st["opts"] = rb.default_opts(precision=rb.RBGS_FP32_REFINE if case["refine"] else rb.RBGS_FP64, check_every=100,
                                     inner_sweeps=100, max_sweeps=case["sweeps"])
    elif kind == "sweep3d":
        st["f"] = _uniform((n, n, n), g)
        u = torch.zeros((n + 2, n + 2, n + 2), dtype=torch.float64, device=DEV)
        x = _coords(n)
        u[0], u[-1] = x[:, None] * x[None, :], 1.0 - x[:, None] * x[None, :]
        st["u0"] = u
        st["out"] = torch.empty_like(u)
    else:
        st["net"] = ru.UNet(seed=int(seed) & 0xFFFF)
        size = (n + 2 + 7) // 8 * 8
        if kind == "guess":
            st["f"], st["ring"], st["size"] = _field(n, g), _linear_ring(n, g), size
        else:
            xs, ts = [], []
            for _ in range(case["batch"]):
                f, ring = _field(n, g), _linear_ring(n, g)
                sol = ru.boundary_blend(ring)
                sol[1:-1, 1:-1] += _poisson_correction(f)
                xs.append(ru.network_input(f, ring, size))
                ts.append(ru.guess_target(sol, ring, size))
            st["x"], st["t"] = torch.stack(xs), torch.stack(ts)
            m = torch.zeros((case["batch"], size, size), dtype=torch.float32, device=DEV)
            m[:, 1:n + 1, 1:n + 1] = 1.0
            st["mask"] = m
            st["grads"] = torch.empty(st["net"].num_params, dtype=torch.float32, device=DEV)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------------- run

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        s = state["solver"]
        s.set_problem(state["f"], state["u0"])
        s.sweep(case["sweeps"])
        rho = s.residual()
        s.get_solution(state["out"])
        return {"u": state["out"], "rho": rho}
    if kind == "solve":
        s = state["solver"]
        s.set_problem(state["f"], state["u0"])
        done, rho, _ = s.solve(0.0, allow_not_converged=True)
        s.get_solution(state["out"])
        return {"u": state["out"], "rho": rho, "sweeps": done}
    if kind == "batched":
        res = rb.rbgs_solve_batched(state["probs"], 0.0, state["views"], state["opts"], allow_failures=True)
        return {"u": state["out"], "rho": np.array([r["rel"] for r in res]),
                "sweeps": np.array([r["sweeps"] for r in res], dtype=np.int64)}
    if kind == "sweep3d":
        n = case["n"]
        with rb.Solver3D(n, _h2(n), state["f"], state["u0"]) as s:
            s.sweep(case["sweeps"])
            rho = s.residual()
            s.get_solution(state["out"])
        return {"u": state["out"], "rho": rho}
    if kind == "train":
        loss = state["net"].train_step(state["x"], state["t"], state["mask"], grads=state["grads"])
        return {"grads": state["grads"], "loss": loss}
    x = ru.network_input(state["f"], state["ring"], state["size"]).unsqueeze(0)
    pred = state["net"].forward(x)
    return {"u0": ru.guess_assemble(state["ring"], pred[0]), "pred": pred}


def _net_shapes(case):
    size = (case["n"] + 2 + 7) // 8 * 8
    return case.get("batch", 1), size


_LAYERS = (  # (inputs, outputs, kernel, level) of the network's convolutions, in order
    (16, 32, 3, 0), (32, 32, 3, 0), (32, 64, 3, 1), (64, 64, 3, 1), (64, 128, 3, 2), (128, 128, 3, 2),
    (128, 256, 3, 3), (256, 256, 3, 3), (384, 128, 3, 2), (128, 128, 3, 2), (192, 64, 3, 1), (64, 64, 3, 1),
    (96, 32, 3, 0), (32, 32, 3, 0), (32, 8, 1, 0))


def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("sweep", "solve"):  # f and u read, u written; 7 operations per update
        return {"bytes": 24.0 * n * n, "flops": 7.0 * n * n * case["sweeps"]}
    if kind == "batched":
        points = sum(m * m for m in _sizes(case))
        return {"bytes": 24.0 * points, "flops": 7.0 * points * case["sweeps"]}
    if kind == "sweep3d":
        return {"bytes": 24.0 * n ** 3, "flops": 9.0 * n ** 3 * case["sweeps"]}
    batch, size = _net_shapes(case)
    flops = params = 0.0
    for cin, cout, k, level in _LAYERS:
        params += k * k * cin * cout + cout
        flops += 2.0 * batch * (size >> level) ** 2 * k * k * (4 if cin == 16 else cin) * (1 if cout == 8 else cout)
    pixels = batch * size * size
    if kind == "train":
        return {"bytes": 4.0 * (6 * pixels + 2 * params), "flops": 3.0 * flops}
    return {"bytes": 8.0 * 2 * n * n + 4.0 * (5 * pixels + params), "flops": flops}


# -------------------------------------------------------------------------------- exact

def _sweeps2(u, f, h2, sweeps):
    """Red-black sweeps of a batch of equal grids in 64 bits: u (.., n+2, n+2), f (.., n, n)."""
    n = f.shape[-1]
    i = torch.arange(n, device=u.device)
    red = ((i[:, None] + i[None, :]) & 1) == 0  # interior points with even i + j
    hf = f * h2
    for _ in range(sweeps):
        for mask in (red, ~red):
            s = hf + u[..., :-2, 1:-1]
            s += u[..., 2:, 1:-1]
            s += u[..., 1:-1, :-2]
            s += u[..., 1:-1, 2:]
            s *= 0.25
            inner = u[..., 1:-1, 1:-1]
            torch.where(mask, s, inner, out=s)
            inner.copy_(s)
    return u


def _rho2(u, f, h2):
    hf = f * h2
    r = hf + u[..., :-2, 1:-1] + u[..., 2:, 1:-1] + u[..., 1:-1, :-2] + u[..., 1:-1, 2:] - 4.0 * u[..., 1:-1, 1:-1]
    b = hf
    b[..., 0, :] += u[..., 0, 1:-1]
    b[..., -1, :] += u[..., -1, 1:-1]
    b[..., :, 0] += u[..., 1:-1, 0]
    b[..., :, -1] += u[..., 1:-1, -1]
    return r.square().sum((-1, -2)).sqrt() / b.square().sum((-1, -2)).sqrt()


def _sweeps3(u, f, h2, sweeps):
    n = f.shape[-1]
    i = torch.arange(n, device=u.device)
    # interior index 0 is grid index 1, so the parity of i + j + k is that of the indices' sum + 1
    red = ((i[:, None, None] + i[None, :, None] + i[None, None, :]) & 1) == 1
    hf = f * h2
    six = torch.full((1,), 6.0, dtype=torch.float64, device=u.device)  # a true division, not a product by 1/6
    c = slice(1, -1)
    for _ in range(sweeps):
        for mask in (red, ~red):
            s = hf + u[:-2, c, c]
            s += u[2:, c, c]
            s += u[c, :-2, c]
            s += u[c, 2:, c]
            s += u[c, c, :-2]
            s += u[c, c, 2:]
            s /= six
            inner = u[c, c, c]
            torch.where(mask, s, inner, out=s)
            inner.copy_(s)
    return u


def _rho3(u, f, h2):
    c = slice(1, -1)
    hf = f * h2
    r = hf + u[:-2, c, c] + u[2:, c, c] + u[c, :-2, c] + u[c, 2:, c] + u[c, c, :-2] + u[c, c, 2:] - 6.0 * u[c, c, c]
    b = hf
    for axis in range(3):
        for side in (0, -1):
            b.select(axis, side).add_(u.select(axis, side)[c, c])
    return float(r.square().sum().sqrt() / b.square().sum().sqrt())


def _conv64(x, w, b, k):
    """NHWC convolution in 64 bits, one product per tap."""
    if k == 1:
        return x @ w[:, 0, 0, :].T + b
    h, wd = x.shape[1], x.shape[2]
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    y = None
    for dy in range(3):
        for dx in range(3):
            t = p[:, dy:dy + h, dx:dx + wd, :] @ w[:, dy, dx, :].T
            y = t if y is None else y + t
    return y + b


def _net64(params, x):
    """The network in 64 bits: x (B, H, W, 4) -> (B, H, W)."""
    ws, at = [], 0
    for cin, cout, k, _ in _LAYERS:
        w = params[at:at + cout * k * k * cin].view(cout, k, k, cin)
        at += cout * k * k * cin
        ws.append((w, params[at:at + cout], k))
        at += cout
    x = torch.nn.functional.pad(x, (0, 12))

    def conv(i, v):
        return torch.relu(_conv64(v, *ws[i]))

    def pool(v):
        b, h, w, c = v.shape
        return v.view(b, h // 2, 2, w // 2, 2, c).mean((2, 4))

    def up(v, skip):
        return torch.cat([v.repeat_interleave(2, 1).repeat_interleave(2, 2), skip], -1)

    s0 = conv(1, conv(0, x))
    s1 = conv(3, conv(2, pool(s0)))
    s2 = conv(5, conv(4, pool(s1)))
    v = conv(7, conv(6, pool(s2)))
    v = conv(9, conv(8, up(v, s2)))
    v = conv(11, conv(10, up(v, s1)))
    v = conv(13, conv(12, up(v, s0)))
    return _conv64(v, *ws[14])[..., 0]


def exact(case, seed):
    st = prepare(case, seed)
    kind, n = case["kind"], case["n"]
    h2 = _h2(n)
    if kind in ("sweep", "solve"):
        st.pop("solver").close()
        u = _sweeps2(st["u0"].clone(), st["f"], h2, case["sweeps"])
        out = {"u": u, "rho": float(_rho2(u, st["f"], h2))}
        if kind == "solve":
            out["sweeps"] = case["sweeps"]
        return out
    if kind == "batched":
        rho = np.zeros(len(st["probs"]))
        for m in sorted({p[0] for p in st["probs"]}):
            at = [q for q, p in enumerate(st["probs"]) if p[0] == m]
            f = torch.stack([st["probs"][q][2] for q in at])
            u = _sweeps2(torch.stack([st["probs"][q][3] for q in at]), f, _h2(m), case["sweeps"])
            for q, v, r in zip(at, u, _rho2(u, f, _h2(m)).tolist()):
                st["views"][q].copy_(v)
                rho[q] = r
        return {"u": st["out"], "rho": rho, "sweeps": np.full(len(rho), case["sweeps"], dtype=np.int64)}
    if kind == "sweep3d":
        u = _sweeps3(st["u0"].clone(), st["f"], h2, case["sweeps"])
        return {"u": u, "rho": _rho3(u, st["f"], h2)}
    params = st["net"].get_params().double()
    if kind == "train":
        # sample by sample: 64-bit activations of a whole batch would be kept for the backward
        grads, loss = torch.zeros_like(params), 0.0
        count = st["mask"].double().sum()
        for x, t, m in zip(st["x"].double(), st["t"].double(), st["mask"].double()):
            p = params.clone().requires_grad_(True)
            part = (m * (_net64(p, x[None])[0] - t) ** 2).sum() / count
            grads += torch.autograd.grad(part, p)[0]
            loss += float(part)
        return {"grads": grads, "loss": loss}
    size = st["size"]
    x, y = torch.zeros((1, size, size, 4), dtype=torch.float64, device=DEV), _coords(n)
    ring = st["ring"]
    a, b = y[:, None], y[None, :]
    corners = ((1 - a) * (1 - b) * ring[0, 0] + (1 - a) * b * ring[0, -1] + a * (1 - b) * ring[-1, 0]
               + a * b * ring[-1, -1])
    blend = (1 - a) * ring[0] + a * ring[-1] + (1 - b) * ring[:, :1] + b * ring[:, -1:] - corners
    one = torch.ones((n + 2, n + 2), dtype=torch.float64, device=DEV)
    x[0, 1:n + 1, 1:n + 1, 0] = st["f"]
    x[0, :n + 2, :n + 2, 1] = _ring(n, one)
    x[0, :n + 2, :n + 2, 2] = ring
    x[0, :n + 2, :n + 2, 3] = blend
    with torch.no_grad():
        pred = _net64(params, x)
    u0 = ring.clone()
    u0[1:-1, 1:-1] = blend[1:-1, 1:-1] + pred[0, 1:n + 1, 1:n + 1]
    return {"u0": u0, "pred": pred}
