"""What is measured: the calls that a program using this package makes, over the sizes it makes them at.

The pressure solve takes nine tenths of a step, so most cases are solves on their own (on device buffers, in each
precision, from the smallest test grid to the largest configuration); the U-Net of the learned warm start is there
forward and in training; four cases are whole steps, one of them a batch of uneven grids.  Grids, bodies and
tolerances are those of ``workloads.py`` (the paper's domain, a uniform block of 30 % of the columns round the body,
geometric stretching outside), the odd sizes are generic.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2402_17337_gb300 as ibm
from paper_2402_17337_gb300 import warmstart
from paper_2402_17337_gb300 import workloads as W

DOMAIN = W.PAPER_DOMAIN
UBOX = W.UBOX
# relaxation factors that Solver.tune_omega finds on the two large grids (a program keeps the value; the probe itself
# takes seconds); elsewhere the package's default
OMEGA = {(2048, 1024): 1.99787, (4096, 2048): 1.99893}
# Tolerance of the standalone solves over the largest right-hand side.  A step leaves 1e-10 of its initial residual; the
# FP32 sweeps and the multigrid variant stop at points that depend on the tile shape chosen, so they take a smaller one
# to fix the solution to as many digits.
RTOL = {0: 1e-10, 1: 1e-11, 2: 1e-11}


def listed():
    return [
        # the smallest parity grid, uniform, in FP64: a call whose time is launches and waits
        {"name": "poisson_fp64_70x45", "kind": "poisson", "precision": 0, "nx": 70, "ny": 45, "stretched": False},
        # the paper's own method (FP64 red-black SOR) on the batch's smallest stretched grid
        {"name": "poisson_fp64_512x256", "kind": "poisson", "precision": 0, "nx": 512, "ny": 256, "stretched": True},
        # odd sizes, FP32 sweeps in FP64 defect correction, every tile edge ragged
        {"name": "poisson_mixed_777x391", "kind": "poisson", "precision": 1, "nx": 777, "ny": 391, "stretched": True},
        # the benchmark's grid
        {"name": "poisson_mixed_2048x1024", "kind": "poisson", "precision": 1, "nx": 2048, "ny": 1024,
         "stretched": True},
        # the largest configuration
        {"name": "poisson_mixed_4096x2048", "kind": "poisson", "precision": 1, "nx": 4096, "ny": 2048,
         "stretched": True},
        # the multigrid variant on the benchmark's grid
        {"name": "poisson_mg_2048x1024", "kind": "poisson", "precision": 2, "nx": 2048, "ny": 1024,
         "stretched": True},
        # the solve for callers that cannot allocate, at its test's odd size
        {"name": "poisson_noalloc_133x67", "kind": "noalloc", "nx": 133, "ny": 67},
        # the warm start's inference on the benchmark's coarse grid
        {"name": "unet_forward_512x1024", "kind": "unet_forward", "H": 512, "W": 1024, "widths": "16,32,32,48"},
        # one training step of the larger network on its configuration's coarse grid
        {"name": "unet_train_256x512", "kind": "unet_train", "H": 256, "W": 512, "widths": "32,64,128,128"},
        # a step of the smallest configuration, FP64 (the validation path)
        {"name": "step_fp64_192x128", "kind": "step", "precision": 0, "nx": 192, "ny": 128, "stretched": False,
         "learned": False},
        # a step of the benchmark: FP32 sweeps in FP64 defect correction, learned warm start
        {"name": "step_learned_2048x1024", "kind": "step", "precision": 1, "nx": 2048, "ny": 1024, "stretched": True,
         "learned": True},
        # cases with uneven grids advancing together (the 64-case batch's recipe; eight, so that a state is made quickly)
        {"name": "batch_8", "kind": "batch", "n": 8, "lo": 512, "hi": 1536},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["poisson", "poisson", "poisson", "poisson", "noalloc", "unet_forward", "unet_train", "step",
                       "step", "batch"])
    if kind == "poisson":
        precision = rng.choice([0, 1, 1, 2])
        nx = _log(rng, *{0: (64, 512), 1: (96, 4000), 2: (128, 2048)}[precision])
        stretched = nx >= 96 and rng.random() < 0.8
        return {"kind": kind, "precision": precision, "nx": nx, "ny": nx // 2 + rng.randrange(-nx // 20, nx // 20 + 1),
                "stretched": stretched}
    if kind == "noalloc":
        nx = _log(rng, 96, 384)
        return {"kind": kind, "nx": nx, "ny": nx // 2 + rng.randrange(-nx // 20, nx // 20 + 1)}
    if kind in ("unet_forward", "unet_train"):
        H = 8 * _log(rng, 4, 64 if kind == "unet_forward" else 32)
        return {"kind": kind, "H": H, "W": 8 * _log(rng, H // 8, H // 4),
                "widths": rng.choice(["16,16,32,32", "16,32,32,48", "32,64,128,128"])}
    if kind == "step":
        precision = rng.choice([0, 1, 1, 2])
        nx = _log(rng, 112, 384 if precision == 0 else 1536)
        return {"kind": kind, "precision": precision, "nx": nx, "ny": nx // 2 + rng.randrange(0, nx // 20 + 1),
                "stretched": True, "learned": False}
    return {"kind": kind, "n": rng.randrange(2, 7), "lo": 64 * _log(rng, 2, 4), "hi": 64 * _log(rng, 6, 16)}


# ---------------------------------------------------------------- grids and right-hand sides


def _domain(case):
    """Domain and spacing of a case's grid (hmin 0: uniform)."""
    if case["kind"] != "noalloc" and not case["stretched"]:
        return (-2.0, 5.0, -2.25, 2.25) if case["kind"] == "poisson" else (-4.0, 8.0, -4.0, 4.0), 0.0
    return DOMAIN, 10.0 / case["nx"]


def _axis(a0, a1, b0, b1, n, hmin):
    """Faces of one axis (Sec. 2.3 of the paper): a uniform block from b0, geometric progressions on both sides."""
    if hmin <= 0.0:
        return a0 + (a1 - a0) / n * np.arange(n + 1)
    nb = round((b1 - b0) / hmin)
    end = b0 + nb * hmin
    left, right = b0 - a0, a1 - end
    nl = math.floor((n - nb) * (left / (left + right)) + 0.5)

    def side(length, m):
        lo, hi = 1.0, 2.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if mid in (lo, hi):
                break
            lo, hi = (mid, hi) if hmin * np.sum(mid ** np.arange(1, m + 1)) < length else (lo, mid)
        return hmin * np.cumsum((0.5 * (lo + hi)) ** np.arange(1, m + 1))

    f = np.concatenate([(b0 - side(left, nl))[::-1], b0 + hmin * np.arange(nb + 1), end + side(right, n - nb - nl)])
    f[0], f[-1] = a0, a1
    return f


def _faces(case):
    d, hmin = _domain(case)
    return (_axis(d[0], d[1], UBOX[0], UBOX[1], case["nx"], hmin),
            _axis(d[2], d[3], UBOX[2], UBOX[3], case["ny"], hmin))


def _rhs(case, seed):
    """A right-hand side of the kind a step makes, on the GPU: jumps from cell to cell where the body has moved, a
    smooth source round it that is weaker, next to nothing in the far field; no net source."""
    xf, yf = _faces(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.tensor(0.5 * (xf[1:] + xf[:-1]), device="cuda")
    y = torch.tensor(0.5 * (yf[1:] + yf[:-1]), device="cuda")
    vol = torch.outer(torch.tensor(np.diff(yf), device="cuda"), torch.tensor(np.diff(xf), device="cuda"))
    r = torch.rand(10, 4, generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    b = 1e-3 * torch.randn(len(y), len(x), generator=g, device="cuda", dtype=torch.float64)
    b *= torch.outer(torch.exp(-(y / 2.0) ** 2), torch.exp(-((x - 1.0) / 3.0) ** 2))
    for cx, cy, s, a in r:
        w = 0.1 + 0.4 * s
        b += (2.0 * a - 1.0) * torch.outer(torch.exp(-((y - (cy - 0.5)) / w) ** 2),
                                           torch.exp(-((x - (2.0 * cx - 0.75)) / w) ** 2))
    spots = torch.randn(len(y), len(x), generator=g, device="cuda", dtype=torch.float64)
    b += 10.0 * spots * torch.outer((torch.abs(y - 0.2 * float(r[0, 0])) < 0.08).double(),
                                    (torch.abs(x) < 0.5).double())
    b *= 1e3
    b -= (b * vol).sum() / vol.sum()
    return b.contiguous()


# ---------------------------------------------------------------- prepare


def _config(case, seed):
    """Flow parameters of a step: the configurations' recipe with the body's motion drawn from the seed."""
    rng = np.random.default_rng([seed, case["nx"]])
    d, hmin = _domain(case)
    dt = W.DT_PER_HMIN * hmin if hmin > 0.0 else 2e-3
    # where a solve stops depends on the tile shape; these leave the fields fixed to ten digits whichever is chosen
    div = 1e-10 if hmin <= 0.0 else 1e-11 if case["nx"] < 512 else 1e-10 if case["nx"] < 1536 else 1e-9
    return W.FlowConfig("case", *d, case["nx"], case["ny"], hmin, Re=float(rng.uniform(300.0, 1000.0)), dt=dt, steps=0,
                        h=float(rng.uniform(0.15, 0.35)), k=float(rng.uniform(1.5, 2.5)), div_tol=div,
                        omega_p=OMEGA.get((case["nx"], case["ny"])), init="uniform" if hmin > 0.0 else "rest")


def _solver(cfg, precision, seed, steps):
    """A running simulation: a few steps into the plunge, a vortex behind the body."""
    rng = np.random.default_rng([seed, 1])
    s = ibm.Solver.from_config(cfg, precision=precision)
    xf, yf = s.grid()
    xc = 0.5 * (xf[1:] + xf[:-1])
    cx, cy, amp = rng.uniform(1.2, 1.8), rng.uniform(-0.3, 0.3), rng.uniform(0.1, 0.2)
    s.set("u", cfg.initial_u(s.shape("u")))
    s.set("v", amp * np.outer(np.exp(-(yf - cy) ** 2 / 0.1), np.exp(-(xc - cx) ** 2 / 0.1)))
    s.step(steps)
    return s


def _pinned(s):
    return {n: torch.empty(s.shape(n), dtype=torch.float64, pin_memory=True).numpy() for n in ("u", "v", "p")}


def _params(widths, seed):
    """He-normal weights, small biases, in the parameter order of the network."""
    rng = np.random.default_rng([seed, 7])
    out = []
    for cin, cout, _ in _layers(widths):
        out.append(rng.standard_normal(cout * 9 * cin) * math.sqrt(2.0 / (9 * cin)))
        out.append(0.05 * rng.standard_normal(cout))
    return np.concatenate(out).astype(np.float32)


def _features(case, seed):
    """Four coarse fields over their largest value (two of them rough near the middle, one a body mask, one smooth) and
    a target of order one."""
    H, Wd = case["H"], case["W"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    y = torch.linspace(-1, 1, H, device="cuda")[:, None]
    x = torch.linspace(-1, 1, Wd, device="cuda")[None, :]
    c = torch.rand(6, 2, generator=g, device="cuda").cpu().numpy() - 0.5
    near = torch.exp(-((x - float(c[0, 0])) ** 2 + (y - float(c[0, 1])) ** 2) / 0.05)
    smooth = sum(torch.sin(3 * (k + 1) * x + 9 * float(c[k, 0])) * torch.cos(2 * (k + 1) * y + 9 * float(c[k, 1]))
                 for k in range(6))
    f = torch.stack([near * torch.randn(H, Wd, generator=g, device="cuda"),
                     near * torch.randn(H, Wd, generator=g, device="cuda") + 0.1 * smooth,
                     (near > 0.7).float(), smooth], dim=2)
    f = f / f.abs().amax(dim=(0, 1), keepdim=True).clamp_min(1e-20)
    t = 0.5 * smooth + near * torch.randn(H, Wd, generator=g, device="cuda")
    return f.contiguous(), (t / t.square().mean().sqrt()).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("poisson", "noalloc"):
        st["b"] = _rhs(case, seed)
        st["phi"] = torch.zeros_like(st["b"])
        bmax = float(st["b"].abs().max())
        if kind == "poisson":
            d, hmin = _domain(case)
            st["stream"] = torch.cuda.Stream()
            st["tol"] = RTOL[case["precision"]] * bmax
            st["solver"] = ibm.Solver(x0=d[0], x1=d[1], y0=d[2], y1=d[3], nx=case["nx"], ny=case["ny"], hmin=hmin,
                                      ubox=UBOX, precision=case["precision"], stream=st["stream"].cuda_stream,
                                      omega_p=OMEGA.get((case["nx"], case["ny"])))
            if case["precision"] == 1:
                st["solver"].tune()  # a program's first solve does it once
        else:
            xf, yf = _faces(case)
            st["faces"] = xf, yf
            st["args"] = case["nx"], case["ny"], ibm.default_omega(case["nx"], case["ny"]), RTOL[0] * bmax
    elif kind in ("unet_forward", "unet_train"):
        widths = tuple(int(w) for w in case["widths"].split(","))
        st["net"] = ibm.UNet(widths, 0)
        st["net"].set_params(_params(widths, seed))
        st["feat"], st["target"] = _features(case, seed)
        st["out"] = torch.empty(case["H"], case["W"], device="cuda")
    elif kind == "step":
        cfg = _config(case, seed)
        s = st["solver"] = _solver(cfg, case["precision"], seed, 2)
        if case["learned"]:
            net, scale, _ = warmstart.load(warmstart.weights_for(f"plunge_{case['nx']}x{case['ny']}"))
            s.set_warmstart(1, net, scale)
        st["host"] = _pinned(s)
    else:
        rng = np.random.default_rng([case["n"], case["lo"], case["hi"]])  # the sizes are the case's, the flows the seed's
        st["solvers"] = []
        for c in range(case["n"]):
            nx = int(rng.choice(np.arange(case["lo"], case["hi"] + 1, 64)))
            sub = {"kind": "step", "nx": nx, "ny": nx // 2, "stretched": True}
            st["solvers"].append(_solver(_config(sub, seed + 1000 * c), 1, seed + 1000 * c, 1))
        st["batch"] = ibm.Batch(st["solvers"])
        st["batch"].step(1)
        st["host"] = [_pinned(s) for s in st["solvers"]]
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- run


def _noalloc(st):
    fn = ibm.lib().ibm_poisson_solve_noalloc
    dp = ctypes.POINTER(ctypes.c_double)
    fn.argtypes = [ctypes.c_int, ctypes.c_int, dp, dp, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double,
                   ctypes.c_double, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.POINTER(ctypes.c_int), dp]
    fn.restype = ctypes.c_int
    nx, ny, omega, tol = st["args"]
    sweeps, res = ctypes.c_int(0), ctypes.c_double(0.0)
    rc = fn(nx, ny, st["faces"][0].ctypes.data_as(dp), st["faces"][1].ctypes.data_as(dp), st["b"].data_ptr(),
            st["phi"].data_ptr(), omega, tol, 8, 0, torch.cuda.current_stream().cuda_stream, ctypes.byref(sweeps),
            ctypes.byref(res))
    if rc:
        raise ibm.IbmError(rc, ibm.lib().ibm_last_error().decode())
    return sweeps.value


def run(state):
    kind = state["kind"]
    if kind == "poisson":
        s = state["solver"]
        with torch.cuda.stream(state["stream"]):
            state["phi"].zero_()
            rc, sweeps, _ = s.poisson_solve(state["b"].data_ptr(), state["phi"].data_ptr(), state["tol"])
        if rc:
            raise ibm.IbmError(rc, ibm.lib().ibm_last_error().decode())
        # the FP64 path's sweep count is fixed by its arithmetic; the others' depend on the tile shape chosen
        return {"phi": state["phi"], "sweeps": sweeps} if s.P.precision == 0 else {"phi": state["phi"]}
    if kind == "noalloc":
        state["phi"].zero_()
        sweeps = _noalloc(state)
        return {"phi": state["phi"], "sweeps": sweeps}
    if kind in ("unet_forward", "unet_train"):
        H, Wd = state["out"].shape
        stream = torch.cuda.current_stream().cuda_stream
        if kind == "unet_forward":
            state["net"].forward(state["feat"].data_ptr(), H, Wd, state["out"].data_ptr(), stream)
            return state["out"]
        loss = state["net"].train_step(state["feat"].data_ptr(), state["target"].data_ptr(), H, Wd, lr=1e-5,
                                       stream=stream)
        return {"loss": loss, "grads": state["net"].grads()}
    if kind == "step":
        st = state["solver"].step(1)
        out = {n: state["solver"].get(n, out=a) for n, a in state["host"].items()}
        return {**out, "cl": st["cl"], "cd": st["cd"]}
    stats = state["batch"].step(1)
    return [{**{n: s.get(n, out=a) for n, a in h.items()}, "cl": st["cl"], "cd": st["cd"]}
            for s, h, st in zip(state["solvers"], state["host"], stats)]


# ---------------------------------------------------------------- work


def work(case):
    kind = case["kind"]
    if kind in ("unet_forward", "unet_train"):
        widths = tuple(int(w) for w in case["widths"].split(","))
        px = case["H"] * case["W"]
        level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
        macs = sum(9 * (4 if k == 0 else cin) * (1 if k == 14 else cout) * (px >> (2 * level[k]))
                   for k, (cin, cout, _) in enumerate(_layers(widths)))
        n = sum(cout * (9 * cin + 1) for cin, cout, _ in _layers(widths))
        if kind == "unet_forward":
            return {"bytes": 4 * (5 * px + n), "flops": 2 * macs}
        return {"bytes": 4 * (5 * px + 8 * n), "flops": 6 * macs}  # weights, both moments read and written, gradient
    if kind in ("poisson", "noalloc"):
        cells = case["nx"] * case["ny"]
        return {"bytes": 16 * cells, "flops": 9 * cells}  # b in, phi out; one application of the operator
    if kind == "step":
        cells = case["nx"] * case["ny"]
    else:
        rng = np.random.default_rng([case["n"], case["lo"], case["hi"]])
        cells = sum(int(rng.choice(np.arange(case["lo"], case["hi"] + 1, 64))) ** 2 // 2 for _ in range(case["n"]))
    # u, v, p, the last increment and two convection histories in and out, and u, v, p to the host
    return {"bytes": 8 * (12 + 3) * cells, "flops": 150 * cells}


# ---------------------------------------------------------------- exact


def _exact_poisson(case, seed):
    """The discrete equation solved directly in 64 bits: both axes diagonalised (the operator is a sum of an x and a y
    part, each self-adjoint in its cell widths), then refined with the five-point residual."""
    xf, yf = (torch.tensor(f, device="cuda") for f in _faces(case))
    b = _rhs(case, seed)

    def axis(f):
        d = f.diff()
        a = 1.0 / (0.5 * (f[1:] + f[:-1])).diff()  # reciprocal centre spacings
        up = torch.cat([a, a.new_zeros(1)]) / d
        dn = torch.cat([a.new_zeros(1), a]) / d
        s = torch.sqrt(d)
        off = a / (s[1:] * s[:-1])
        lam, q = torch.linalg.eigh(torch.diag(-(up + dn)) + torch.diag(off, 1) + torch.diag(off, -1))
        return up, dn, s, lam, q

    ux, dx, sx, lx, qx = axis(xf)
    uy, dy, sy, ly, qy = axis(yf)
    den = ly[:, None] + lx[None, :]
    den[-1, -1] = math.inf  # the constant: the last eigenvalue of each axis is zero

    def solve(r):
        return (qy @ ((qy.T @ (r * sy[:, None] * sx) @ qx) / den) @ qx.T) / (sy[:, None] * sx)

    def lap(p):
        gx, gy = p.diff(dim=1), p.diff(dim=0)
        r = torch.zeros_like(p)
        r[:, :-1] += ux[:-1] * gx
        r[:, 1:] -= dx[1:] * gx
        r[:-1] += uy[:-1, None] * gy
        r[1:] -= dy[1:, None] * gy
        return r

    phi = solve(b)
    for _ in range(3):
        phi = phi + solve(b - lap(phi))
    return phi - phi[0, -1]


def _layers(w):
    """(input channels, output channels, level) of the network's fifteen convolutions, in parameter order."""
    out = [(16, w[0], 0), (w[0], w[0], 0)]
    for l in (1, 2, 3):
        out += [(w[l - 1], w[l], l), (w[l], w[l], l)]
    for l in (2, 1, 0):
        out += [(w[l + 1] + w[l], w[l], l), (w[l], w[l], l)]
    return out + [(w[0], 16, 0)]


def _exact_unet(case, seed, grads):
    """The network in 64 bits from torch's own convolutions, and the gradient of its mean squared error."""
    widths = tuple(int(w) for w in case["widths"].split(","))
    flat = torch.tensor(_params(widths, seed), device="cuda", dtype=torch.float64).requires_grad_(grads)
    feat, target = _features(case, seed)
    F = torch.nn.functional
    ws, off = [], 0
    for cin, cout, _ in _layers(widths):
        w = flat[off:off + cout * 9 * cin].view(cout, 3, 3, cin).permute(0, 3, 1, 2)
        off += cout * 9 * cin
        ws.append((w, flat[off:off + cout]))
        off += cout

    def conv(k, x):
        w, c = ws[k]
        H, Wd = x.shape[2:]
        xp, y = F.pad(x, (1, 1, 1, 1)), 0.0
        for t in range(9):  # one matrix product a tap: in 64 bits faster than the library's convolution
            y = y + torch.einsum("oi,bihw->bohw", w[:, :, t // 3, t % 3], xp[:, :, t // 3:t // 3 + H, t % 3:t % 3 + Wd])
        return y + c[None, :, None, None]

    x = F.pad(feat.double().permute(2, 0, 1)[None], (0, 0, 0, 0, 0, 12))
    enc, h = [], x
    for l in range(4):
        if l:
            h = F.avg_pool2d(h, 2)
        h = torch.relu(conv(2 * l + 1, torch.relu(conv(2 * l, h))))
        enc.append(h)
    for l, k in ((2, 8), (1, 10), (0, 12)):
        h = torch.cat([F.interpolate(h, scale_factor=2, mode="nearest"), enc[l]], dim=1)
        h = torch.relu(conv(k + 1, torch.relu(conv(k, h))))
    out = conv(14, h)[0, 0]
    if not grads:
        return out
    loss = (out - target.double()).square().mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grads": flat.grad}


def exact(case, seed):
    if case["kind"] == "poisson":
        return {"phi": _exact_poisson(case, seed), "sweeps": None}
    if case["kind"] == "noalloc":
        return {"phi": _exact_poisson(case, seed), "sweeps": None}
    if case["kind"] == "unet_forward":
        return _exact_unet(case, seed, False)
    if case["kind"] == "unet_train":
        return _exact_unet(case, seed, True)
    return None  # whole steps: the state after the steps before is known from the run itself only
