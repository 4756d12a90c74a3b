"""Performance cases of the solver: what a program that uses this package has it
do, each through the public entry point that such a program calls.

``listed()`` names the cases, ``draw()`` gives more of the same ranges,
``prepare()`` makes what the caller holds before the call (inputs on the GPU,
workspaces, solvers), ``run()`` is one pass, ``work()`` what a pass cannot do
without, and ``exact()`` the same results in 64 bits from plain torch, written
out here from the definitions (cone-beam geometry, Eqs. 1, 2, A.1, A.5, A.8).

The sizes are those of the tests and of the benchmark: 64x64x32 voxels with a
128x96 detector (tiny), 256x256x100 with 512x384 (sequence), 512x512x160 with
1024x768 (precision), 128^2x64 ... 256^2x128 with 256x192 ... 1024x768
(batch), and ragged ones between.  ``ct`` is the reference CT: "phantom" is
piecewise constant, as the benchmark's; "textured" has tissue that varies from
voxel to voxel inside the body, as a reconstructed CT does.

The library computes in float32 and carries only sums in double, so J, (a, b),
dJ/dw and the coefficients are returned as float32 values.  The localisation
alone computes in double throughout and keeps it.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1102_1712_gb300 import autograd as A
from paper_1102_1712_gb300 import pcasolve as P

_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


# ------------------------------------------------------------------ cases
def _case(name, op, n, s, det, pitch, angle, K=3, dtype="f32", ct="phantom", mean=False, off=(0.0, 0.0), **kw):
    c = dict(op=op, nx=n[0], ny=n[1], nz=n[2], sx=s[0], sy=s[1], sz=s[2], nu=det[0], nv=det[1], du=pitch[0],
             dv=pitch[1], off_u=off[0], off_v=off[1], angle=angle, K=K, dtype=dtype, ct=ct, mean=mean, **kw)
    if name:
        c["name"] = name
    return c


_TINY = ((64, 64, 32), (4.0, 4.0, 4.0), (128, 96), (3.1, 3.1))
_SEQ = ((256, 256, 100), (2.0, 2.0, 2.5), (512, 384), (0.776, 0.776))
_PREC = ((512, 512, 160), (1.0, 1.0, 2.0), (1024, 768), (0.388, 0.388))


def listed():
    return [
        # one localisation after a solve: the smallest call, a chain of dependent steps
        _case("localize", "localize", *_SEQ, 0.4),
        # a DRR of a small volume, as an interactive viewer or a registration inner loop renders it
        _case("drr_tiny", "drr", *_TINY, 0.0),
        # the projector at the size of the sequence, at an oblique angle, on a CT with texture
        _case("drr_sequence", "drr", *_SEQ, 0.6, ct="textured"),
        # the transposed projector at the same size: the backprojection of a residual image
        _case("adjoint_sequence", "adjoint", *_SEQ, 2.2),
        # simulated measurements: Siddon's exact path, every frame of a synthetic sequence
        _case("siddon_sequence", "siddon", *_SEQ, 1.2),
        # the deformed CT itself, for display or dose: Eq. (1) and the warp, with a mean field
        _case("deform_precision", "deform", *_PREC, 0.0, K=5, mean=True, ct="textured"),
        # cost and gradient for a caller's own optimiser: ragged sizes, one component, shifted detector
        _case("cost_grad_ragged", "cost_grad", (61, 53, 29), (4.0, 3.5, 4.5), (127, 95), (3.1, 3.3), 2.3, K=1,
              ct="textured", mean=True, off=(7.0, -5.0)),
        # the same at the size of the sequence
        _case("cost_grad_sequence", "cost_grad", *_SEQ, 0.8, ct="textured"),
        # and at the largest size, the motion model stored in 16 bits
        _case("cost_grad_precision", "cost_grad", *_PREC, 5.2, K=5, dtype="bf16", ct="textured"),
        # differentiation with respect to the coefficients and the reference CT: forward and backward
        _case("autograd_ragged", "autograd", (149, 131, 67), (3.0, 3.2, 3.5), (301, 223), (1.3, 1.3), 1.0, K=2,
              ct="textured"),
        # the host-driven solve of the tiny problem, from rest
        _case("solve_tiny", "solve", *_TINY, 0.0, iters=6, mu_min=0.025),
        # consecutive projections of the sequence through the device-driven solver: warm start, solve, localisation
        _case("run_sequence", "run", *_SEQ, 0.5, frames=3, iters=2, mu_min=0.025),
    ]


# Largest in-plane extent (voxels) and detector width (pixels) of a drawn case
# of each entry point: the precision sizes where a pass stays below the largest
# listed case, smaller where it is many evaluations or visits every voxel.
_LIMIT = {"localize": (512, 1024), "drr": (512, 1024), "adjoint": (256, 512), "siddon": (256, 512),
          "deform": (448, 1024), "cost_grad": (448, 896), "autograd": (224, 448), "solve": (224, 512),
          "run": (256, 512)}


def draw(rng):
    op = rng.choice(sorted(_LIMIT))
    top, wide = _LIMIT[op]

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    nx = spread(48, top)
    ny = max(40, min(top, int(nx * rng.uniform(0.75, 1.2))))
    nz = spread(24, max(32, min(160, nx // 2)))
    nu = spread(96, wide)
    nv = max(64, int(nu * rng.uniform(0.6, 0.9)))
    fov, axial, side = rng.uniform(380.0, 520.0), rng.uniform(180.0, 300.0), rng.uniform(360.0, 420.0)
    s = (round(fov / nx, 4), round(fov / ny * rng.uniform(0.85, 1.0), 4), round(axial / nz, 4))
    pitch = (round(side / nu, 4), round(side / nu * rng.uniform(0.9, 1.1), 4))
    off = (0.0, 0.0) if rng.random() < 0.5 else (round(rng.uniform(-20, 20), 2), round(rng.uniform(-10, 10), 2))
    kw = dict(K=rng.choice((1, 2, 3, 3, 4, 5)), ct=rng.choice(("phantom", "textured")), mean=rng.random() < 0.3,
              off=off)
    if op in ("cost_grad", "solve", "run", "localize"):
        kw["dtype"] = rng.choice(("f32", "f32", "bf16", "f16"))
    if op == "solve":
        kw.update(iters=rng.choice((2, 3, 4)), mu_min=0.025)
    if op == "run":
        kw.update(frames=rng.choice((2, 3)), iters=2, mu_min=0.025)
    return _case(None, op, (nx, ny, nz), s, (nu, nv), pitch, round(rng.uniform(0.0, 2 * math.pi), 4), **kw)


# ----------------------------------------------------------------- inputs
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _vol(c):
    return dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], sx=c["sx"], sy=c["sy"], sz=c["sz"],
                ox=-0.5 * (c["nx"] - 1) * c["sx"], oy=-0.5 * (c["ny"] - 1) * c["sy"], oz=-0.5 * (c["nz"] - 1) * c["sz"])


def _cb(c, angle=None):
    return dict(sad=1000.0, sdd=1500.0, nu=c["nu"], nv=c["nv"], du=c["du"], dv=c["dv"], off_u=c["off_u"],
                off_v=c["off_v"], angle=c["angle"] if angle is None else angle)


def _step(c):
    return 0.5 * min(c["sx"], c["sy"], c["sz"])


def _params(c):
    """The appendix's constants for O(1) coefficients; a real-time budget of
    iterations, and steps down to 0.025 (a quarter of a millimetre)."""
    return dict(mu0=0.2, alpha=0.1, beta=0.5, mu_min=c["mu_min"], max_iter=c["iters"], max_trials=30, step=_step(c))


def _fields(c, count, g):
    """Smooth random vector fields [count, 3, N], white noise on an 8 mm grid
    smoothed by one cell and interpolated; the largest component peaks at 10 mm."""
    n, s = (c["nz"], c["ny"], c["nx"]), (c["sz"], c["sy"], c["sx"])
    m = [max(4, int(math.ceil(a * b / 8.0)) + 1) for a, b in zip(n, s)]
    f = torch.from_numpy(g.standard_normal((1, 3 * count, *m)))
    for ax in range(3):                                   # Gaussian of one cell, zero outside
        i = torch.arange(m[ax], dtype=torch.float64)
        T = torch.exp(-0.5 * (i[:, None] - i[None, :]) ** 2) / math.sqrt(2 * math.pi)
        f = torch.movedim(torch.tensordot(f, T, dims=([2 + ax], [0])), -1, 2 + ax)
    f = f.reshape(count, 3, -1)
    peak = f.abs().amax(dim=2)
    peak = torch.cat([peak[:1, 2], peak[1:].amax(dim=1)])       # first field: along the body axis
    f = (f * (10.0 / peak)[:, None, None]).float().reshape(1, 3 * count, *m).to(_dev())
    out = torch.empty(3 * count, *n, device=f.device)
    for q in range(3 * count):
        out[q] = F.interpolate(f[:, q:q + 1], size=n, mode="trilinear", align_corners=True)[0, 0]
    return out.reshape(count, 3, -1)


def _grid(c):
    ax = [torch.arange(c[n], device=_dev(), dtype=torch.float32) for n in ("nz", "ny", "nx")]
    v = _vol(c)
    return [(v[o] + v[s] * a) for a, o, s in zip(ax, ("oz", "oy", "ox"), ("sz", "sy", "sx"))]


def _ct(c, g):
    """Chest phantom (body 0.02/mm, lungs 0.005/mm, a tumour of 15 mm radius in
    the right lung) and the tumour's centre; "textured": tissue varies by 10 %."""
    Z, Y, X = _grid(c)
    ext = np.array([c["nx"] * c["sx"], c["ny"] * c["sy"], c["nz"] * c["sz"]])

    def inside(ctr, ax):
        return (((Z - ctr[2]) / ax[2]) ** 2)[:, None, None] + (((Y - ctr[1]) / ax[1]) ** 2)[None, :, None] + \
            (((X - ctr[0]) / ax[0]) ** 2)[None, None, :] <= 1.0

    f = torch.zeros(c["nz"], c["ny"], c["nx"], device=X.device)
    f[inside(0.01 * ext * g.uniform(-1, 1, 3), np.array([0.44, 0.34, 0.62]) * ext * (1 + 0.03 * g.uniform(-1, 1, 3)))] = 0.02
    ctr = None
    for side in (1.0, -1.0):
        lc = np.array([side * 0.2, 0.02, 0.05]) * ext + 0.01 * ext * g.uniform(-1, 1, 3)
        f[inside(lc, np.array([0.14, 0.2, 0.38]) * ext * (1 + 0.05 * g.uniform(-1, 1, 3)))] = 0.005
        ctr = lc if ctr is None else ctr
    ctr = ctr + 4.0 * g.uniform(-1, 1, 3)
    f[inside(ctr, np.full(3, 15.0))] = 0.02
    if c["ct"] == "textured":
        t = torch.Generator(device=f.device).manual_seed(int(g.integers(1 << 31)))
        f *= 1.0 + 0.1 * (2.0 * torch.rand(f.shape, device=f.device, generator=t) - 1.0)
    return f.reshape(-1), ctr


def _trace(n, fps=10.0, period=4.0, K=3, t0=0.0):
    """Regular breathing: w_1 up to 1.5 (15 mm), the others smaller and shifted."""
    t = t0 + np.arange(n) / fps
    lag, scale = [0.0, -0.125, 0.125, 0.25, 0.375], [1.5, 0.45, 0.225, 0.15, 0.1]
    return np.stack([scale[k] * 0.5 * (1 - np.cos(2 * math.pi * (t / period + lag[k]))) for k in range(K)], axis=1)


def _measured(c, f0, mean, U, w, cb, g):
    """A measured image: the projection of the CT moved by w (coarser ray steps
    than the solver's), in other units, with 1 % noise."""
    x = torch.zeros(3, f0.numel(), device=f0.device) if mean is None else mean.float().clone()
    for k in range(U.shape[0]):
        x += float(w[k]) * U[k].float()
    p = _project(_warp(f0.float(), x, c), c, cb, 4.0 * _step(c))
    t = torch.Generator(device=p.device).manual_seed(int(g.integers(1 << 31)))
    y = (p - 0.2) / 1.3
    return (y + 0.01 * y.abs().max() * torch.randn(y.shape, device=y.device, generator=t)).float().contiguous()


def _inputs(c, seed):
    """Every input of a case, from the seed alone."""
    g = np.random.default_rng(seed)
    op, dt, K = c["op"], _TYPES[c["dtype"]], c["K"]
    i = {}
    if op == "adjoint":
        t = torch.Generator(device=_dev()).manual_seed(int(g.integers(1 << 31)))
        i["img"] = torch.randn(c["nv"] * c["nu"], device=_dev(), generator=t)
        return i
    f0, i["c_ref"] = _ct(c, g)
    i["f0"] = f0
    if op in ("drr", "siddon"):
        return i
    U = _fields(c, K, g)
    mean = 0.3 * _fields(c, 1, g)[0] if c["mean"] else None
    i["w"] = np.array([1.0, -0.4, 0.3, 0.2, -0.2])[:K] * g.uniform(0.6, 1.2, K)
    i["f0"], i["U"] = f0.to(dt), U.to(dt)
    i["mean"] = None if mean is None else mean.to(dt)
    if op in ("localize", "deform"):
        return i
    if op == "run":                     # consecutive views 0.6 degrees apart, mid-breath
        at = 10 + int(g.integers(10))
        w = _trace(at + c["frames"], K=K)
        i["angles"] = [c["angle"] + math.radians(0.6) * q for q in range(c["frames"])]
        i["y"] = [_measured(c, i["f0"], i["mean"], i["U"], w[at + q], _cb(c, i["angles"][q]), g) for q in range(c["frames"])]
        i["hist"] = w[at - 2:at][::-1] + 0.04 * g.uniform(-1, 1, (2, K))     # the solutions before
        i["train"] = _trace(400, K=K, t0=0.37)
        return i
    w_true = i["w"]
    i["y"] = _measured(c, i["f0"], i["mean"], i["U"], w_true, _cb(c), g)
    if op in ("cost_grad", "autograd"):
        i["w"] = w_true + 0.3 * g.uniform(-1, 1, K)          # somewhere on the way to the solution
    elif op == "solve":
        i["w"] = np.zeros(K)
    return i


def prepare(case, seed):
    c = case
    i = _inputs(c, seed)
    s = {"case": c, "vol": P.vol_struct(_vol(c)), "cb": P.cb_struct(_cb(c)), "step": _step(c), **i}
    flat = lambda t: None if t is None else t.reshape(-1)  # noqa: E731
    if "U" in i:
        s["U"], s["mean"] = flat(i["U"]), flat(i["mean"])
    op = c["op"]
    if op in ("cost_grad", "solve"):
        s["ws"] = P.Workspace(s["vol"], s["cb"], c["K"])
    if op == "autograd":
        s["prob"] = A.problem(s["U"], s["y"], s["vol"], s["cb"], s["step"], mean=s["mean"])
        s["wt"] = torch.tensor(i["w"], dtype=torch.float32)
    if op in ("solve", "run"):
        s["params"] = P.params_struct(_params(c))
    if op == "run":
        s["solver"] = P.Solver(s["f0"], s["mean"], s["U"], s["vol"], s["cb"], s["params"])
        s["lp"] = P.lp_fit(i["train"], 2)
    return s


def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "drr":
        return P.drr_forward(s["f0"], s["vol"], s["cb"], s["step"])
    if op == "siddon":
        return P.drr_siddon(s["f0"], s["vol"], s["cb"])
    if op == "adjoint":
        return P.drr_adjoint(s["img"], s["vol"], s["cb"], s["step"])
    if op == "deform":
        x = P.pca_dvf(s["mean"], s["U"], s["w"], s["vol"])
        return {"dvf": x, "f": P.warp_volume(s["f0"], x, s["vol"])}
    if op == "localize":
        pos, ok = P.localize_tumor(s["mean"], s["U"], s["w"], s["vol"], s["c_ref"])
        return {"c": pos, "ok": ok}
    if op == "cost_grad":
        J, G, ab = P.cost_grad(s["f0"], s["mean"], s["U"], s["w"], s["y"], s["vol"], s["cb"], s["step"], ws=s["ws"])
        return {"J": float(J), "G": G.astype(np.float32), "ab": np.float32(ab)}
    if op == "autograd":
        w, f0 = s["wt"].clone().requires_grad_(True), s["f0"].detach().requires_grad_(True)
        J = A.pca_cost(w, f0, s["prob"])
        J.backward()
        return {"J": float(J.detach()), "w": w.grad, "f0": f0.grad}
    if op == "solve":
        w, st = P.solve_projection(s["f0"], s["mean"], s["U"], s["y"], s["vol"], s["cb"], s["w"], s["params"], ws=s["ws"])
        return _solved(w, st)
    if op == "run":
        s["solver"].seq_begin(s["lp"], s["c_ref"], w_hist=s["hist"])
        got = s["solver"].solve_sequence(s["y"], s["angles"])
        return [dict(_solved(w, st), c=pos.astype(np.float32)) for w, st, pos, _ in got]
    raise ValueError(op)


def _solved(w, st):
    return {"w": w.astype(np.float32), "J": float(st["J"]), "ab": np.float32((st["a"], st["b"])),
            "iters": int(st["iters"]), "evals": int(st["evals"])}


# ------------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once; 24 operations a ray sample (its
    position and seven interpolations), the same for each of its adjoint's, 4 a
    voxel face crossed by Siddon's path, 50 a warped voxel."""
    c = case
    N, M, K = c["nx"] * c["ny"] * c["nz"], c["nu"] * c["nv"], c["K"]
    e = 4 if c["dtype"] == "f32" else 2
    X, Y, Z = c["nx"] * c["sx"], c["ny"] * c["sy"], c["nz"] * c["sz"]
    sa, ca = abs(math.sin(c["angle"])), abs(math.cos(c["angle"]))
    chord = min(X / max(sa, 1e-9), Y / max(ca, 1e-9))              # of the central ray
    hit = min(1.0, 1.5 * Z / (c["nv"] * c["dv"])) * min(1.0, 1.5 * (X * ca + Y * sa) / (c["nu"] * c["du"]))
    rays = M * hit * chord / _step(c) * 24
    model = e * 3 * N * (K + (1 if c["mean"] else 0))
    warp = 50.0 * N + 6.0 * K * N
    op = c["op"]
    if op == "drr":
        return {"bytes": 4 * N + 4 * M, "flops": rays}
    if op == "siddon":
        return {"bytes": 4 * N + 4 * M, "flops": M * hit * chord * (sa / c["sx"] + ca / c["sy"]) * 4}
    if op == "adjoint":
        return {"bytes": 4 * N + 4 * M, "flops": rays}
    if op == "deform":
        return {"bytes": model + 4 * N + 16 * N, "flops": warp}
    if op == "localize":
        return {"bytes": 8 * e * 3 * (K + 1) + 32, "flops": 50 * 8 * 6 * K}
    one = {"bytes": model + e * N + 4 * M, "flops": 2 * rays + 2 * warp}       # cost and gradient
    if op == "cost_grad":
        return one
    if op == "autograd":
        return {"bytes": 2 * one["bytes"] + 4 * N, "flops": 1.5 * one["flops"] + warp}
    if op == "solve":                  # per iteration a gradient and one more evaluation
        return {"bytes": c["iters"] * one["bytes"], "flops": 1.5 * c["iters"] * one["flops"]}
    return {"bytes": c["frames"] * c["iters"] * one["bytes"], "flops": 2.5 * c["frames"] * c["iters"] * one["flops"]}


# ------------------------------------------- the definitions, in plain torch
def _frame(c, cb):
    a = cb["angle"]
    S = np.array([cb["sad"] * math.sin(a), -cb["sad"] * math.cos(a), 0.0])
    return S, np.array([-math.sin(a), math.cos(a), 0.0]), np.array([math.cos(a), math.sin(a), 0.0])


def _unit(c, cb, n, dtype):
    """Unit directions (mm) of rays n (u fastest): three tensors."""
    _, ew, eu = _frame(c, cb)
    u = ((n % c["nu"]).to(dtype) - 0.5 * (c["nu"] - 1)) * cb["du"] + cb["off_u"]
    v = (torch.div(n, c["nu"], rounding_mode="floor").to(dtype) - 0.5 * (c["nv"] - 1)) * cb["dv"] + cb["off_v"]
    r = torch.sqrt(u * u + v * v + cb["sdd"] ** 2)
    return (cb["sdd"] * ew[0] + u * eu[0]) / r, (cb["sdd"] * ew[1] + u * eu[1]) / r, v / r


def _padded(f, c, halo=2):
    return F.pad(f.reshape(c["nz"], c["ny"], c["nx"]), (halo,) * 6).reshape(-1)


def _taps(q, c, halo=2):
    """Index of the first tap of each position's cell in the padded volume, and the fractions."""
    n = (c["nx"], c["ny"], c["nz"])
    at, z = None, []
    for a, stride in zip(range(3), (1, n[0] + 2 * halo, (n[0] + 2 * halo) * (n[1] + 2 * halo))):
        p = q[a].clamp(-1.5, n[a] + 0.5)                # zero there either way
        fl = torch.floor(p)
        z.append(p - fl)
        l = (fl.to(torch.int64) + halo) * stride
        at = l if at is None else at + l
    return at, z, (n[0] + 2 * halo, (n[0] + 2 * halo) * (n[1] + 2 * halo))


def _interp(fp, q, c, grad=False):
    """Eq. (A.5) at positions q (voxels), zero outside; grad: also Eq. (A.8)."""
    at, (x, y, z), (sy, sz) = _taps(q, c)
    t = lambda o: fp[at + o]  # noqa: E731
    a0, a1 = t(0), t(1)
    b0, b1 = t(sy), t(sy + 1)
    dx = (a1 - a0) * (1 - y) + (b1 - b0) * y if grad else None
    lo = (a0 + x * (a1 - a0)), (b0 + x * (b1 - b0))
    a0, a1 = t(sz), t(sz + 1)
    b0, b1 = t(sz + sy), t(sz + sy + 1)
    hi = (a0 + x * (a1 - a0)), (b0 + x * (b1 - b0))
    lo_y, hi_y = lo[0] + y * (lo[1] - lo[0]), hi[0] + y * (hi[1] - hi[0])
    v = lo_y + z * (hi_y - lo_y)
    if not grad:
        return v
    dx = dx * (1 - z) + ((a1 - a0) * (1 - y) + (b1 - b0) * y) * z
    dy = (lo[1] - lo[0]) * (1 - z) + (hi[1] - hi[0]) * z
    return v, (dx, dy, hi_y - lo_y)


def _positions(x, c, lo, hi):
    """Voxel positions v + x(v) / s of voxels lo ... hi - 1 for a field x [3, N] in mm."""
    n = torch.arange(lo, hi, device=x.device)
    ijk = n % c["nx"], torch.div(n, c["nx"], rounding_mode="floor") % c["ny"], torch.div(n, c["nx"] * c["ny"], rounding_mode="floor")
    return [ijk[a].to(x.dtype) + x[a, lo:hi] / c["s" + "xyz"[a]] for a in range(3)]


_BLOCK = 1 << 23


def _warp(f0, x, c):
    fp = _padded(f0.to(x.dtype), c)
    return torch.cat([_interp(fp, _positions(x, c, b, min(b + _BLOCK, x.shape[1])), c) for b in range(0, x.shape[1], _BLOCK)])


def _marches(c, cb, step, dtype, device):
    """Blocks of rays and their sample positions: (rays, [qx, qy, qz] of shape [rays, samples])."""
    v = _vol(c)
    S, _, _ = _frame(c, cb)
    o, s = (v["ox"], v["oy"], v["oz"]), (c["sx"], c["sy"], c["sz"])
    n = (c["nx"], c["ny"], c["nz"])
    M = c["nu"] * c["nv"]
    b0 = 0
    most = int(math.sqrt(sum((n[a] + 1) ** 2 * s[a] ** 2 for a in range(3))) / step) + 3
    while b0 < M:
        b1 = min(M, b0 + max(1, 2 * _BLOCK // most))
        D = _unit(c, cb, torch.arange(b0, b1, device=device), torch.float64)
        tl = torch.full((b1 - b0,), -1e30, device=device, dtype=torch.float64)
        th = -tl
        for a in range(3):
            d = torch.where(D[a] == 0, torch.full_like(D[a], 1e-300), D[a])
            p, q = (o[a] - s[a] - S[a]) / d, (o[a] + n[a] * s[a] - S[a]) / d
            tl, th = torch.maximum(tl, torch.minimum(p, q)), torch.minimum(th, torch.maximum(p, q))
        i0, i1 = torch.ceil(tl / step), torch.floor(th / step)
        live = tl <= th
        if bool(live.any()):
            # each ray's samples from its own first one; the last ones of a short ray lie outside, where taps are zero
            cnt = int((i1 - i0)[live].max().item()) + 1
            i = torch.where(live, i0, torch.zeros_like(i0))[:, None] + torch.arange(max(cnt, 0), device=device, dtype=torch.float64)
            far = torch.where(live[:, None], (i * step), torch.full_like(i, 1e7))
            yield b0, b1, [((S[a] - o[a]) / s[a] + far * (D[a] / s[a])[:, None]).to(dtype) for a in range(3)]
        b0 = b1


def _project(f, c, cb, step):
    fp = _padded(f, c)
    p = torch.zeros(c["nu"] * c["nv"], device=f.device, dtype=f.dtype)
    for b0, b1, q in _marches(c, cb, step, f.dtype, f.device):
        p[b0:b1] = _interp(fp, q, c).sum(dim=1) * step
    return p


def _backproject(img, c, cb, step):
    g = torch.zeros((c["nx"] + 4) * (c["ny"] + 4) * (c["nz"] + 4), device=img.device, dtype=img.dtype)
    for b0, b1, q in _marches(c, cb, step, img.dtype, img.device):
        at, (x, y, z), (sy, sz) = _taps(q, c)
        r = img[b0:b1, None] * step
        for t in range(8):
            w = (x if t & 1 else 1 - x) * (y if t & 2 else 1 - y) * (z if t & 4 else 1 - z) * r
            g.index_add_(0, (at + (t & 1) + (sy if t & 2 else 0) + (sz if t & 4 else 0)).reshape(-1), w.reshape(-1))
    return g.reshape(c["nz"] + 4, c["ny"] + 4, c["nx"] + 4)[2:-2, 2:-2, 2:-2].reshape(-1)


def _field(i, w):
    U, mean = i["U"], i["mean"]
    x = torch.zeros(3, U.shape[2], device=U.device, dtype=torch.float64) if mean is None else mean.double()
    for k in range(U.shape[0]):
        x = x + float(w[k]) * U[k].double()
    return x


def _fit(p, y):
    """Eq. (A.1)."""
    M, Sp, Sy, Syp, Syy = p.numel(), p.sum(), y.sum(), (y * p).sum(), (y * y).sum()
    det = M * Syy - Sy * Sy
    return float((M * Syp - Sy * Sp) / det), float((Syy * Sp - Sy * Syp) / det)


class _Exact:
    """Eq. (2) and its gradients for one image."""

    def __init__(self, i, c, y, cb):
        self.i, self.c, self.y, self.cb = i, c, y.double(), cb
        self.f0 = i["f0"].double()

    def image(self, w):
        return _project(_warp(self.f0, _field(self.i, w), self.c), self.c, self.cb, _step(self.c))

    def gradient(self, w, p, want_f0=False):
        c, U = self.c, self.i["U"]
        a, b = _fit(p, self.y)
        r = p - a * self.y - b
        z = 2.0 * _backproject(r, c, self.cb, _step(c))
        x, fp = _field(self.i, w), _padded(self.f0, c)
        G = np.zeros(U.shape[0])
        df = torch.zeros_like(fp) if want_f0 else None
        for lo in range(0, z.numel(), _BLOCK):
            hi = min(lo + _BLOCK, z.numel())
            q = _positions(x, c, lo, hi)
            _, d = _interp(fp, q, c, grad=True)
            for k in range(U.shape[0]):
                G[k] += float(sum((z[lo:hi] * d[e] / c["s" + "xyz"[e]] * U[k, e, lo:hi].double()).sum() for e in range(3)))
            if want_f0:
                at, (u, v, t), (sy, sz) = _taps(q, c)
                for m in range(8):
                    wt = (u if m & 1 else 1 - u) * (v if m & 2 else 1 - v) * (t if m & 4 else 1 - t)
                    df.index_add_(0, at + (m & 1) + (sy if m & 2 else 0) + (sz if m & 4 else 0), wt * z[lo:hi])
        if want_f0:
            df = df.reshape(c["nz"] + 4, c["ny"] + 4, c["nx"] + 4)[2:-2, 2:-2, 2:-2].reshape(-1)
        return float((r * r).sum()), G, (a, b), df

    def solve(self, w, prm):
        """The appendix's loop: fit (a, b), one normalised gradient step under Armijo's rule."""
        w, p, evals, iters = np.array(w, float), self.image(w), 1, 0
        a = b = J = 0.0
        for _ in range(prm["max_iter"]):
            J, G, (a, b), _ = self.gradient(w, p)
            norm = float(np.linalg.norm(G))
            if norm == 0.0:
                break
            iters += 1
            mu, trials, taken = prm["mu0"], 0, False
            while mu >= prm["mu_min"] and trials < prm["max_trials"]:
                pt = self.image(w - mu * G / norm)
                r = pt - a * self.y - b
                Jt = float((r * r).sum())
                trials += 1
                evals += 1
                if Jt <= J - prm["alpha"] * mu * norm:
                    w, p, J, taken = w - mu * G / norm, pt, Jt, True
                    break
                mu *= prm["beta"]
            if not taken:
                break
        return {"w": w, "J": J, "ab": np.array((a, b)), "iters": iters, "evals": evals}


def _locate(i, c, w, c_ref, cap=50, tol=1e-6):
    """Sec. II.A: c = c_ref - x(c) by fixed point, x interpolated and zero outside."""
    v = _vol(c)
    n, s = (c["nx"], c["ny"], c["nz"]), (c["sx"], c["sy"], c["sz"])
    o = (v["ox"], v["oy"], v["oz"])
    y, ok = np.zeros(3), False
    for _ in range(cap):
        q = [min(max((c_ref[a] + y[a] - o[a]) / s[a], -2.0), n[a] + 1.0) for a in range(3)]
        fl = [math.floor(t) for t in q]
        x = np.zeros(3)
        for t in range(8):
            b = [(t >> a) & 1 for a in range(3)]
            l = [fl[a] + b[a] for a in range(3)]
            wt = np.prod([(q[a] - fl[a]) if b[a] else 1 - (q[a] - fl[a]) for a in range(3)])
            if wt != 0.0 and all(0 <= l[a] < n[a] for a in range(3)):
                at = (l[2] * n[1] + l[1]) * n[0] + l[0]
                m = i["U"][:, :, at].double().cpu().numpy()
                x += wt * ((0 if i["mean"] is None else i["mean"][:, at].double().cpu().numpy()) + w @ m)
        change = np.abs(-x - y).max()
        y = -x
        if change < tol:
            ok = True
            break
    return c_ref + y, ok


def _siddon(f, c, cb):
    """Sum over the voxels a ray crosses of the length inside times the value:
    every face crossing inside the volume sorted, each segment's midpoint looked up."""
    v = _vol(c)
    S, _, _ = _frame(c, cb)
    n, s = (c["nx"], c["ny"], c["nz"]), (c["sx"], c["sy"], c["sz"])
    o = (v["ox"], v["oy"], v["oz"])
    M, dev = c["nu"] * c["nv"], f.device
    out = torch.zeros(M, device=dev, dtype=torch.float64)
    rows = max(1, _BLOCK // (sum(n) + 5))
    for b0 in range(0, M, rows):
        b1 = min(M, b0 + rows)
        D = _unit(c, cb, torch.arange(b0, b1, device=dev), torch.float64)
        tin = torch.zeros(b1 - b0, device=dev, dtype=torch.float64)
        tout = torch.full_like(tin, 1e30)
        planes = []
        for a in range(3):
            d = torch.where(D[a] == 0, torch.full_like(D[a], 1e-300), D[a])
            t = (o[a] + (torch.arange(n[a] + 1, device=dev, dtype=torch.float64) - 0.5) * s[a] - S[a])[None, :] / d[:, None]
            tin, tout = torch.maximum(tin, t.amin(1)), torch.minimum(tout, t.amax(1))
            planes.append(t)
        live = tin < tout
        t = torch.cat(planes, dim=1)
        t = torch.minimum(torch.maximum(t, tin[:, None]), torch.maximum(tin, tout)[:, None]).sort(dim=1).values
        mid, ln = 0.5 * (t[:, 1:] + t[:, :-1]), t[:, 1:] - t[:, :-1]
        at = None
        for a, stride in zip(range(3), (1, n[0], n[0] * n[1])):
            l = torch.floor((S[a] + mid * D[a][:, None] - o[a]) / s[a] + 0.5).clamp(0, n[a] - 1).to(torch.int64) * stride
            at = l if at is None else at + l
        out[b0:b1] = torch.where(live, (ln * f.double()[at]).sum(1), torch.zeros_like(tin))
    return out


def exact(case, seed):
    c = case
    op = c["op"]
    i = _inputs(c, seed)
    if op == "drr":
        return _project(i["f0"].double(), c, _cb(c), _step(c))
    if op == "siddon":
        return _siddon(i["f0"], c, _cb(c))
    if op == "adjoint":
        return _backproject(i["img"].double(), c, _cb(c), _step(c))
    if op == "deform":
        x = _field(i, i["w"])
        return {"dvf": x.reshape(-1), "f": _warp(i["f0"].double(), x, c)}
    if op == "localize":
        pos, ok = _locate(i, c, i["w"], i["c_ref"])
        return {"c": pos, "ok": ok}
    if op in ("cost_grad", "autograd"):
        E = _Exact(i, c, i["y"], _cb(c))
        w = np.asarray(i["w"], np.float32).astype(float) if op == "autograd" else i["w"]
        J, G, ab, df = E.gradient(w, E.image(w), want_f0=op == "autograd")
        return {"J": J, "w": G, "f0": df} if op == "autograd" else {"J": J, "G": G, "ab": np.array(ab)}
    if op == "solve":
        return _Exact(i, c, i["y"], _cb(c)).solve(i["w"], _params(c))
    h = [np.array(r) for r in i["hist"]]
    lp = _predictor(i["train"])
    out = []
    for q in range(c["frames"]):
        w0 = lp[:, 0] * h[0] + lp[:, 1] * h[1]
        r = _Exact(i, c, i["y"][q], _cb(c, i["angles"][q])).solve(w0, _params(c))
        h = [r["w"], h[0]]
        out.append(dict(r, c=_locate(i, c, r["w"], i["c_ref"])[0]))
    return out


def _predictor(tr):
    """Eq. (3) with two terms: least squares per coefficient."""
    return np.stack([np.linalg.lstsq(np.stack([tr[1:-1, k], tr[:-2, k]], axis=1), tr[2:, k], rcond=None)[0]
                     for k in range(tr.shape[1])])
