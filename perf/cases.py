"""Timed cases of the registration framework, through its public entry points.

A case is a dict of plain values with a ``kind``:

  pair    Context.pairwise: one operator application (a live view, a spot check of two frames)
  scan    Context.scan of one stored series and, for the nonrigid model, the registered mean made
          from its control grids: the offline job of the framework
  batch   Context.scan_batch of several series of one size, the elements alone
  stream  Stream: frames submitted as an acquisition delivers them, results polled
  warp    Context.warp with prefixes that are already known: the registered series and its mean
  energy  Context.energy_grid / energy_rigid: one energy and gradient evaluation

The frames are the package's seeded synthetic lattice series.  Drift, field and noise take the
values of its named workloads (c1: +-3 px drift per frame, SNR 10; c2: +-1 px, field 1.5 px;
c3: SNR 3-20 and sudden jumps).
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_2010_12478_gb300 import binding as B
from paper_2010_12478_gb300 import synth

DEV = "cuda"
MAX_PIXELS = 1024 * 512 * 512     # frames x pixels of the largest listed case
ELEM = np.dtype([("i", "<i4"), ("k", "<i4"), ("p", "<f4", (3,))])


def listed():
    return [
        # the smallest call: one pair of thumbnails, rigid, as a drift monitor makes it.  The pairs bound
        # the steps per level, as a live view bounds its latency: four rigid and six nonrigid ones are
        # about what the default stop takes on such frames
        dict(name="pair rigid 160x128", kind="pair", mode="rigid", storage="f32", H=160, W=128, step=3.0, snr=10.0,
             init=False, max_iter=4),
        # a small nonrigid pair, and one of the ordinary size
        dict(name="pair nonrigid 128x128", kind="pair", mode="nonrigid", storage="f32", H=128, W=128, step=3.0,
             snr=10.0, init=False, max_iter=6),
        dict(name="pair nonrigid 512x512", kind="pair", mode="nonrigid", storage="f32", H=512, W=512, step=1.0,
             snr=10.0, init=False, max_iter=6),
        # a large odd frame in reduced precision, from a known initial field (operator B by itself)
        dict(name="pair nonrigid 741x1003 bf16", kind="pair", mode="nonrigid", storage="bf16", H=741, W=1003,
             step=1.0, snr=10.0, init=True, max_iter=6),
        # a short rigid series with the default executor: one launch per depth of the scan
        dict(name="scan rigid 24x256x256", kind="scan", mode="rigid", storage="f32", N=24, H=256, W=256, step=3.0,
             snr_lo=10.0, snr_hi=10.0, jump=0.0, exec="level", host=False),
        # a rigid series that lies in page-locked host memory: staging, pyramids, scan, results
        dict(name="scan rigid 128x512x512 host", kind="scan", mode="rigid", storage="f32", N=128, H=512, W=512,
             step=1.0, snr_lo=10.0, snr_hi=10.0, jump=0.0, exec="persistent", host=True),
        # the ordinary job: 256 frames of 512x512, nonrigid, through the device queue, then the mean
        dict(name="scan nonrigid 256x512x512", kind="scan", mode="nonrigid", storage="f32", N=256, H=512, W=512,
             step=1.0, snr_lo=10.0, snr_hi=10.0, jump=0.0, exec="persistent", host=False),
        # the largest: a long load-imbalanced series (SNR 3-20, 5 % jumps)
        dict(name="scan nonrigid 1024x512x512", kind="scan", mode="nonrigid", storage="f32", N=1024, H=512, W=512,
             step=1.0, snr_lo=3.0, snr_hi=20.0, jump=0.05, exec="persistent", host=False),
        # independent series of small frames sharing one queue, FP16 pyramids
        dict(name="batch nonrigid 8x32x256x256 f16", kind="batch", mode="nonrigid", storage="f16", S=8, N=32, H=256,
             W=256, step=3.0, snr_lo=3.0, snr_hi=20.0),
        # the serving path: one acquisition stream, frames submitted as fast as they are accepted
        dict(name="stream nonrigid 32x256x256", kind="stream", mode="nonrigid", N=32, H=256, W=256, step=3.0,
             snr=10.0, lookback=2),
        # registered frames and mean of a series whose control grids are known
        dict(name="warp nonrigid 256x512x512", kind="warp", mode="nonrigid", N=256, H=512, W=512, out=True),
        # one energy and gradient at a given control grid (inspection of a result)
        dict(name="energy nonrigid 512x512", kind="energy", mode="nonrigid", H=512, W=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "scan", "scan", "scan", "batch", "stream", "warp", "warp", "energy"])
    mode = rng.choice(["rigid", "nonrigid", "nonrigid"])
    H, W = _log(rng, 160, 1040), _log(rng, 160, 1040)
    if kind == "pair":
        return dict(kind=kind, mode=mode, storage=rng.choice(["f32", "f32", "bf16", "f16"]), H=H, W=W,
                    step=rng.choice([1.0, 3.0]) if mode == "nonrigid" else 3.0, snr=10.0,
                    init=mode == "nonrigid" and rng.random() < 0.3, max_iter=6 if mode == "nonrigid" else 4)
    if kind == "energy":
        return dict(kind=kind, mode=mode, H=H, W=W)
    if kind == "warp":
        return dict(kind=kind, mode=mode, N=_log(rng, 8, max(9, min(400, 256 * 512 * 512 // (H * W)))), H=H, W=W,
                    out=rng.random() < 0.6)
    H, W = _log(rng, 240, 720), _log(rng, 240, 720)
    most = max(33, min(700, MAX_PIXELS // (2 * H * W)))
    if kind == "stream":
        return dict(kind=kind, mode=mode, N=_log(rng, 24, 64), H=H, W=W, step=3.0, snr=10.0,
                    lookback=rng.choice([1, 2, 4]))
    if kind == "batch":
        S = rng.choice([2, 4, 8])
        return dict(kind=kind, mode=mode, storage=rng.choice(["f32", "f16"]), S=S,
                    N=_log(rng, 24, max(25, min(96, most // S))), H=H, W=W, step=3.0, snr_lo=3.0, snr_hi=20.0)
    # a long series drifts slowly, as one that keeps its overlap with the first frame does
    N = _log(rng, 24, most if mode == "nonrigid" else min(160, most))
    return dict(kind=kind, mode=mode, storage="f32", N=N, H=H, W=W, step=1.0 if N > 96 else rng.choice([2.0, 3.0]),
                snr_lo=rng.choice([3.0, 10.0]), snr_hi=20.0,
                jump=rng.choice([0.0, 0.05]) if mode == "nonrigid" else 0.0,
                exec=rng.choice(["persistent", "persistent", "level"]), host=rng.random() < 0.25)


# ------------------------------------------------------------------ inputs
def _series(N, H, W, step, snr_lo, snr_hi, seed, series=0, jump=0.0, out=None):
    return synth.make_series(
        synth.SeriesSpec(N, H, W, step=step, field_amp=1.5, snr=(snr_lo, snr_hi), jump_frac=jump,
                         jump_max=3.0 if jump else 0.0, seed=seed, series=series), device=DEV, frames_out=out)


def _smooth_grids(n, ny, nx, seed):
    """n control grids: a random-walk drift and a slowly varying sinusoidal field, as prefixes have."""
    rng = np.random.Generator(np.random.PCG64([seed, 77]))
    drift = torch.from_numpy(np.cumsum(rng.uniform(-1.0, 1.0, (n, 2)), axis=0)).to(DEV)
    ph = torch.from_numpy(rng.uniform(0.0, 2.0 * math.pi, (2, 3))).to(DEV)
    t = torch.arange(n, device=DEV, dtype=torch.float64).view(-1, 1, 1) * 0.1
    y = torch.linspace(0, 2.0 * math.pi, ny, device=DEV, dtype=torch.float64).view(1, -1, 1)
    x = torch.linspace(0, 2.0 * math.pi, nx, device=DEV, dtype=torch.float64).view(1, 1, -1)
    g = [0.7 * torch.sin(x + ph[a, 0] + t) + 0.7 * torch.sin(y + x + ph[a, 1] + t) + drift[:, a].view(-1, 1, 1)
         for a in range(2)]
    return torch.stack(g, -1).to(torch.float32).contiguous()


def _rigid_prefixes(n, seed):
    rng = np.random.Generator(np.random.PCG64([seed, 78]))
    e = np.zeros(n, ELEM)
    e["k"] = np.arange(1, n + 1)
    e["p"][:, 0] = rng.uniform(-0.005, 0.005, n)
    e["p"][:, 1:] = np.cumsum(rng.uniform(-1.0, 1.0, (n, 2)), axis=0)
    return e


def _inputs(case, seed):
    kind, H, W = case["kind"], case["H"], case["W"]
    if kind in ("pair", "energy"):
        s = _series(2, H, W, case.get("step", 1.0), case.get("snr", 10.0), case.get("snr", 10.0), seed)
        d = dict(R=s.frames[0], T=s.frames[1], field=None)
        if kind == "pair" and case["init"]:
            # an earlier estimate: the drift, off by a few tenths of a pixel
            off = np.random.Generator(np.random.PCG64([seed, 79])).uniform(-0.3, 0.3, 2) + s.truth_shift[1]
            d["field"] = torch.from_numpy(off).to(DEV, torch.float32).view(2, 1, 1).expand(2, H, W).contiguous()
        if kind == "energy":
            if case["mode"] == "rigid":
                d["theta"] = [0.001, float(s.truth_shift[1, 0]) + 0.21, float(s.truth_shift[1, 1]) - 0.17]
            else:
                nx, ny, _ = B.grid_dims(W, H, levels=1)
                d["grid"] = _smooth_grids(1, ny, nx, seed)[0].contiguous()
        return d
    if kind == "batch":
        fr = torch.empty((case["S"], case["N"], H, W), device=DEV)
        for q in range(case["S"]):
            _series(case["N"], H, W, case["step"], case["snr_lo"], case["snr_hi"], seed, q, out=fr[q])
        return dict(frames=fr)
    if kind == "warp":
        N = case["N"]
        d = dict(frames=_series(N, H, W, 1.0, 10.0, 10.0, seed).frames)
        if case["mode"] == "rigid":
            d["elems"] = torch.from_numpy(_rigid_prefixes(N - 1, seed).view(np.uint8).copy()).to(DEV)
        else:
            nx, ny, _ = B.grid_dims(W, H)
            d["grids"] = _smooth_grids(N - 1, ny, nx, seed)
        return d
    lo, hi = (case["snr"], case["snr"]) if kind == "stream" else (case["snr_lo"], case["snr_hi"])
    fr = _series(case["N"], H, W, case["step"], lo, hi, seed, jump=case.get("jump", 0.0)).frames
    if case.get("host"):
        fr = fr.cpu().pin_memory()
    return dict(frames=fr)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["ctx"] = B.Context(B.Config(mode=case["mode"], storage=case.get("storage", "f32"),
                                  max_iter=case.get("max_iter", 500)))
    kind, H, W = case["kind"], case["H"], case["W"]
    nonrigid = case["mode"] == "nonrigid"
    # result buffers, which a program allocates once
    if kind == "pair" and nonrigid:
        s["field_out"] = torch.empty((2, H, W), device=DEV)
    if kind == "energy" and nonrigid:
        s["grad"] = torch.empty_like(s["grid"])
    if kind == "scan":
        s["mean"] = torch.empty((H, W), device=DEV)
        s["dframes"] = None if case["host"] else s["frames"]
        if nonrigid:
            nx, ny, _ = B.grid_dims(W, H)
            s["grids"] = torch.empty((case["N"] - 1, ny, nx, 2), device=DEV)
    if kind == "warp":
        s["mean"] = torch.empty((H, W), device=DEV)
        s["out"] = torch.empty((case["N"], H, W), device=DEV) if case["out"] else None
    return s


# ------------------------------------------------------------------ the call
def _elements(el):
    return np.frombuffer(el, ELEM)["p"].copy()


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "pair":
        if case["mode"] == "rigid":
            e, _ = ctx.pairwise(s["R"], s["T"])
            return np.array(e[2:], np.float32)
        ctx.pairwise(s["R"], s["T"], field_in=s["field"], field_out=s["field_out"])
        return s["field_out"]
    if kind == "energy":
        if case["mode"] == "rigid":
            E, g = ctx.energy_rigid(s["R"], s["T"], s["theta"])
            return [E, g.astype(np.float32)]
        return [ctx.energy_grid(s["R"], s["T"], s["grid"], s["grad"]), s["grad"]]
    if kind == "scan":
        el, _ = ctx.scan(s["frames"], exec=case["exec"], raw=True)
        if s["dframes"] is None:
            return [_elements(el)]
        if case["mode"] == "rigid":
            ctx.warp(s["dframes"], elems=el, mean=s["mean"])
        else:
            ctx.scan_grids(s["grids"])
            ctx.warp(s["dframes"], grids=s["grids"], mean=s["mean"])
        return [_elements(el), s["mean"]]
    if kind == "batch":
        el, _ = ctx.scan_batch(s["frames"], raw=True)
        return _elements(el)
    if kind == "warp":
        ctx.warp(s["frames"], elems=s.get("elems"), grids=s.get("grids"), out=s["out"], mean=s["mean"])
        return [s["out"], s["mean"]] if case["out"] else [s["mean"]]
    # stream: a first-in first-out feed; a refused frame waits for a result
    N = case["N"]
    st = B.Stream(ctx, case["W"], case["H"])
    st.set_lookback(case["lookback"])
    res, i, give_up = [], 0, time.monotonic() + 20.0
    while len(res) < N:
        if i < N and st.submit(s["frames"][i], i) == B.REG_OK:
            i += 1
            continue
        res += st.poll(64, 1000)
        if time.monotonic() > give_up:
            raise RuntimeError("the stream does not finish")
    st.close()
    return np.array([r["elem"][2:] for r in res], np.float32)


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: every input read and every result written once.  Operations: a pixel evaluation of
    the rigid model is taken as 40 and of the nonrigid one as 90 floating-point operations
    (sample, derivative, moments, gradient), and an operator application as 13 evaluations at
    full resolution with a quarter of that per coarser level (six steps and the level's start)."""
    P = case["H"] * case["W"]
    kind, nonrigid = case["kind"], case["mode"] == "nonrigid"
    per_eval = 90.0 if nonrigid else 40.0
    op = per_eval * P * 13 * 1.25
    Nc = (P // 256 if nonrigid else 1) * 8
    if kind == "pair":
        return {"bytes": 4.0 * P * (2 + (2 if nonrigid else 0) + (2 if case["init"] else 0)), "flops": op}
    if kind == "energy":
        return {"bytes": 8.0 * P + 2 * Nc, "flops": per_eval * P}
    if kind == "warp":
        N = case["N"]
        return {"bytes": 4.0 * P * (N * (2 if case["out"] else 1) + 1) + N * Nc, "flops": 25.0 * P * N}
    S, N = case.get("S", 1), case["N"]
    mean = kind == "scan" and not case["host"]
    return {"bytes": S * (4.0 * P * N + 20.0 * N) + (4.0 * P * (N + 1) if mean else 0.0),
            "flops": S * 3.0 * N * op + (25.0 * P * N if mean else 0.0)}


# ------------------------------------------------------------------ in 64 bits
def _down(a):
    """2x2 box average, the last odd row and column repeated."""
    H, W = a.shape
    r1 = torch.clamp(torch.arange(0, H, 2, device=a.device) + 1, max=H - 1)
    c1 = torch.clamp(torch.arange(0, W, 2, device=a.device) + 1, max=W - 1)
    b = a[0::2] + a[r1]
    return 0.25 * (b[:, 0::2] + b[:, c1])


def _bilinear(T, px, py):
    """Bilinear value with clamp-to-edge."""
    H, W = T.shape
    px, py = px.clamp(0, W - 1), py.clamp(0, H - 1)
    x, y = px.detach().floor().clamp(max=W - 2), py.detach().floor().clamp(max=H - 2)
    fx, fy = px - x, py - y
    i = (y * W + x).long()
    t = T.reshape(-1)
    top = (1 - fx) * t[i] + fx * t[i + 1]
    bot = (1 - fx) * t[i + W] + fx * t[i + W + 1]
    return (1 - fy) * top + fy * bot


def _bspline(T, px, py):
    """Quadratic B-spline model of the samples, which are the mean beyond the border; its value and
    its two derivatives."""
    H, W = T.shape
    E = torch.nn.functional.pad(T[None, None], (3, 3, 3, 3), value=float(T.mean()))[0, 0]
    Wp, t = W + 6, E.reshape(-1)
    x, y = (px.detach() + 0.5).floor(), (py.detach() + 0.5).floor()
    tx, ty = px - x, py - y
    i = ((y.clamp(-2, H + 1) + 3) * Wp + x.clamp(-2, W + 1) + 3).long()
    wx = [0.5 * (0.5 - tx) ** 2, 0.75 - tx ** 2, 0.5 * (0.5 + tx) ** 2]
    wy = [0.5 * (0.5 - ty) ** 2, 0.75 - ty ** 2, 0.5 * (0.5 + ty) ** 2]
    dx, dy = [tx - 0.5, -2 * tx, tx + 0.5], [ty - 0.5, -2 * ty, ty + 0.5]
    v = gx = gy = 0.0
    for r in (-1, 0, 1):
        row = [t[i + r * Wp + k] for k in (-1, 0, 1)]
        a = wx[0] * row[0] + wx[1] * row[1] + wx[2] * row[2]
        b = dx[0] * row[0] + dx[1] * row[1] + dx[2] * row[2]
        v, gx, gy = v + wy[r + 1] * a, gx + wy[r + 1] * b, gy + dy[r + 1] * a
    return v, gx, gy


def _ncc_energy(R, t):
    r, t = R - R.mean(), t - t.mean()
    return 1.0 - (r * t).sum() / torch.sqrt((r * r).sum() * (t * t).sum())


class _Rigid:
    """The rigid model at one level: parameters (alpha, Gx, Gy), metric diag(rho^2, 1, 1)."""

    def __init__(self, R, T):
        H, W = R.shape
        self.R, self.T = R, T
        self.y, self.x = torch.meshgrid(torch.arange(H, device=DEV).double() - 0.5 * (H - 1),
                                        torch.arange(W, device=DEV).double() - 0.5 * (W - 1), indexing="ij")
        self.m = torch.tensor([(0.25 * (W + H)) ** 2, 1.0, 1.0], device=DEV, dtype=torch.float64)
        self.n = 1.0

    def energy(self, c):
        H, W = self.R.shape
        ca, sa = torch.cos(c[0]), torch.sin(c[0])
        return _ncc_energy(self.R, _bilinear(self.T, ca * self.x - sa * self.y + 0.5 * (W - 1) + c[1],
                                             sa * self.x + ca * self.y + 0.5 * (H - 1) + c[2]))

    def largest(self, d):
        return math.sqrt(float((self.m * d * d).sum()))


class _Field:
    """The control-grid model at level l: parameters [ny, nx, 2] in that level's pixels, the
    Gauss-Newton scalar product at `c0`, regulariser weight lam."""

    def __init__(self, R, T, spacing, nx, ny, level, lam, c0=None):
        self.T, self.P, self.lam = T, R.numel(), lam
        H, W = R.shape
        iy, ix = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(),
                                indexing="ij")
        self.R = _bspline(R, ix, iy)[0]
        self.px, self.py = ix, iy
        gx = ((2 ** level * ix + (2 ** level - 1) / 2) / spacing).clamp(max=nx - 1)
        gy = ((2 ** level * iy + (2 ** level - 1) / 2) / spacing).clamp(max=ny - 1)
        cx, cy = gx.floor().clamp(max=nx - 2), gy.floor().clamp(max=ny - 2)
        fx, fy = gx - cx, gy - cy
        base = (cy * nx + cx).long()
        self.taps = [(base + a * nx + b, (fy if a else 1 - fy) * (fx if b else 1 - fx)) for a in (0, 1) for b in (0, 1)]
        self.n = float(nx * ny)
        self.m = torch.ones((ny, nx, 2), device=DEV, dtype=torch.float64)
        if c0 is None:
            return
        ux, uy = self._u(c0)
        t, dx, dy = _bspline(T, ix + ux, iy + uy)
        m = torch.zeros((ny * nx, 2), device=DEV, dtype=torch.float64)
        for i, w in self.taps:
            for a, g in ((0, dx), (1, dy)):
                m[:, a].index_add_(0, i.reshape(-1), (w * w * g * g).reshape(-1))
        nb = torch.full((ny, nx), 4.0, device=DEV, dtype=torch.float64)
        nb[0] -= 1; nb[-1] -= 1; nb[:, 0] -= 1; nb[:, -1] -= 1
        m = m.view(ny, nx, 2) / (self.P * t.var(unbiased=False)) + (lam / self.P) * nb[..., None]
        self.m = torch.clamp(m / m.mean(), min=1e-3)

    def _u(self, c):
        q = c.reshape(-1, 2)
        u = sum(w[..., None] * q[i] for i, w in self.taps)
        return u[..., 0], u[..., 1]

    def energy(self, c):
        ux, uy = self._u(c)
        e = _ncc_energy(self.R, _bspline(self.T, self.px + ux, self.py + uy)[0])
        reg = ((c[1:] - c[:-1]) ** 2).sum() + ((c[:, 1:] - c[:, :-1]) ** 2).sum()
        return e + 0.5 * self.lam / self.P * reg

    def largest(self, d):
        return math.sqrt(float((d * d).sum(-1).max()))


def _flow(model, c, tol, max_iter):
    """Gradient flow in the model's metric: Armijo backtracking with safeguarded quadratic
    interpolation, Barzilai-Borwein first steps capped at half a pixel."""
    def grad(c):
        c = c.detach().requires_grad_(True)
        return -model.n * torch.autograd.grad(model.energy(c), c)[0] / model.m

    def dot(a, b):
        return float((model.m * a * b).sum()) / model.n

    E, d, tau, d_old, step = float(model.energy(c)), grad(c), 1.0, None, 0.0
    for _ in range(max_iter):
        slope = -dot(d, d)
        if not -slope >= tol * tol:
            break
        if d_old is not None and dot(d_old, d_old - d) > 0:
            tau = step * dot(d_old, d_old - d) / dot(d_old - d, d_old - d)
        tau = min(tau, 0.5 / model.largest(d))
        for _ in range(31):
            Et = float(model.energy(c + tau * d))
            den = Et - E - slope * tau
            q = -slope * tau * tau / (2 * den) if den > 0 else None
            if Et <= E + 0.25 * tau * slope:
                break
            tau = 0.5 * tau if q is None else min(max(q, 0.1 * tau), 0.5 * tau)
        else:
            return c
        c, d_old, step = c + tau * d, d, tau
        tau = 2 * tau if q is None else min(max(q, 0.5 * tau), 4 * tau)
        if not Et < E:
            return c
        E, d = Et, grad(c)
    return c


def _exact_pair(case, s):
    R = [s["R"].double(), _down(s["R"].double())]
    T = [s["T"].double(), _down(s["T"].double())]
    H, W = case["H"], case["W"]
    if case["mode"] == "rigid":
        c = torch.zeros(3, device=DEV, dtype=torch.float64)
        for l in (1, 0):
            c = _flow(_Rigid(R[l], T[l]), c, 3e-5 if l == 0 else 3e-4, case["max_iter"])
            if l:
                c = c * torch.tensor([1.0, 2.0, 2.0], device=DEV, dtype=torch.float64)
        return c
    nx, ny, sp = B.grid_dims(W, H)
    c = torch.zeros((ny, nx, 2), device=DEV, dtype=torch.float64)
    if s["field"] is not None:
        yy, xx = [torch.clamp(torch.arange(n, device=DEV) * sp, max=m - 1) for n, m in ((ny, H), (nx, W))]
        c = s["field"].double()[:, yy][:, :, xx].permute(1, 2, 0) / 2
    for l in (1, 0):
        c = _flow(_Field(R[l], T[l], sp, nx, ny, l, 2.0, c), c, 3e-5 if l == 0 else 3e-4, case["max_iter"])
        c = c * (2.0 if l else 1.0)
    f = _Field(R[0], T[0], sp, nx, ny, 0, 2.0)
    return torch.stack(f._u(c))


def _exact_energy(case, s):
    R, T = s["R"].double(), s["T"].double()
    H, W = case["H"], case["W"]
    if case["mode"] == "rigid":
        m, c = _Rigid(R, T), torch.tensor(s["theta"], device=DEV, dtype=torch.float64)
    else:
        nx, ny, sp = B.grid_dims(W, H, levels=1)
        m, c = _Field(R, T, sp, nx, ny, 0, 2.0), s["grid"].double()
    c = c.requires_grad_(True)
    E = m.energy(c)
    return [E.detach(), torch.autograd.grad(E, c)[0]]


def _exact_warp(case, s):
    N, H, W = case["N"], case["H"], case["W"]
    mean = torch.zeros((H, W), device=DEV, dtype=torch.float64)
    out = torch.empty((N, H, W), device=DEV, dtype=torch.float64) if case["out"] else None
    iy, ix = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(), indexing="ij")
    if case["mode"] == "rigid":
        el = _rigid_prefixes(N - 1, s["seed"])["p"].astype(np.float64)
    else:
        nx, ny, sp = B.grid_dims(W, H)
        f = _Field(s["frames"][0].double(), s["frames"][0].double(), sp, nx, ny, 0, 2.0)
    for k in range(N):
        if k == 0:
            px, py = ix, iy
        elif case["mode"] == "rigid":
            a, gx, gy = (float(v) for v in el[k - 1])
            cx, cy = 0.5 * (W - 1), 0.5 * (H - 1)
            px = math.cos(a) * (ix - cx) - math.sin(a) * (iy - cy) + cx + gx
            py = math.sin(a) * (ix - cx) + math.cos(a) * (iy - cy) + cy + gy
        else:
            ux, uy = f._u(s["grids"][k - 1].double())
            px, py = ix + ux, iy + uy
        v = _bilinear(s["frames"][k].double(), px, py)
        mean += v
        if out is not None:
            out[k] = v
    mean /= N
    return [out, mean] if out is not None else [mean]


def exact(case, seed):
    if case["kind"] not in ("pair", "energy", "warp"):
        return None   # dozens to thousands of registrations: far over the time there is
    s = _inputs(case, seed)
    s["seed"] = seed
    return {"pair": _exact_pair, "energy": _exact_energy, "warp": _exact_warp}[case["kind"]](case, s)
