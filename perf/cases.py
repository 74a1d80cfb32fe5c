"""The calls that users of the library time: inputs, one pass, its work and its value in 64 bits.

A case is a dict of plain values; `listed` gives the fixed ones, `draw` one more of the same
ranges.  The physics cases use seeded layered models (4-8 layers, 1500-4500 m/s, Gaussian
anomalies, Gardner density), Ricker wavelets and receivers on a grid at z = 4 cells, which is how
the package's own synthetic workloads are laid out.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2502_12350_gb300 import cnn, mamute

DEV = "cuda:0"
CERJAN = 0.015


# ------------------------------------------------------------------ the cases

def _physics(name, kind, nx, ny, nz, border, nt, fpeak, **kw):
    """One modelling, gradient or label problem; h and dt keep 4500 m/s inside the CFL bound."""
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, border=border, nt=nt, fpeak=fpeak, h=12.5,
             dt=1e-3, density=False, shots=1, rec_step=2, free_surface=0, interp=0, pml=0, slots=0,
             aperture=0)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: quick-look modelling and the inner loop of a line search on a small
        # model; a few microseconds of work per time step, so launches and set-up count.
        _physics("model_64cube", "model", 64, 64, 64, 16, 500, 15.0, h=10.0, rec_step=8),
        # The bench's headline grid (data generation with variable density), fewer time steps.
        _physics("model_512x512x256_density", "model", 512, 512, 256, 32, 400, 10.0, density=True),
        # A small marine survey: odd sizes, free surface, off-grid positions, four shots a call.
        _physics("model_surface_offgrid_4shots", "model", 203, 151, 97, 20, 300, 12.0, density=True,
                 shots=4, rec_step=3, free_surface=1, interp=1),
        # Modelling with the convolutional PML, the boundary chosen for quiet edges.
        _physics("model_pml_384x384x192", "model", 384, 384, 192, 32, 300, 10.0, density=True, pml=1),
        # FWI's inner call on one shot, every imaging term kept (the automatic storage).
        _physics("gradient_256cube", "gradient", 256, 256, 256, 32, 400, 10.0, h=15.0, dt=1.2e-3),
        # The same call on a memory budget: binomial checkpointing with 16 slots, with density.
        _physics("gradient_checkpoints_181x170x131", "gradient", 181, 170, 131, 16, 300, 10.0, h=15.0,
                 dt=1.2e-3, density=True, slots=16),
        # A survey's gradient: shots with apertures of their own batched into each launch.
        _physics("gradient_8shots_apertures", "gradient", 300, 300, 100, 20, 250, 8.0, h=15.0,
                 dt=1.2e-3, shots=8, aperture=128, rec_step=3),
        # The gradient with the convolutional PML.
        _physics("gradient_pml_192cube", "gradient", 192, 192, 192, 32, 250, 10.0, h=15.0, dt=1.2e-3,
                 pml=1),
        # Gauss-Newton diagonal of a small model (a training label of the preconditioner network).
        _physics("gn_labels_96x80x64", "gn", 96, 80, 64, 20, 500, 8.0, h=15.0, dt=1.2e-3, shots=4,
                 rec_step=18),
        # One hidden layer of the preconditioner network on its training volume: forward with ReLU,
        # weight gradient and input gradient.
        dict(name="conv_layer_80x160x160", kind="conv", nz=80, ny=160, nx=160),
        # Gradient preconditioning of a survey-size gradient (Bessel filter).
        dict(name="smooth_600x600x200_bessel", kind="smooth", nx=600, ny=600, nz=200, mode=1, cells=4.0),
        # Recorded data brought to the inversion's coarser time axis (sinc).
        dict(name="resample_65536x4000_sinc", kind="resample", traces=65536, nt_in=4000, nt_out=1000,
             dt_in=5e-4, dt_out=2e-3, mode=2, adjoint=0),
    ]


def _cost(c):
    """A pass's work in bytes moved or the equivalent of its operations, to order drawn cases."""
    w = work(c)
    return max(w["bytes"] / 6.8e12, w["flops"] / (1.9e15 if c["kind"] == "conv" else 8e13))


def draw(rng):
    """One more case: a kind of the listed ones, sizes over the logarithm of its range."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["model", "model", "model", "gradient", "gradient", "gradient", "gn", "conv",
                       "smooth", "resample"])
    most = max(_cost(c) for c in listed() if c["kind"] == kind)
    while True:
        if kind in ("model", "gradient"):
            grad = kind == "gradient"
            pml = int(rng.random() < 0.3)
            lim = 256 if grad else 512
            nt = size(100, 400 if grad else 600)
            c = _physics("", kind, size(40, lim), size(40, lim), size(32, 256), rng.randrange(8, 37), nt,
                         rng.uniform(8.0, 15.0), h=15.0 if grad else 12.5, dt=1.2e-3 if grad else 1e-3,
                         density=rng.random() < 0.5, shots=rng.choice([1, 1, 2, 3, 5]),
                         rec_step=rng.randrange(2, 7), free_surface=int(rng.random() < 0.25),
                         interp=int(rng.random() < 0.25), pml=pml)
            if grad and not pml and rng.random() < 0.35:
                c["slots"] = rng.randrange(6, 33)
            if rng.random() < 0.3 and min(c["nx"], c["ny"]) >= 80:
                c["aperture"] = rng.randrange(48, 73)
            small = _store_bytes(c) < 3e10
        elif kind == "gn":
            c = _physics("", kind, size(40, 96), size(40, 96), size(32, 64), rng.randrange(8, 21),
                         size(150, 500), 8.0, h=15.0, dt=1.2e-3, density=rng.random() < 0.5,
                         shots=rng.randrange(1, 5), rec_step=rng.randrange(12, 25))
            small = True
        elif kind == "conv":
            c = dict(kind=kind, nz=size(8, 96), ny=size(16, 200), nx=size(16, 200))
            small = True
        elif kind == "smooth":
            c = dict(kind=kind, nx=size(40, 700), ny=size(40, 700), nz=size(20, 300),
                     mode=rng.choice([1, 2]), cells=round(rng.uniform(1.0, 12.0), 2))
            small = True
        else:
            nt_in, q = size(300, 4000), rng.uniform(0.4, 5.0)
            c = dict(kind=kind, traces=size(500, 65536), nt_in=nt_in, nt_out=max(8, int(nt_in / q)),
                     dt_in=5e-4, dt_out=5e-4 * q, mode=rng.choice([1, 2, 2]),
                     adjoint=int(rng.random() < 0.4))
            small = True
        if small and _cost(c) <= most:
            c.pop("name", None)
            return c


# ------------------------------------------------------------------ geometry

def _windows(c):
    """Per shot: source cell (x, y, z) and the model columns (x0, x1, y0, y1) it propagates over."""
    nx, ny, n = c["nx"], c["ny"], c["shots"]
    cols = max(1, int(math.ceil(math.sqrt(n))))
    rows = (n + cols - 1) // cols
    out = []
    for s in range(n):
        i, j = s % cols, s // cols
        sx, sy = int((i + 0.5) * nx / cols), int((j + 0.5) * ny / rows)
        sz = min(8, c["nz"] - 2)
        if not c["aperture"]:
            out.append(((sx, sy, sz), (0, nx, 0, ny)))
            continue
        lx, ly = min(nx, c["aperture"] + (37 * s) % 53), min(ny, c["aperture"] + (23 * s + 11) % 47)
        x0 = max(0, min(nx - lx, sx - lx // 2))
        x0 -= x0 % 4
        y0 = max(0, min(ny - ly, sy - ly // 2))
        out.append(((sx, sy, sz), (x0, x0 + lx, y0, y0 + ly)))
    return out


def _geometry(c, seed):
    """(sources [n][3], receiver offsets, receivers [m][3], apertures or None), metres."""
    rng = np.random.default_rng(seed + 17)
    h, k = c["h"], c["rec_step"]
    src, rec, off, ap = [], [], [0], []
    for (sx, sy, sz), (x0, x1, y0, y1) in _windows(c):
        src.append((sx, sy, sz))
        gx, gy = np.meshgrid(np.arange(x0 + 1, x1 - 1, k), np.arange(y0 + 1, y1 - 1, k), indexing="xy")
        rec.append(np.stack([gx.ravel(), gy.ravel(), np.full(gx.size, 4)], axis=1))
        off.append(off[-1] + gx.size)
        ap.append((x0, x1, y0, y1))
    src, rec = np.array(src, np.float64), np.concatenate(rec).astype(np.float64)
    if c["interp"]:
        src += rng.uniform(0.1, 0.4, src.shape)
        rec += rng.uniform(0.05, 0.45, rec.shape)
    return ((src * h).astype(np.float32), np.array(off, np.int32), (rec * h).astype(np.float32),
            np.array(ap, np.int32) if c["aperture"] else None)


def _ricker(c):
    tau = np.arange(c["nt"]) * c["dt"] - 1.0 / c["fpeak"]
    a = (math.pi * c["fpeak"] * tau) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


def _model(c, seed):
    """(velocity, density or None), float32 [nz][ny][nx] on the GPU."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    rng = np.random.default_rng(seed)
    z = torch.arange(nz, device=DEV, dtype=torch.float32)[:, None, None]
    y = torch.arange(ny, device=DEV, dtype=torch.float32)[None, :, None]
    x = torch.arange(nx, device=DEV, dtype=torch.float32)[None, None, :]
    n = int(rng.integers(4, 9))
    depth = np.sort(rng.uniform(0.05, 0.95, n - 1)) * nz
    slope = rng.uniform(-0.05, 0.05, (n - 1, 2))
    v = np.sort(rng.uniform(1500.0, 4000.0, n))
    width = 0.3 if c["kind"] == "model" else 4.0  # gradients are taken at a smooth model
    vel = torch.full((nz, ny, nx), float(v[0]), device=DEV)
    for k in range(n - 1):
        face = float(depth[k]) + float(slope[k, 0]) * (x - nx / 2) + float(slope[k, 1]) * (y - ny / 2)
        vel += float(v[k + 1] - v[k]) * torch.sigmoid((z - face) / width)
    for _ in range(2):
        amp = float(rng.uniform(-0.1, 0.1))
        cx, cy, cz = (float(q) for q in rng.uniform(0.2, 0.8, 3) * (nx, ny, nz))
        s = 0.12
        e = -0.5 * (((x - cx) / (s * nx)) ** 2 + ((y - cy) / (s * ny)) ** 2 + ((z - cz) / (s * nz)) ** 2)
        vel *= 1.0 + amp * torch.exp(e)
    vel = vel.clamp_(1400.0, 4500.0).contiguous()
    rho = (310.0 * vel.double() ** 0.25).float().contiguous() if c["density"] else None
    return vel, rho


def _observed(c, src, off, rec, seed):
    """Observed traces: direct waves of a slightly different velocity and one weak echo, with the
    1 / (4 pi c^2 r) amplitude that the modelled ones have, [n_rec][nt] on the GPU."""
    rng = np.random.default_rng(seed + 29)
    v = float(rng.uniform(1700.0, 2300.0))
    t = torch.arange(c["nt"], device=DEV, dtype=torch.float32)[None, :] * c["dt"]
    rows = []
    for s in range(len(src)):
        r = torch.from_numpy(rec[off[s]:off[s + 1]]).to(DEV)
        d = (r - torch.from_numpy(src[s]).to(DEV)).norm(dim=1).clamp_min(c["h"])[:, None]
        out = torch.zeros((r.shape[0], c["nt"]), device=DEV)
        for path, amp in ((d, 1.0), (torch.sqrt(d * d + (0.8 * c["nz"] * c["h"]) ** 2), 0.3)):
            a = (math.pi * c["fpeak"] * (t - path / v - 1.0 / c["fpeak"])) ** 2
            out += amp * (1.0 - 2.0 * a) * torch.exp(-a) / (4.0 * math.pi * v * v * path)
        rows.append(out)
    return torch.cat(rows).contiguous()


def _grid(c):
    return mamute.make_grid(c["nx"], c["ny"], c["nz"], c["border"], c["h"], c["dt"], c["nt"],
                            cerjan=CERJAN, free_surface=c["free_surface"], xyz_interp=c["interp"],
                            pml=c["pml"], pml_f0=c["fpeak"])


def _gn_receivers(c):
    """The receiver set that every shot of the label computation records at."""
    k = c["rec_step"]
    gx, gy = np.meshgrid(np.arange(4, c["nx"] - 4, k), np.arange(4, c["ny"] - 4, k), indexing="xy")
    return (np.stack([gx.ravel(), gy.ravel(), np.full(gx.size, 4)], axis=1) * c["h"]).astype(np.float32)


# ------------------------------------------------------------------ the pass

def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV).manual_seed(seed)
    st = {"case": c, "ctx": mamute.Context(0)}
    if c["kind"] in ("model", "gradient", "gn"):
        st["vel"], st["rho"] = _model(c, seed)
        src, off, rec, ap = _geometry(c, seed)
        if c["kind"] == "gn":
            one = _gn_receivers(c)
            rec = np.concatenate([one] * c["shots"])
            off = np.arange(c["shots"] + 1, dtype=np.int32) * len(one)
            st["hdiag"] = torch.empty_like(st["vel"])
        st.update(grid=_grid(c), src=src, off=off, rec=rec, wav=_ricker(c))
        st["opts"] = {} if ap is None else {"aperture": ap}
        if c["kind"] == "model":
            st["seis"] = torch.empty((int(off[-1]), c["nt"]), device=DEV)
        elif c["kind"] == "gradient":
            st["d_obs"] = _observed(c, src, off, rec, seed)
            st["grad"] = torch.empty_like(st["vel"])
            st["opts"]["n_snapshots"] = c["slots"]
    elif c["kind"] == "conv":
        # activations after a ReLU, He-sized weights, a sparse output gradient
        shape = (c["nz"], c["ny"], c["nx"], cnn.C)
        st["x"] = torch.randn(shape, device=DEV, generator=gen).clamp_min_(0).bfloat16()
        st["gy"] = (1e-3 * torch.randn(shape, device=DEV, generator=gen)).bfloat16()
        st["w"] = torch.randn((cnn.TAPS, cnn.C, cnn.C), device=DEV, generator=gen) * (2.0 / (cnn.TAPS * cnn.C)) ** 0.5
        st["bias"] = 0.1 * torch.randn(cnn.C, device=DEV, generator=gen)
        st["lib"] = cnn._bind(st["ctx"].lib)
        st["fwd"], st["bwd"] = (torch.empty((cnn.TAPS, cnn.C, cnn.C), device=DEV, dtype=torch.bfloat16) for _ in range(2))
        st["y"], st["gx"] = (torch.empty(shape, device=DEV, dtype=torch.bfloat16) for _ in range(2))
        st["gw"], st["gb"] = torch.empty_like(st["w"]), torch.empty_like(st["bias"])
        st["ctx"]._check(st["lib"].mamute_conv3d_pack(st["ctx"]._h, _p(st["w"]), _p(st["fwd"]), _p(st["bwd"])))
    elif c["kind"] == "smooth":
        st["inp"] = torch.randn((c["nz"], c["ny"], c["nx"]), device=DEV, generator=gen)
        st["out"] = torch.empty_like(st["inp"])
    else:
        rows, cols = (c["nt_out"], c["nt_in"]) if c["adjoint"] else (c["nt_in"], c["nt_out"])
        st["x"] = torch.randn((c["traces"], rows), device=DEV, generator=gen)
        st["y"] = torch.empty((c["traces"], cols), device=DEV)
    return st


def _p(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    if c["kind"] == "model":
        ctx.model(s["grid"], s["vel"], s["rho"], s["src"], s["wav"], s["off"], s["rec"], s["seis"],
                  **s["opts"])
        return s["seis"]
    if c["kind"] == "gradient":
        J = ctx.gradient(s["grid"], s["vel"], s["rho"], s["src"], s["wav"], s["off"], s["rec"],
                         s["d_obs"], s["grad"], **s["opts"])
        return {"misfit": J, "grad": s["grad"]}
    if c["kind"] == "gn":
        ctx.gn_diagonal(s["grid"], s["vel"], s["rho"], s["src"], s["wav"], s["off"], s["rec"], s["hdiag"])
        return s["hdiag"]
    if c["kind"] == "conv":
        lib, h, dims = s["lib"], ctx._h, (c["nz"], c["ny"], c["nx"])
        ctx._check(lib.mamute_conv3d(h, *dims, _p(s["x"]), _p(s["fwd"]), _p(s["bias"]), 1, None, None, _p(s["y"])))
        ctx._check(lib.mamute_conv3d_wgrad(h, *dims, _p(s["x"]), _p(s["gy"]), _p(s["gw"]), _p(s["gb"])))
        ctx._check(lib.mamute_conv3d(h, *dims, _p(s["gy"]), _p(s["bwd"]), None, 0, _p(s["x"]), None, _p(s["gx"])))
        return {"y": s["y"], "gw": s["gw"], "gb": s["gb"], "gx": s["gx"]}
    if c["kind"] == "smooth":
        ctx.smooth(10.0, c["mode"], s["inp"], s["out"], [10.0 * c["cells"]] * 3)
        return s["out"]
    ctx.resample(s["x"], c["dt_in"], c["nt_out"], c["dt_out"], c["mode"], s["y"], adjoint=bool(c["adjoint"]))
    return s["y"]


# ------------------------------------------------------------------ its work

def _points(c):
    """(padded points, layer points summed over the axes, model points in the windows) of all shots."""
    b = c["border"]
    pad = lay = inner = 0
    for _, (x0, x1, y0, y1) in _windows(c):
        nx, ny, nz = x1 - x0 + 2 * b, y1 - y0 + 2 * b, c["nz"] + 2 * b
        pad += nx * ny * nz
        lay += 2 * b * (ny * nz + nx * nz + nx * ny)
        wx = min(x1 + b, c["nx"]) - max(0, x0 - b)
        wy = min(y1 + b, c["ny"]) - max(0, y0 - b)
        inner += wx * wy * c["nz"]
    return pad, lay, inner


def _store_bytes(c):
    return 0 if c["kind"] != "gradient" or c["slots"] else 4 * c["nt"] * _points(c)[2]


def work(case):
    """Time-stepping paths: per step, both wavefield levels and the coefficients read, one level
    written (and per layer point and axis of the PML two memory variables read and written); the
    gradient's reverse step reads and writes the accumulator, and its imaging terms are written
    once and read once.  Checkpointing is credited with one forward sweep and the recomputed field."""
    c = case
    if c["kind"] in ("model", "gradient", "gn"):
        pad, lay, inner = _points(c)
        nt, step = c["nt"], 20 if c["density"] else 16
        nrec = sum(((x1 - x0 - 2 + c["rec_step"] - 1) // c["rec_step"]) * ((y1 - y0 - 2 + c["rec_step"] - 1) // c["rec_step"])
                   for _, (x0, x1, y0, y1) in _windows(c))
        cells = c["nx"] * c["ny"] * c["nz"] * (2 if c["density"] else 1)
        per = pad * step + (16 * lay if c["pml"] else 0)
        flops = pad * 38 + (40 * lay if c["pml"] else 0)
        if c["kind"] == "model":
            return {"bytes": 4 * cells + nt * per + 4 * nt * nrec, "flops": nt * flops}
        if c["kind"] == "gradient":
            img = 4 * pad if c["slots"] else 8 * inner
            return {"bytes": 4 * cells + nt * (2 * per + 8 * inner + img) + 4 * nt * nrec,
                    "flops": nt * 2 * flops + nt * 2 * inner}
        props = c["shots"] + len(_gn_receivers(c))
        pts = (c["nx"] + 2 * c["border"]) * (c["ny"] + 2 * c["border"]) * (c["nz"] + 2 * c["border"])
        n = c["nx"] * c["ny"] * c["nz"]
        bins = 7.2 * c["fpeak"] * c["nt"] * c["dt"]  # kept bins of a Ricker spectrum above 1e-4 of its peak
        return {"bytes": 4 * cells + 4 * n + nt * props * (pts * step + 8 * n),
                "flops": nt * props * (38 * pts + 4 * bins * n)}
    if c["kind"] == "conv":
        n = c["nz"] * c["ny"] * c["nx"]
        return {"bytes": n * 32 * 7, "flops": 3 * n * 2 * 27 * 256}
    if c["kind"] == "smooth":
        n = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": 8 * n, "flops": 24 * n}
    taps = 1 if c["mode"] == 1 else 16 * max(c["dt_in"], c["dt_out"]) / c["dt_in"]
    return {"bytes": 4 * c["traces"] * (c["nt_in"] + c["nt_out"]), "flops": int(2 * taps * c["traces"] * c["nt_out"])}


# ------------------------------------------------------------------ in 64 bits

C2 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)
C1 = (4.0 / 5.0, -1.0 / 5.0, 4.0 / 105.0, -1.0 / 280.0)


def _shifted(f, axis, out, weights, odd):
    """out += sum_m weights[m] (f(+m) +- f(-m)) along an axis, zero outside."""
    n = f.shape[axis]
    for m, w in enumerate(weights, 1):
        if m >= n:
            break
        out.narrow(axis, 0, n - m).add_(f.narrow(axis, m, n - m), alpha=w)
        out.narrow(axis, m, n - m).add_(f.narrow(axis, 0, n - m), alpha=-w if odd else w)
    return out


def _d2(f, axis):
    return _shifted(f, axis, f * C2[0], C2[1:], False)


def _d1(f, axis):
    return _shifted(f, axis, torch.zeros_like(f), C1, True)


class _Shot:
    """One shot's window in 64 bits: coefficients, profiles, source and receivers."""

    def __init__(self, c, vel, rho, window, src, rec, vmax):
        x0, x1, y0, y1 = window
        b, h, dt = c["border"], float(np.float32(c["h"])), float(np.float32(c["dt"]))
        self.b, self.h, self.dt, self.window = b, h, dt, window
        nx, ny, nz = c["nx"], c["ny"], c["nz"]

        def at(n, start, count, extra=0):
            return (torch.arange(start - extra, start + count + extra, device=DEV) - b).clamp(0, n - 1)

        nxw, nyw, nzw = x1 - x0 + 2 * b, y1 - y0 + 2 * b, nz + 2 * b
        iz, iy, ix = at(nz, 0, nzw), at(ny, y0, nyw), at(nx, x0, nxw)
        cv = vel.double()[iz][:, iy][:, :, ix]
        self.A = (cv * dt / h) ** 2
        self.M = None
        if rho is not None:
            e = [at(nz, 0, nzw, 4), at(ny, y0, nyw, 4), at(nx, x0, nxw, 4)]
            s = rho.double().sqrt()[e[0]][:, e[1]][:, :, e[2]]
            m = sum(_d2(s, a) for a in range(3))[4:-4, 4:-4, 4:-4] / s[4:-4, 4:-4, 4:-4]
            self.M = m * self.A
            del s, m
        self.zs = b if c["free_surface"] else -1
        self.pml = bool(c["pml"])
        alpha = 0.0 if self.pml else float(np.float32(CERJAN))

        def damp(n, low=True):
            i = torch.arange(n, device=DEV, dtype=torch.float64)
            d = torch.clamp(i - (n - 1 - b), min=0)
            if low:
                d = d + torch.clamp(b - i, min=0)
            return torch.exp(-(alpha * d) ** 2)

        gz = damp(nzw, self.zs < 0)
        if self.zs >= 0:
            gz[:self.zs + 1] = 0.0
        self.g = gz[:, None, None] * damp(nyw)[None, :, None] * damp(nxw)[None, None, :]
        if self.pml:
            self.prof = [self._layer(c, nzw, vmax, self.zs < 0, (-1, 1, 1)),
                         self._layer(c, nyw, vmax, True, (1, -1, 1)),
                         self._layer(c, nxw, vmax, True, (1, 1, -1))]
        self.shape = (nzw, nyw, nxw)
        self.src = self._nodes(c, src[None], rho, x0, y0)
        self.rec = self._nodes(c, rec, rho, x0, y0)
        self.inv_h3 = dt * dt / h ** 3

    def _layer(self, c, n, vmax, low, shape):
        b = self.b
        f0 = float(np.float32(c["fpeak"]))
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        dist = torch.clamp(i - (n - 1 - b), min=0)
        if low:
            dist = dist + torch.clamp(b - i, min=0)
        r = dist / max(b, 1)
        d = -3.0 * vmax * math.log(1e-3) / (2.0 * b * self.h) * r * r
        a = torch.where(dist > 0, math.pi * f0 * (1.0 - r), torch.zeros_like(r))
        bb = torch.exp(-(d + a) * self.dt)
        cc = torch.where(d + a > 0, d * (bb - 1.0) / torch.where(d + a > 0, d + a, torch.ones_like(d)), torch.zeros_like(d))
        return bb.reshape(shape), cc.reshape(shape)

    def _nodes(self, c, xyz, rho, x0, y0):
        """(flat node, weight, sqrt(rho), point) of the nodes that the points use."""
        f = torch.from_numpy(np.asarray(xyz, np.float64) / self.h).to(DEV)
        base = torch.floor(f) if c["interp"] else torch.floor(f + 0.5)
        t = f - base if c["interp"] else torch.zeros_like(f)
        nz, ny, nx = c["nz"] + 2 * self.b, self.g.shape[1], self.g.shape[2]
        out = []
        for k in range(8):
            up = torch.tensor([k & 1, (k >> 1) & 1, (k >> 2) & 1], device=DEV, dtype=torch.float64)
            w = torch.where(up > 0, t, 1.0 - t).prod(dim=1)
            node = (base + up).long()
            keep = w != 0
            if self.zs >= 0:
                keep = keep & (node[:, 2] != 0)
            node, w, p = node[keep], w[keep], torch.nonzero(keep).flatten()
            sr = rho.double()[node[:, 2], node[:, 1], node[:, 0]].sqrt() if rho is not None else torch.ones_like(w)
            flat = ((node[:, 2] + self.b) * ny + node[:, 1] + self.b - y0) * nx + node[:, 0] + self.b - x0
            out.append((flat, w, sr, p))
        return [torch.cat(q) for q in zip(*out)]

    def state(self, n):
        return [torch.zeros(self.shape, device=DEV, dtype=torch.float64) for _ in range(n)]

    def laplacian(self, u):
        if self.zs >= 0:
            for m in range(1, 5):
                u[self.zs - m] = -u[self.zs + m]
        out = u * (3.0 * C2[0])
        for a in range(3):
            _shifted(u, a, out, C2[1:], False)
        if self.zs >= 0:
            u[:self.zs + 1] = 0.0
        return out

    def d2z(self, u):
        """Second difference along z with the surface's image planes."""
        if self.zs >= 0:
            for m in range(1, 5):
                u[self.zs - m] = -u[self.zs + m]
        out = _d2(u, 0)
        if self.zs >= 0:
            u[:self.zs + 1] = 0.0
        return out

    def forward(self, s, wn):
        """One step on s = [u, prev, memory variables...]: (new state, the term A lap u - M u)."""
        u = s[0]
        t = self.laplacian(u)
        for a in range(3 if self.pml else 0):
            bb, cc = self.prof[a]
            psi, zeta = s[2 + a], s[5 + a]
            psi.mul_(bb).add_(cc * _d1(u, a))
            dp = _d1(psi, a)
            zeta.mul_(bb).add_(cc * ((self.d2z(u) if a == 0 else _d2(u, a)) + dp))
            t += dp
            t += zeta
        t *= self.A
        if self.M is not None:
            t -= self.M * u
        new = self.g * (2.0 * u + t - self.g * s[1])
        flat, w, sr, _ = self.src
        new.view(-1).index_add_(0, flat, w * self.inv_h3 / sr * wn)
        return [new, u] + s[2:], t

    def sample(self, u, n):
        flat, w, sr, p = self.rec
        return torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, p, w * sr * u.reshape(-1)[flat])

    def reverse(self, s, res):
        """One adjoint step on s = [psi, prev, multipliers...] with the residual row injected."""
        q = s[0]
        extra = None
        for a in range(3 if self.pml else 0):
            bb, cc = self.prof[a]
            pb, zb = s[2 + a], s[5 + a]
            zb += q
            y = cc * zb
            zb *= bb
            pb -= _d1(q + y, a)
            z = cc * pb
            pb *= bb
            e = (self.d2z(y) if a == 0 else _d2(y, a)) - _d1(z, a)
            extra = e if extra is None else extra.add_(e)
        t = self.laplacian(q)
        if extra is not None:
            t += extra
        t *= self.A
        if self.M is not None:
            t -= self.M * q
        new = self.g * (2.0 * q + t - self.g * s[1])
        flat, w, sr, p = self.rec
        gA = self.g.reshape(-1)[flat] * self.A.reshape(-1)[flat] * self.h ** 2
        new.view(-1).index_add_(0, flat, w * gA * sr * res[p])
        return [new, q] + s[2:]


def _shots(c, seed):
    vel, rho = _model(c, seed)
    src, off, rec, _ = _geometry(c, seed)
    vmax = float(vel.max())
    for s, (_, window) in enumerate(_windows(c)):
        yield s, vel, off, rec, _Shot(c, vel, rho, window, src[s], rec[off[s]:off[s + 1]], vmax)


def _exact_model(c, seed):
    out, wav = [], _ricker(c).astype(np.float64)
    for s, _, off, _, S in _shots(c, seed):
        n = int(off[s + 1] - off[s])
        seis = torch.empty((c["nt"], n), device=DEV, dtype=torch.float64)
        st = S.state(8 if S.pml else 2)
        for k in range(c["nt"]):
            st, _ = S.forward(st, float(wav[k]))
            seis[k] = S.sample(st[0], n)
        out.append(seis.T)
    return torch.cat(out)


def _exact_gradient(c, seed):
    """Forward sweep with a state kept every `seg` steps, then each segment's terms made again."""
    wav = _ricker(c).astype(np.float64)
    src, off, rec, _ = _geometry(c, seed)
    d_obs = _observed(c, src, off, rec, seed).double()
    nt, seg, J, grad = c["nt"], 20, 0.0, None
    for s, vel, off, _, S in _shots(c, seed):
        n = int(off[s + 1] - off[s])
        res = torch.empty((nt, n), device=DEV, dtype=torch.float64)
        st, kept = S.state(8 if S.pml else 2), []
        for k in range(nt):
            if k % seg == 0:
                kept.append([f.clone() for f in st])
            st, _ = S.forward(st, float(wav[k]))
            res[k] = S.sample(st[0], n)
        res -= d_obs[off[s]:off[s + 1]].T
        J += 0.5 * float((res * res).sum())
        del st
        adj = S.state(8 if S.pml else 2)
        acc = S.state(1)[0]
        for k0 in range((nt - 1) // seg * seg, -1, -seg):
            st, terms = kept.pop(), []
            for k in range(k0, min(nt, k0 + seg)):
                st, t = S.forward(st, float(wav[k]))
                terms.append(t)
            for k in range(min(nt, k0 + seg) - 1, k0 - 1, -1):
                adj = S.reverse(adj, res[k])
                acc.addcmul_(adj[0], terms.pop())
        if grad is None:
            grad = torch.zeros(vel.shape, device=DEV, dtype=torch.float64)
        b, (x0, x1, y0, y1) = S.b, S.window
        lo = [0, max(0, y0 - b), max(0, x0 - b)]
        hi = [c["nz"], min(c["ny"], y1 + b), min(c["nx"], x1 + b)]
        o = [b, b - y0, b - x0]
        w = acc[lo[0] + o[0]:hi[0] + o[0], lo[1] + o[1]:hi[1] + o[1], lo[2] + o[2]:hi[2] + o[2]]
        grad[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] += w
    dt = float(np.float32(c["dt"]))
    return {"misfit": J, "grad": 2.0 * grad / (vel.double() ** 3 * dt * dt)}


def _exact_gn(c, seed):
    vel, rho = _model(c, seed)
    src, _, _, _ = _geometry(c, seed)
    one, wav, nt = _gn_receivers(c), _ricker(c).astype(np.float64), c["nt"]
    mag = np.abs(np.fft.rfft(wav, 2 * nt))
    bins = np.nonzero(mag >= float(np.float32(1e-4)) * mag.max())[0]
    wts = np.where((bins == 0) | (bins == nt), 1.0, 2.0)
    ph = -2.0 * np.pi * np.outer(bins, np.arange(nt)) / (2 * nt)
    W = torch.from_numpy(np.concatenate([np.cos(ph), np.sin(ph)])).to(DEV)
    nb, b, dt = len(bins), c["border"], float(np.float32(c["dt"]))
    cut = (slice(b, b + c["nz"]), slice(b, b + c["ny"]), slice(b, b + c["nx"]))
    n = vel.numel()
    power = []
    for side in (0, 1):
        P = torch.zeros((nb, n), device=DEV, dtype=torch.float64)
        for k in range(c["shots"] if side == 0 else len(one)):
            S = _Shot(c, vel, rho, (0, c["nx"], 0, c["ny"]), src[min(k, len(src) - 1)], one[k:k + 1] if side else one, 0.0)
            V = torch.empty((nt, n), device=DEV, dtype=torch.float64)
            st = S.state(2)
            for t in range(nt):
                if side == 0:
                    st, term = S.forward(st, float(wav[t]))
                    V[t] = term[cut].reshape(-1)
                else:
                    st = S.reverse(st, torch.full((1,), 1.0 if t == 0 else 0.0, device=DEV, dtype=torch.float64))
                    V[t] = st[0][cut].reshape(-1)
            F = W @ V
            P += F[:nb] ** 2 + F[nb:] ** 2
            del V, F
        power.append(P)
    H = (torch.from_numpy(wts).to(DEV)[:, None] * power[0] * power[1]).sum(0) / (2 * nt)
    v = vel.double()
    # term and impulse response each carry A = c^2 dt^2: dA/dc / A^2 = 2 / (c^3 dt^2)
    return H.reshape(vel.shape) * (2.0 / (v ** 3 * dt * dt)) ** 2


def _taps(x):
    """The 27 shifted views of a zero-padded [D][H][W][16] volume, in (dz, dy, dx) order."""
    D, H, W, _ = x.shape
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    for k in range(27):
        dz, dy, dx = k // 9, (k // 3) % 3, k % 3
        yield k, p[dz:dz + D, dy:dy + H, dx:dx + W].reshape(-1, cnn.C)


def _exact_conv(c, seed):
    st = prepare(c, seed)
    x, gy = st["x"].double(), st["gy"].double()
    w = st["w"].bfloat16().double()
    y = torch.zeros((x[..., 0].numel(), cnn.C), device=DEV, dtype=torch.float64)
    gw = torch.empty((27, cnn.C, cnn.C), device=DEV, dtype=torch.float64)
    g2 = gy.reshape(-1, cnn.C)
    for k, v in _taps(x):
        y += v @ w[k].T
        gw[k] = g2.T @ v
    gx = torch.zeros_like(y)
    for k, v in _taps(gy):
        gx += v @ w[26 - k]
    y = (y + st["bias"].double()).clamp_min(0)
    return {"y": y.reshape(x.shape), "gw": gw, "gb": g2.sum(0),
            "gx": torch.where(x > 0, gx.reshape(x.shape), torch.zeros_like(x))}


def _exact_smooth(c, seed):
    u = prepare(c, seed)["inp"].double()
    lam = []
    for a, n in enumerate((c["nz"], c["ny"], c["nx"])):
        k = torch.arange(n, device=DEV, dtype=torch.float64)
        C = torch.cos(math.pi * k[:, None] * (k[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
        C[0] *= math.sqrt(0.5)
        u = torch.tensordot(C, u, dims=([1], [a])).movedim(0, a)
        l2 = (float(np.float32(10.0 * c["cells"])) / 10.0) ** 2
        lam.append((4.0 * l2 * torch.sin(math.pi * k / (2.0 * n)) ** 2, C))
    lz, ly, lx = lam[0][0][:, None, None], lam[1][0][None, :, None], lam[2][0][None, None, :]
    u = u / (1.0 + lx + ly + lz) if c["mode"] == 1 else u / ((1.0 + lx) * (1.0 + ly) * (1.0 + lz))
    for a in range(3):
        u = torch.tensordot(lam[a][1].T, u, dims=([1], [a])).movedim(0, a)
    return u.contiguous()


def _exact_resample(c, seed):
    x = prepare(c, seed)["x"].double()
    di, do = float(np.float32(c["dt_in"])), float(np.float32(c["dt_out"]))
    m = torch.arange(c["nt_out"], device=DEV, dtype=torch.float64)[:, None]
    n = torch.arange(c["nt_in"], device=DEV, dtype=torch.float64)[None, :]
    if c["mode"] == 1:
        K = (n == torch.floor(m * do / di + 0.5)).double()
    else:
        D = max(di, do)
        u = (m * do - n * di) / D
        K = torch.where(u.abs() < 8, di / D * torch.sinc(u) * 0.5 * (1.0 + torch.cos(math.pi * u / 8)), torch.zeros_like(u))
    return x @ (K if c["adjoint"] else K.T)


def exact(case, seed):
    """What `run` returns in 64 bits, or None where that would take too long."""
    c = case
    if c["kind"] in ("model", "gradient"):
        pad, lay, _ = _points(c)
        seconds = c["nt"] * (pad + (3 * lay if c["pml"] else 0)) * 25 * 24 / 5e12 + c["nt"] * c["shots"] * 6e-4 * (3 if c["pml"] else 1)
        if seconds * (3 if c["kind"] == "gradient" else 1) > 18.0:
            return None
    return {"model": _exact_model, "gradient": _exact_gradient, "gn": _exact_gn, "conv": _exact_conv,
            "smooth": _exact_smooth, "resample": _exact_resample}[c["kind"]](c, seed)
