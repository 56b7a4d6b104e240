"""Performance cases of the framework: what its users run, at the sizes they run it.

A case is one call (or one short, fixed sequence of calls) of the public Python API on a
stated geometry. `listed()` names the standing cases, `draw()` gives further ones of the
same ranges, `prepare()` makes what a program holds before the call, `run()` makes the
call, `work()` says what it cannot do without, and `exact()` computes the same results
with plain torch in 64 bits.

Inputs are synthetic: phantoms of random ellipsoids (attenuation 0 to 0.04 /mm, as in soft
tissue and bone) with a little noise, as an iterate of the reconstruction carries, and scans
of such phantoms in closed form (chords through ellipsoids) with Poisson noise.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1008_2042_gb300 as cb
from paper_1008_2042_gb300 import autograd

SAD, SDD = 1000.0, 1500.0  # source to axis and source to imager, mm
MU = 5e-4                  # threshold of the shrinkage
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}

# Scan geometries: voxels, voxel size (mm), imager pixels, pitch (mm), views
SMALL = dict(nx=64, ny=64, nz=16, dx=1.0, dy=1.0, dz=1.0, nu=128, nv=32, du=0.8, dv=0.8, u_off=0.0, v_off=0.0, views=40)
MID = dict(nx=256, ny=256, nz=64, dx=1.0, dy=1.0, dz=1.0, nu=256, nv=192, du=1.5, dv=1.5, u_off=0.0, v_off=0.0, views=60)
PAPER = dict(nx=512, ny=512, nz=70, dx=0.5, dy=0.5, dz=2.5, nu=512, nv=384, du=0.776, dv=0.776, u_off=0.0, v_off=0.0,
             views=40)
# odd sizes on every axis, anisotropic voxels, an imager shifted by a quarter of a pixel
RAGGED = dict(nx=211, ny=197, nz=51, dx=0.9, dy=1.1, dz=1.7, nu=243, nv=157, du=1.3, dv=1.1, u_off=0.325, v_off=0.275,
              views=37)


def listed():
    return [
        # a small scan from start to end: latency of many short launches
        dict(name="recon_small", op="recon", levels=1, iters="20", storage="f32", **SMALL),
        # the reconstruction of a clinical-size scan with the fast protocol, 5/10/15 iterations
        # on three grids: the workload that the framework is built for
        dict(name="recon_paper", op="recon", levels=3, iters="5,10,15", storage="f32", **PAPER),
        # a request of the medium class with 16-bit iteration vectors
        dict(name="recon_mid_f16", op="recon", levels=3, iters="5,10,15", storage="f16", **MID),
        # P and its adjoint on the small scan: the smallest operator calls
        dict(name="pair_small", op="pair", storage="f32", **SMALL),
        # one forward projection at clinical size (simulating a scan, a user's own iteration)
        dict(name="project_paper", op="project", storage="f32", **PAPER),
        # one exact backprojection at clinical size
        dict(name="backproject_paper", op="backproject", storage="f32", **PAPER),
        # P to 16-bit projections and the adjoint of such a stack, sizes ragged on every axis
        dict(name="pair_ragged_f16", op="pair", storage="f16", **RAGGED),
        # a training step through the differentiable projector: batch of 8, forward and backward
        dict(name="gradient_batch8", op="gradient", batch=8, **MID),
        # the frame transform's coefficients of a clinical-size volume, for users who keep them
        dict(name="analyze_paper", op="analyze", storage="f32", nx=512, ny=512, nz=70),
        # shrinkage and synthesis of such coefficients
        dict(name="synthesize_paper", op="synthesize", storage="f32", nx=512, ny=512, nz=70),
        # both transforms with coefficients kept in 16 bits
        dict(name="frame_pair_bf16", op="frame_pair", storage="bf16", nx=256, ny=256, nz=64),
        # the regularisation step in one pass (denoising a clinical-size volume)
        dict(name="shrink_paper", op="shrink", nx=512, ny=512, nz=70),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_geometry(rng, cap):
    """A scan of 24..512 voxels across, 8..120 views, whose trace steps (views x imager columns x
    voxels crossed x slabs) stay below cap."""
    while True:
        nx = _log_int(rng, 24, 512)
        ny = max(16, min(512, int(nx * rng.uniform(0.8, 1.2))))
        nz = max(6, int(min(nx, ny) * rng.uniform(0.12, 0.3)))
        dx = min(rng.uniform(0.5, 2.0), 260.0 / max(nx, ny))
        dy = dx * rng.choice([1.0, 1.0, rng.uniform(0.8, 1.25)])
        dz = min(dx * rng.uniform(1.0, 4.0), 200.0 / nz)
        du, dv = 1.5 * dx * rng.uniform(0.7, 1.3), 1.5 * dx * rng.uniform(0.7, 1.5)
        nu = max(16, int(1.5 * nx * dx / du * rng.uniform(0.8, 1.4)))
        nv = max(8, int(1.5 * nz * dz / dv * rng.uniform(0.8, 1.4)))
        views = _log_int(rng, 8, 120)
        if nu > 768 or nv > 768 or views * nu * (nx + ny) * nz > cap:
            continue
        # an odd imager is shifted by a quarter of a pixel: its central ray would lie in a voxel plane
        return dict(nx=nx, ny=ny, nz=nz, dx=dx, dy=dy, dz=dz, nu=nu, nv=nv, du=du, dv=dv,
                    u_off=0.25 * du if nu % 2 else 0.0, v_off=0.25 * dv if nv % 2 else 0.0, views=views)


def draw(rng):
    op = rng.choice(["recon", "recon", "project", "backproject", "pair", "gradient", "analyze", "synthesize", "frame_pair",
                     "shrink"])
    paper = PAPER["views"] * PAPER["nu"] * (PAPER["nx"] + PAPER["ny"]) * PAPER["nz"]
    if op == "recon":
        levels = rng.randint(1, 3)
        iters = [rng.randint(2, 6) * (k + 1) for k in range(levels)]
        return dict(op=op, levels=levels, iters=",".join(map(str, iters)), storage=rng.choice(["f32", "f32", "f16"]),
                    **_draw_geometry(rng, 12 * paper / sum(iters)))
    if op in ("project", "backproject", "pair"):
        return dict(op=op, storage=rng.choice(["f32", "f32", "bf16", "f16"]), **_draw_geometry(rng, 2 * paper))
    if op == "gradient":
        batch = rng.randint(1, 8)
        return dict(op=op, batch=batch, **_draw_geometry(rng, paper / batch))
    nx = _log_int(rng, 24, 512)
    ny = max(16, min(512, int(nx * rng.uniform(0.8, 1.2))))
    nz = max(6, int(min(nx, ny) * rng.uniform(0.12, 0.4)))
    case = dict(op=op, nx=nx, ny=ny, nz=min(nz, 128))
    if op != "shrink":
        case["storage"] = rng.choice(["f32", "bf16", "f16"])
    return case


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------

def _device():
    return torch.device("cuda")


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _angles(c):
    return 2.0 * np.pi * np.arange(c["views"]) / c["views"]


def _ellipsoids(c, seed, n=12):
    """(cx, cy, cz, ax, ay, az, phi, value) of a body and n - 1 ellipsoids inside it, whose values add."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    hx, hy, hz = (0.5 * c[a] * c[d] for a, d in (("nx", "dx"), ("ny", "dy"), ("nz", "dz")))
    out = [(0.0, 0.0, 0.0, 0.85 * hx, 0.65 * hy, 1.3 * hz, 0.0, 0.02)]
    for _ in range(n - 1):
        r, a = 0.55 * math.sqrt(rng.uniform()), rng.uniform(0.0, 2.0 * math.pi)
        out.append((r * hx * math.cos(a), 0.7 * r * hy * math.sin(a), rng.uniform(-0.6, 0.6) * hz,
                    rng.uniform(0.04, 0.25) * hx, rng.uniform(0.04, 0.2) * hy, rng.uniform(0.15, 0.8) * hz,
                    rng.uniform(0.0, math.pi), rng.uniform(-0.006, 0.02)))
    return out


def _volume(c, seed):
    """The phantom on the grid with a little noise, float32 (nz, ny, nx)."""
    g = {"dx": 1.0, "dy": 1.0, "dz": 1.0, **c}
    x, y, z = ((torch.arange(g[n], device=_device(), dtype=torch.float32) + (0.5 - 0.5 * g[n])) * g[d]
               for n, d in (("nx", "dx"), ("ny", "dy"), ("nz", "dz")))
    f = torch.zeros((g["nz"], g["ny"], g["nx"]), device=_device())
    for cx, cy, cz, ax, ay, az, phi, val in _ellipsoids(g, seed):
        xs, ys, (co, si) = x[None, :] - cx, y[:, None] - cy, (math.cos(phi), math.sin(phi))
        plane = ((xs * co + ys * si) / ax) ** 2 + ((ys * co - xs * si) / ay) ** 2
        f += ((plane[None] + ((z - cz) / az)[:, None, None] ** 2) <= 1.0) * val
    f += 1e-3 * torch.randn(f.shape, device=_device(), generator=_generator(seed))
    return f.contiguous()


def _scan(c, seed, photons=5e4):
    """Line integrals of the phantom in closed form with Poisson noise, float32 (views, nv, nu)."""
    dev, d64 = _device(), torch.float64
    t = torch.as_tensor(_angles(c), device=dev, dtype=d64)
    u = c["u_off"] + (torch.arange(c["nu"], device=dev, dtype=d64) - 0.5 * (c["nu"] - 1)) * c["du"]
    v = c["v_off"] + (torch.arange(c["nv"], device=dev, dtype=d64) - 0.5 * (c["nv"] - 1)) * c["dv"]
    co, si = torch.cos(t)[:, None], torch.sin(t)[:, None]
    sx, sy = SAD * co, SAD * si                                  # source (views, 1)
    dx, dy = -SDD * co - u * si, -SDD * si + u * co              # source to pixel (views, nu)
    p = torch.zeros((c["views"], c["nv"], c["nu"]), device=dev, dtype=d64)
    for cx, cy, cz, ax, ay, az, phi, val in _ellipsoids(c, seed):
        cp, sp = math.cos(phi), math.sin(phi)
        ox, oy = ((sx - cx) * cp + (sy - cy) * sp) / ax, ((sy - cy) * cp - (sx - cx) * sp) / ay
        ex, ey = (dx * cp + dy * sp) / ax, (dy * cp - dx * sp) / ay
        ez, oz = (v / az)[None, :, None], -cz / az
        a = (ex * ex + ey * ey)[:, None, :] + ez * ez
        b = (ox * ex + oy * ey)[:, None, :] + oz * ez
        cc = (ox * ox + oy * oy - 1.0)[:, None, :] + oz * oz
        p += val * 2.0 * torch.sqrt(torch.clamp(b * b - a * cc, min=0.0)) / a
    length = torch.sqrt((dx * dx + dy * dy)[:, None, :] + (v * v)[None, :, None])
    counts = torch.poisson(photons * torch.exp(-p * length), generator=_generator(seed))
    return (-torch.log(torch.clamp(counts, min=1.0) / photons)).to(torch.float32).contiguous()


def _iters(c):
    return [int(v) for v in c["iters"].split(",")]


def prepare(case, seed):
    c, op = case, case["op"]
    s = {"case": c}
    if op in ("analyze", "shrink", "frame_pair"):
        s["f"] = _volume(c, seed)
    elif op == "synthesize":
        s["alpha"] = _analysis(_volume(c, seed)).to(DTYPES[c["storage"]]).contiguous()
    else:
        # the scan's geometry handle: made once, kept by the program
        s["geom"] = cb.Geometry(nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=c["dx"], dy=c["dy"], dz=c["dz"], nu=c["nu"],
                                nv=c["nv"], du=c["du"], dv=c["dv"], u_off=c["u_off"], v_off=c["v_off"], sad=SAD, sdd=SDD,
                                n_views=c["views"])
        if op in ("project", "pair"):
            s["f"] = _volume(c, seed)
        if op in ("recon", "backproject", "pair"):
            s["y"] = _scan(c, seed + 1000).to(DTYPES[c["storage"]] if op != "recon" else torch.float32)
        if op == "gradient":
            s["f"] = torch.stack([_volume(c, seed + 17 * b) for b in range(c["batch"])]).requires_grad_(True)
            s["y"] = torch.stack([_scan(c, seed + 17 * b + 5) for b in range(c["batch"])])
    return s


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "recon":
        return cb.reconstruct(state["geom"], state["y"], MU, c["levels"], _iters(c), storage=c["storage"])
    if op == "project":
        return cb.project(state["geom"], state["f"], dtype=c["storage"])
    if op == "backproject":
        return cb.backproject(state["geom"], state["y"])
    if op == "pair":
        return (cb.project(state["geom"], state["f"], dtype=c["storage"]), cb.backproject(state["geom"], state["y"]))
    if op == "gradient":
        f = state["f"]
        f.grad = None
        p = autograd.project(state["geom"], f)
        r = p - state["y"]
        loss = 0.5 * (r * r).sum()
        loss.backward()
        return {"projections": p.detach(), "gradient": f.grad}
    if op == "analyze":
        return cb.tf_analyze(state["f"], dtype=c["storage"])
    if op == "synthesize":
        return cb.tf_synthesize_shrink(state["alpha"], MU)
    if op == "frame_pair":
        alpha = cb.tf_analyze(state["f"], dtype=c["storage"])
        return alpha, cb.tf_synthesize_shrink(alpha, MU)
    return cb.tf_shrink(state["f"], MU)


# ---------------------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------------------

def _updates(c):
    """Voxels crossed, summed over all rays (the non-zeros of P), estimated on up to 8 views."""
    ks = np.unique(np.linspace(0, c["views"] - 1, min(8, c["views"])).astype(int))
    t = _angles(c)[ks][:, None, None]
    u = (c["u_off"] + (np.arange(c["nu"]) - 0.5 * (c["nu"] - 1)) * c["du"])[None, None, :]
    v = (c["v_off"] + (np.arange(c["nv"]) - 0.5 * (c["nv"] - 1)) * c["dv"])[None, :, None]
    s = (SAD * np.cos(t), SAD * np.sin(t), np.zeros_like(t))
    d = (-SDD * np.cos(t) - u * np.sin(t), -SDD * np.sin(t) + u * np.cos(t), v)
    lo, hi, rate = 0.0, 1.0, 0.0
    for o, e, n, h in zip(s, d, (c["nx"], c["ny"], c["nz"]), (c["dx"], c["dy"], c["dz"])):
        e = np.where(np.abs(e) < 1e-9, 1e-9, e)
        a, b = (-0.5 * n * h - o) / e, (0.5 * n * h - o) / e
        lo, hi = np.maximum(lo, np.minimum(a, b)), np.minimum(hi, np.maximum(a, b))
        rate = rate + np.abs(e) / h
    return float(np.where(hi > lo, (hi - lo) * rate + 1.0, 0.0).sum()) * c["views"] / len(ks)


def _level(c, k):
    s = 2 ** k
    return {**c, **{n: -(-c[n] // s) for n in ("nx", "ny", "nz")}, **{d: c[d] * s for d in ("dx", "dy", "dz")}}


def work(case):
    c, op = case, case["op"]
    n = c["nx"] * c["ny"] * c["nz"]
    size = 4 if c.get("storage", "f32") == "f32" else 2
    triple = 6  # operations of one 3-tap filter triple; 13 triples per voxel and direction
    if op == "analyze":
        return {"bytes": 4 * n + 27 * size * n, "flops": 13 * triple * n}
    if op == "synthesize":
        return {"bytes": 4 * n + 27 * size * n, "flops": (13 * triple + 80) * n}
    if op == "frame_pair":
        return {"bytes": 8 * n + 2 * 27 * size * n, "flops": (26 * triple + 80) * n}
    if op == "shrink":
        return {"bytes": 8 * n, "flops": (26 * triple + 80) * n}
    m = c["views"] * c["nu"] * c["nv"]
    if op == "recon":
        # per iteration: four projections, three backprojections (three CGLS updates), the shrinkage
        flops = 0.0
        for k, it in enumerate(reversed(_iters(c))):
            lc = _level(c, k)
            flops += it * (7 * 2.0 * _updates(lc) + (26 * triple + 80 + 20) * lc["nx"] * lc["ny"] * lc["nz"])
        return {"bytes": 4 * m + 4 * n, "flops": flops}
    updates = 2.0 * _updates(c)
    if op in ("project", "backproject"):
        return {"bytes": 4 * n + size * m, "flops": updates}
    if op == "pair":
        return {"bytes": 2 * (4 * n + size * m), "flops": 2 * updates}
    return {"bytes": c["batch"] * (8 * n + 12 * m), "flops": 2 * c["batch"] * updates}


# ---------------------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------------------

_H = ((0.25, 0.5, 0.25), (math.sqrt(2.0) / 4.0, 0.0, -math.sqrt(2.0) / 4.0), (-0.25, 0.5, -0.25))  # taps at -1, 0, +1


def _filter(f, taps, dim, adjoint):
    s = -1 if adjoint else 1  # analysis: sum_k h(k) f(x - k); synthesis: sum_k h(k) a(x + k)
    out = taps[0] * torch.roll(f, -s, dim) + taps[2] * torch.roll(f, s, dim)
    return out if taps[1] == 0.0 else out + taps[1] * f


def _analysis(f):
    """(27, nz, ny, nx), channel l + 3 m + 9 n: filter l along x, m along y, n along z."""
    out = torch.empty((27,) + tuple(f.shape), dtype=f.dtype, device=f.device)
    for n in range(3):
        fz = _filter(f, _H[n], 0, False)
        for m in range(3):
            fy = _filter(fz, _H[m], 1, False)
            for l in range(3):
                out[l + 3 * m + 9 * n] = _filter(fy, _H[l], 2, False)
    return out


def _synthesis(alpha, mu):
    a = alpha.to(torch.float64)
    norm = torch.sqrt((a[1:] * a[1:]).sum(0))
    mu = float(np.float32(mu))  # the threshold that the entry point takes
    scale = torch.where(norm > mu, 1.0 - mu / torch.where(norm > mu, norm, torch.ones_like(norm)), torch.zeros_like(norm))
    f = torch.zeros_like(norm)
    for n in range(3):
        for m in range(3):
            for l in range(3):
                ch = l + 3 * m + 9 * n
                t = a[ch] * scale if ch else a[0]
                f += _filter(_filter(_filter(t, _H[l], 2, True), _H[m], 1, True), _H[n], 0, True)
    return torch.clamp(f, min=0.0)


class _Exact:
    """P and P^T in 64 bits: the transverse (x, y) trace of every (view, imager column) by sorting its plane
    crossings; along z the integral over a segment from the antiderivative of the voxel column (P) or of
    the row sums below a slab plane (P^T)."""

    def __init__(self, c):
        dev, d64 = _device(), torch.float64
        self.c, self.tc = c, SAD / SDD
        u = c["u_off"] + (torch.arange(c["nu"], device=dev, dtype=d64) - 0.5 * (c["nu"] - 1)) * c["du"]
        self.v = c["v_off"] + (torch.arange(c["nv"], device=dev, dtype=d64) - 0.5 * (c["nv"] - 1)) * c["dv"]
        t = torch.as_tensor(_angles(c), device=dev, dtype=d64)[:, None]
        co, si = torch.cos(t), torch.sin(t)
        self.dx, self.dy = (-SDD * co - u * si).reshape(-1), (-SDD * si + u * co).reshape(-1)
        self.qx, self.qy = (-self.tc * u * si + 0.0 * co).reshape(-1), (self.tc * u * co + 0.0 * si).reshape(-1)
        self.len = torch.sqrt((self.dx ** 2 + self.dy ** 2)[:, None] + (self.v ** 2)[None, :])  # (columns, nv)

    def _trace(self, sel):
        """tau of the segment boundaries (sorted) and the voxel column of every segment, for some columns."""
        c = self.c
        dx, dy, qx, qy = (a[sel][:, None] for a in (self.dx, self.dy, self.qx, self.qy))
        planes = [(torch.arange(c[n] + 1, device=dx.device, dtype=dx.dtype) - 0.5 * c[n]) * c[d]
                  for n, d in (("nx", "dx"), ("ny", "dy"))]
        tx, ty = (planes[0] - qx) / dx, (planes[1] - qy) / dy
        lo = torch.maximum(tx.amin(1), ty.amin(1))[:, None].clamp(min=-self.tc)
        hi = torch.minimum(tx.amax(1), ty.amax(1))[:, None].clamp(max=1.0 - self.tc)
        hi = torch.maximum(lo, hi)
        tau = torch.sort(torch.minimum(torch.maximum(torch.cat([tx, ty], 1), lo), hi), 1).values
        mid = 0.5 * (tau[:, 1:] + tau[:, :-1])
        ix = torch.floor((qx + mid * dx) / c["dx"] + 0.5 * c["nx"]).clamp(0, c["nx"] - 1).long()
        iy = torch.floor((qy + mid * dy) / c["dy"] + 0.5 * c["ny"]).clamp(0, c["ny"] - 1).long()
        return tau, iy * c["nx"] + ix

    def _chunks(self, inner):
        n, steps = self.dx.numel(), self.c["nx"] + self.c["ny"] + 2
        per = max(1, int(1.2e8 // (steps * inner)))
        return [slice(i, min(n, i + per)) for i in range(0, n, per)]

    def project(self, f):
        c = self.c
        col = f.to(torch.float64).reshape(c["nz"], -1).t()  # (columns of voxels, nz)
        cum = torch.zeros((col.shape[0], c["nz"] + 1), dtype=col.dtype, device=col.device)
        torch.cumsum(col * c["dz"], 1, out=cum[:, 1:])
        cum = cum.reshape(-1)
        out = torch.empty_like(self.len)
        v = self.v[None, None, :]

        def upto(base, tau):  # integral of the voxel column from its bottom to the ray's height at tau
            z = (v * (self.tc + tau[:, :, None]) / c["dz"] + 0.5 * c["nz"]).clamp(0.0, float(c["nz"]))
            k = torch.floor(z).clamp(max=c["nz"] - 1)
            at = base + k.long()
            low = cum[at]
            return low + (z - k) * (cum[at + 1] - low)

        for sel in self._chunks(c["nv"]):
            tau, which = self._trace(sel)
            base = (which * (c["nz"] + 1))[:, :, None]
            out[sel] = ((upto(base, tau[:, 1:]) - upto(base, tau[:, :-1])).sum(1) / self.v) * self.len[sel]
        return out.reshape(c["views"], c["nu"], c["nv"]).transpose(1, 2)

    def backproject(self, g):
        c = self.c
        w = g.to(torch.float64).transpose(1, 2).reshape(-1, c["nv"]) * self.len
        zero = torch.zeros((w.shape[0], 1), dtype=w.dtype, device=w.device)
        below = torch.cat([zero, torch.cumsum(w, 1)], 1)           # sum of the rows below row m
        tilt = torch.cat([zero, torch.cumsum(w / self.v, 1)], 1)
        z = ((torch.arange(c["nz"] + 1, device=w.device, dtype=w.dtype) - 0.5 * c["nz"]) * c["dz"])[None, None, :]
        out = torch.zeros((c["nx"] * c["ny"], c["nz"]), dtype=w.dtype, device=w.device)
        first = float(self.v[0])
        for sel in self._chunks(c["nz"] + 1):
            tau, which = self._trace(sel)
            s = self.tc + tau[:, :, None]
            m = torch.ceil((z / s - first) / c["dv"]).clamp(0, c["nv"]).long()  # rows below plane z at s
            row = torch.arange(sel.start, sel.stop, device=w.device)[:, None, None] * (c["nv"] + 1) + m
            a = s * below.reshape(-1)[row] - z * tilt.reshape(-1)[row]  # antiderivative in s of that sum
            i = a[:, 1:] - a[:, :-1]
            out.index_add_(0, which.reshape(-1), (i[:, :, 1:] - i[:, :, :-1]).reshape(-1, c["nz"]))
        return out.t().reshape(c["nz"], c["ny"], c["nx"]).contiguous()


def _exact_recon(c, y):
    """Algorithm A2 on one grid: three CGLS updates from the momentum point, shrinkage, momentum."""
    e, y = _Exact(c), y.to(torch.float64)
    f = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=y.device)
    x, t = f, 1.0
    for _ in range(_iters(c)[0]):
        r = y - e.project(x)
        s = e.backproject(r)
        p, gamma = s, (s * s).sum()
        for l in range(3):
            q = e.project(p)
            a = gamma / (q * q).sum()
            x = x + a * p
            if l == 2:
                break
            r = r - a * q
            s = e.backproject(r)
            new = (s * s).sum()
            p, gamma = s + (new / gamma) * p, new
        fn = _synthesis(_analysis(x), MU)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        x, f, t = fn + ((t - 1.0) / tn) * (fn - f), fn, tn
    return f


def exact(case, seed):
    c, op = case, case["op"]
    if op == "recon":
        steps = sum(_iters(c)) * 7 * c["views"] * c["nu"] * (c["nx"] + c["ny"]) * (c["nv"] + c["nz"])
        if c["levels"] > 1 or c["storage"] != "f32" or steps > 3e10:
            return None  # too long, or a result of 16-bit vectors
        return _exact_recon(c, _scan(c, seed + 1000))
    if op in ("project", "backproject", "pair"):
        e, out = _Exact(c), []
        if op != "backproject":
            out.append(e.project(_volume(c, seed)))
        if op != "project":
            out.append(e.backproject(_scan(c, seed + 1000).to(DTYPES[c["storage"]])))
        return out[0] if len(out) == 1 else tuple(out)
    if op == "gradient":
        e, p, g = _Exact(c), [], []
        for b in range(c["batch"]):
            p.append(e.project(_volume(c, seed + 17 * b)))
            g.append(e.backproject(p[-1] - _scan(c, seed + 17 * b + 5)))
        return {"projections": torch.stack(p), "gradient": torch.stack(g)}
    if op == "analyze":
        return _analysis(_volume(c, seed).to(torch.float64))
    if op == "synthesize":
        return _synthesis(_analysis(_volume(c, seed)).to(DTYPES[c["storage"]]), MU)
    if op == "frame_pair":
        return _analysis(_volume(c, seed).to(torch.float64)), None  # the second reads rounded coefficients
    return _synthesis(_analysis(_volume(c, seed).to(torch.float64)), MU)
