"""The calls whose speed counts, with their inputs and their values in 64 bits.

Every case is one call (or one training step) through the package's public
entry points at a size of this project's presets, tests or benchmark:

* whole reconstructions of the small and the medium configuration, and a
  batch of uneven orbits (latency, launches, host path);
* the layers of the large ones alone: the shift-variant filter, the
  cone-beam backprojection, their reverse modes, the Gaussian layer on the
  redundancy weight and the Eq. 9 weights.

`exact` restates each call in plain torch FP64: the line sums and their
transpose as products with sparse matrices of Joseph weights, the
backprojection by bilinear sampling of each view.  It assumes what the
generators here make: square pixels and the principal point in the middle of
the detector for every view.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2410_14900_gb300 import api
from paper_2410_14900_gb300.autograd import DefriseClackNet, gauss_smooth

SID, SDD = 750.0, 1200.0   # source to isocentre, source to detector (mm)
DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------- cases
def _case(name, op, orbit, views, rows, cols, pitch, n_mu, n_s, nz, ny, nx, voxel, **more):
    c = dict(name=name, op=op, orbit=orbit, views=views, rows=rows, cols=cols, pitch=pitch,
             n_mu=n_mu, n_s=n_s, ds=pitch, nz=nz, ny=ny, nx=nx, voxel=voxel, batch=1,
             store="f32", kahan=False, relu=False, weights=False)
    c.update(more)
    return c


# the presets' shapes: orbit, views, detector, pitch, planes, volume, voxel
_SMALL = ("circle", 64, 64, 64, 2.0, 180, 64, 64, 64, 64, 2.0)
_MEDIUM = ("sinusoid", 360, 256, 256, 1.2, 360, 256, 256, 256, 256, 0.75)
_LARGE = ("circle_arc", 496, 384, 512, 0.6, 720, 512, 512, 512, 512, 0.375)
_PAPER = ("tilted", 400, 480, 620, 0.616, 360, 785, 128, 512, 512, 0.25)
_STEP = ("sinusoid", 90, 128, 128, 2.4, 180, 128, 128, 128, 128, 1.5)


def listed():
    return [
        # a preview or an inner iteration on the smallest preset: launches and latency
        _case("recon_small", "recon", *_SMALL),
        # a scan of the medium preset, reconstructed as it comes
        _case("recon_medium", "recon", *_MEDIUM),
        # several scans of different protocols in one call (uneven orbits, one launch)
        _case("batch_uneven", "batch", "circle", 203, 264, 304, 1.0, 360, 304, 128, 128, 128, 1.5,
              store="f32x2", batch=4),
        # the filter of a 512^3 scan with orbit-specific weights, in the form that the
        # backprojection reads without a conversion
        _case("filter_large", "filter", *_LARGE, store="f32x2", weights=True),
        # the paper's own detector (rows of 620, 785 planes), g^F kept in 16 bits
        _case("filter_paper", "filter", *_PAPER, store="f16"),
        # the backprojection of a 512^3 scan
        _case("backproject_large", "backproject", *_LARGE, store="f32x2"),
        # the paper's flat volume from 16-bit storage with compensated sums
        _case("backproject_paper", "backproject", *_PAPER, store="bf16", kahan=True),
        # training on the medium preset, batch of 4: the two reverse modes
        _case("backproject_adjoint_train", "backproject_adjoint", *_MEDIUM, batch=4, relu=True),
        _case("filter_adjoint_train", "filter_adjoint", *_MEDIUM, batch=4, weights=True),
        # the Gaussian layer on the learned weight, forward and backward
        _case("smooth_train", "smooth", *_MEDIUM),
        # the analytic weights of an orbit (Eq. 9), once per protocol
        _case("crofton_medium", "crofton", *_MEDIUM),
        # a whole training step (forward and backward) on a coarse grid, batch of 2
        _case("train_step_coarse", "train", *_STEP, batch=2, relu=True, weights=True),
    ]


# the largest listed work of each kind: Joseph steps and voxel updates
_MOST_STEPS, _MOST_UPDATES = 7.0e10, 6.6e10


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["recon", "recon", "filter", "filter", "backproject", "backproject",
                     "backproject_adjoint", "filter_adjoint", "smooth", "crofton", "train",
                     "batch"])
    views = _log_int(rng, 48, 500)
    cols = _log_int(rng, 64, 640)
    rows = max(48, min(480, int(cols * rng.uniform(0.6, 1.0))))
    if rng.random() < 0.5:              # detectors usually have rows of whole vectors
        cols = max(64, cols // 8 * 8)
    store = rng.choice(["f32", "f32x2", "bf16", "f16"])
    batch = 1
    if op == "batch":                   # takes rows of whole 16-byte units
        cols, views, batch = min(320, max(64, cols // 8 * 8)), min(views, 240), rng.randint(2, 5)
        rows = min(rows, cols)
    if op in ("backproject_adjoint", "filter_adjoint", "train"):
        store, batch = "f32", rng.randint(1, 4)
    if op == "train":
        views, cols = min(views, 180), min(cols, 200)
        rows = min(rows, cols)
    pitch = 0.6 * 512 / cols
    n_mu = rng.choice([90, 180, 200, 360, 361, 720]) if cols > 128 else rng.choice([90, 135, 180])
    n_s = max(48, int(cols * rng.uniform(0.9, 1.25)))
    n = _log_int(rng, 48, 512)
    nz = max(32, int(n * rng.uniform(0.25, 1.0)))
    voxel = 192.0 / n if rng.random() < 0.7 else 140.0 / n
    if op == "train":
        n, nz = min(n, 160), min(nz, 160)
        voxel = 192.0 / n
    if op == "batch":
        n, nz = min(n, 192), min(nz, 192)
        voxel = 192.0 / n
    if op == "smooth":
        n_mu, n_s, views = rng.randint(90, 400), rng.randint(64, 400), min(views, 360)
    if op == "crofton":
        n_mu, n_s, views = min(n_mu, 360), min(n_s, 300), min(views, 360)
    orbit = rng.choice(["circle", "sinusoid", "tilted", "circle_arc"])
    if op in ("crofton", "train"):
        orbit = rng.choice(["circle", "sinusoid", "tilted"])
    # no more than the largest listed case
    steps = 0.9 * views * batch * n_mu * rows * cols
    if steps > _MOST_STEPS:
        views = max(48, int(views * _MOST_STEPS / steps))
    upd = 1.0 * views * batch * nz * n * n
    if upd > _MOST_UPDATES / 2 and op not in ("filter", "filter_adjoint", "smooth", "crofton"):
        views = max(48, int(views * _MOST_UPDATES / 2 / upd))
    c = _case("", op, orbit, views, rows, cols, pitch, n_mu, n_s, nz, n, n, voxel, store=store,
              batch=batch, kahan=store in ("bf16", "f16"),
              relu=op in ("backproject_adjoint", "train") or rng.random() < 0.2,
              weights=op in ("filter_adjoint", "train") or rng.random() < 0.5)
    if op in ("filter", "recon") and rng.random() < 0.25:
        c["ds"] = pitch * rng.choice([0.8, 1.25, 1.5])
    del c["name"]
    return c


# ------------------------------------------------------------------ geometry
def _orbit(kind, V):
    """Sources [V, 3], tangents a'(lambda) dlambda [V, 3] and whether it is closed."""
    t = 2.0 * math.pi * np.arange(V) / V
    one = np.ones_like(t)
    if kind == "circle":
        a = np.stack([SID * np.cos(t), SID * np.sin(t), 0 * one], 1)
        v = np.stack([-SID * np.sin(t), SID * np.cos(t), 0 * one], 1) * (2 * math.pi / V)
        return a, v, True
    if kind == "sinusoid":              # axial offset 40 mm sin(2 phi)
        a = np.stack([SID * np.cos(t), SID * np.sin(t), 40.0 * np.sin(2 * t)], 1)
        v = np.stack([-SID * np.sin(t), SID * np.cos(t), 80.0 * np.cos(2 * t)], 1)
        return a, v * (2 * math.pi / V), True
    if kind == "tilted":                # the paper's sphere-surface sinusoid, 20 degrees, f = 5
        th, tm, f = t - math.pi, math.radians(20.0), 5.0
        ph, dp = tm * np.cos(f * th), -tm * f * np.sin(f * th)
        a = SID * np.stack([np.cos(ph) * np.cos(th), np.cos(ph) * np.sin(th), np.sin(ph)], 1)
        v = SID * np.stack([-np.sin(ph) * dp * np.cos(th) - np.cos(ph) * np.sin(th),
                            -np.sin(ph) * dp * np.sin(th) + np.cos(ph) * np.cos(th),
                            np.cos(ph) * dp], 1)
        return a, v * (2 * math.pi / V), True
    if kind == "circle_arc":            # circle plus a perpendicular 60-degree arc
        nc = max(2, round(V * 360 / 496))
        na = max(2, V - nc)
        a, v, _ = _orbit("circle", V - na)
        half = math.radians(30.0)
        psi = np.linspace(-half, half, na)
        a2 = SID * np.stack([np.cos(psi), 0 * psi, np.sin(psi)], 1)
        v2 = SID * np.stack([-np.sin(psi), 0 * psi, np.cos(psi)], 1) * (2 * half / (na - 1))
        return np.concatenate([a, a2]), np.concatenate([v, v2]), False
    raise ValueError(kind)


def _frames(a):
    lz = a / np.linalg.norm(a, axis=1, keepdims=True)
    ly = np.array([[0.0, 0.0, 1.0]]) - lz[:, 2:3] * lz
    ly /= np.linalg.norm(ly, axis=1, keepdims=True)
    return np.cross(ly, lz), ly, lz


def _matrices(c, a):
    lx, ly, lz = _frames(a)
    f, cu, cv = SDD / c["pitch"], (c["cols"] - 1) / 2.0, (c["rows"] - 1) / 2.0
    A = np.stack([f * lx - cu * lz, f * ly - cv * lz, -lz], 1)
    return np.concatenate([A, -np.einsum("vij,vj->vi", A, a)[:, :, None]], 2)


def _geometry(c):
    a, v, closed = _orbit(c["orbit"], c["views"])
    desc = dict(n_views=c["views"], det_rows=c["rows"], det_cols=c["cols"], n_mu=c["n_mu"],
                n_s=c["n_s"], pitch=c["pitch"], ds=c["ds"], vol_x=c["nx"], vol_y=c["ny"],
                vol_z=c["nz"], voxel=(c["voxel"],) * 3, closed_orbit=int(closed))
    return api.Geometry(desc, _matrices(c, a), v)


def _problems(c):
    """The problems of a batch: other orbits, view counts, detectors and volumes."""
    kinds = ["circle", "sinusoid", "circle_arc", "tilted"]
    out = []
    for k in range(c["batch"]):
        s = 1.0 - 0.17 * k
        cols = max(64, int(c["cols"] * s) // 8 * 8)
        n = max(32, int(c["nx"] * (1.0 - 0.11 * k)))
        p = c["pitch"] * c["cols"] / cols
        out.append(dict(c, orbit=kinds[(kinds.index(c["orbit"]) + k) % 4], batch=1,
                        views=max(40, c["views"] - 31 * k), rows=max(48, int(c["rows"] * s)),
                        cols=cols, pitch=p, ds=p, n_s=cols, nx=n, ny=n,
                        nz=max(32, int(c["nz"] * (1.0 - 0.11 * k))),
                        voxel=c["voxel"] * c["nx"] / n))
    return out


# -------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _blobs(c, seed, n=16):
    """Seeded ellipsoids inside the field of view: centre, semi-axes, rotation, density."""
    rng = np.random.default_rng(int(seed))
    e = 0.5 * min(c["cols"] * c["pitch"], c["rows"] * c["pitch"], c["n_s"] * c["ds"])
    r = SID * math.sin(math.atan(e / SDD))
    out = []
    for _ in range(n):
        ax = rng.uniform(0.05, 0.3, 3) * r
        d = rng.normal(size=3)
        ctr = d / np.linalg.norm(d) * max(0.95 * r - ax.max(), 0.0) * rng.uniform() ** (1 / 3)
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        out.append((ctr, (q / ax).T, rng.uniform(0.0, 1.0)))
    return out


def _projections(c, seed):
    """Line integrals of a seeded phantom, [V, H, W] FP32, with counting noise."""
    a, _, _ = _orbit(c["orbit"], c["views"])
    lx, ly, lz = (torch.tensor(t, device=DEV, dtype=torch.float32) for t in _frames(a))
    H, W, p = c["rows"], c["cols"], c["pitch"]
    x = (torch.arange(W, device=DEV) - (W - 1) / 2.0) * p
    y = (torch.arange(H, device=DEV) - (H - 1) / 2.0) * p
    n = torch.sqrt(SDD ** 2 + x[None, :] ** 2 + y[:, None] ** 2)
    g = torch.zeros((c["views"], H, W), device=DEV)
    for ctr, T, rho in _blobs(c, seed):
        Tt = torch.tensor(T, device=DEV, dtype=torch.float32)
        y0 = torch.tensor((a - ctr) @ T.T, device=DEV, dtype=torch.float32)   # [V, 3]
        tx, ty, tz = lx @ Tt.T, ly @ Tt.T, lz @ Tt.T
        for v0 in range(0, c["views"], 64):
            s = slice(v0, min(v0 + 64, c["views"]))
            dd = bd = 0.0
            for k in range(3):
                d = (x[None, None, :] * tx[s, k, None, None] + y[None, :, None]
                     * ty[s, k, None, None] - SDD * tz[s, k, None, None]) / n
                dd = dd + d * d
                bd = bd + d * y0[s, k, None, None]
            disc = bd * bd - dd * ((y0[s] ** 2).sum(1)[:, None, None] - 1.0)
            g[s] += (2.0 * rho) * torch.sqrt(disc.clamp_(min=0.0)) / dd
    g += 0.02 * torch.sqrt(g) * torch.randn(g.shape, device=DEV, generator=_gen(seed))
    return g.contiguous()


def _filtered(c, seed):
    """What filtered projections look like: rows of a phantom's projections
    through a ramp filter, at the scale of g^F."""
    g = _projections(c, seed)
    n = 2 * c["cols"]
    ramp = torch.fft.rfftfreq(n, device=DEV)
    for v0 in range(0, c["views"], 64):
        s = slice(v0, min(v0 + 64, c["views"]))
        g[s] = torch.fft.irfft(torch.fft.rfft(g[s], n=n) * ramp, n=n)[..., :c["cols"]]
    return (g * (2000.0 / c["views"])).contiguous()


def _volume(c, seed):
    """A phantom on the voxel grid, [Z, Y, X] FP32."""
    ax = [(torch.arange(n, device=DEV) - (n - 1) / 2.0) * c["voxel"]
          for n in (c["nz"], c["ny"], c["nx"])]
    out = torch.zeros((c["nz"], c["ny"], c["nx"]), device=DEV)
    for ctr, T, rho in _blobs(c, seed):
        T = torch.tensor(T, dtype=torch.float32).tolist()
        q = 0.0
        for k in range(3):
            q = q + (T[k][0] * (ax[2] - ctr[0])[None, None, :] + T[k][1]
                     * (ax[1] - ctr[1])[None, :, None] + T[k][2] * (ax[0] - ctr[2])[:, None, None]) ** 2
        out += rho * (q <= 1.0)
    return out


def _weights(c, seed):
    """A learned redundancy weight: smooth about 1/2, with a little texture."""
    m = torch.arange(c["n_mu"], device=DEV)[None, :, None] / c["n_mu"]
    k = torch.arange(c["n_s"], device=DEV)[None, None, :] / c["n_s"]
    v = torch.arange(c["views"], device=DEV)[:, None, None] / c["views"]
    w = 0.5 + 0.2 * torch.sin(6.28 * (v + 2 * m)) * torch.cos(3.14 * k)
    return w + 0.02 * torch.randn(w.shape, device=DEV, generator=_gen(seed + 7))


def _many(f, c, seed):
    return torch.stack([f(c, 1000 * seed + b) for b in range(c["batch"])])


def _stored(c, gF):
    """g^F [B, V, H, W] FP32 in a storage form: (tensor, scale or None)."""
    s = c["store"]
    if s == "f32":
        return gF, None
    if s == "bf16":
        return gF.to(torch.bfloat16), None
    if s == "f32x2":
        right = F.pad(gF, (0, 1))[..., 1:]
        return torch.stack([gF, right - gF], -1).contiguous(), None
    _, e = torch.frexp(gF.abs().amax((2, 3)))
    scale = torch.ldexp(torch.ones_like(gF[:, :, 0, 0]), e - 15)
    return (gF / scale[..., None, None]).to(torch.float16), scale


def _inputs(c, seed):
    """The arrays of a case, on the GPU, from the seed alone."""
    op = c["op"]
    d = {}
    if op == "batch":
        d["g"] = [_projections(q, 1000 * seed + k) for k, q in enumerate(_problems(c))]
    elif op in ("recon", "filter"):
        d["g"] = _many(_projections, c, seed)
        d["W"] = _weights(c, seed) if c["weights"] else None
    elif op == "backproject":
        d["gF"], d["scale"] = _stored(c, _many(_filtered, c, seed))
    elif op == "backproject_adjoint":
        f = _many(_volume, c, seed)
        noise = torch.randn(f.shape, device=DEV, generator=_gen(seed))
        d["vol"] = (f + 0.05 * noise).clamp_(min=0.0)      # a reconstruction behind the ReLU
        d["grad"] = (d["vol"] - f) * (2.0 / f.numel())
    elif op == "filter_adjoint":
        d["grad"] = _many(_filtered, c, seed) * 1e-6
        shp = (c["batch"], c["views"], c["n_mu"], c["n_s"])
        S = torch.randn(shp, device=DEV, generator=_gen(seed + 3))
        k = (torch.arange(c["n_s"], device=DEV) + 0.5) / c["n_s"] - 0.5
        S *= 30.0 * torch.exp(-8.0 * k * k)
        S[..., -1] = 0.0
        d["S"] = S
        d["W"] = _weights(c, seed)
    elif op == "smooth":
        d["W"] = torch.rand((c["views"], c["n_mu"], c["n_s"]), device=DEV, generator=_gen(seed))
        d["grad"] = torch.randn(d["W"].shape, device=DEV, generator=_gen(seed + 1)) * 1e-4
    elif op == "crofton":               # the orbit is the input: scans start at other angles
        d["turn"] = float(np.random.default_rng(seed).uniform(0.0, 2.0 * math.pi))
    elif op == "train":
        d["g"] = _many(_projections, c, seed)
        d["ref"] = _many(_volume, c, seed)
        d["W"] = _weights(c, seed)
    return d


def _turned(a, phi):
    R = np.array([[math.cos(phi), -math.sin(phi), 0.0], [math.sin(phi), math.cos(phi), 0.0],
                  [0.0, 0.0, 1.0]])
    return a @ R.T


# ------------------------------------------------------------- prepare / run
def prepare(case, seed):
    c = case
    d = _inputs(c, seed)
    op = c["op"]
    d["c"] = c
    if op == "batch":
        probs = _problems(c)
        d["geoms"] = [_geometry(q) for q in probs]
        d["vols"] = [torch.empty((q["nz"], q["ny"], q["nx"]), device=DEV) for q in probs]
        d["batch"] = api.Batch(d["geoms"], c["store"], kahan=c["kahan"], relu=c["relu"])
        return d
    if op == "smooth":
        d["W"].requires_grad_(True)
        return d
    if op == "crofton":
        a, v, closed = _orbit(c["orbit"], c["views"])
        a, v = _turned(a, d["turn"]), _turned(v, d["turn"])
        desc = dict(n_views=c["views"], det_rows=c["rows"], det_cols=c["cols"], n_mu=c["n_mu"],
                    n_s=c["n_s"], pitch=c["pitch"], ds=c["ds"], vol_x=c["nx"], vol_y=c["ny"],
                    vol_z=c["nz"], voxel=(c["voxel"],) * 3, closed_orbit=int(closed))
        d["geom"] = api.Geometry(desc, _matrices(c, a), v)
        return d
    d["geom"] = _geometry(c)
    if op == "train":
        net = DefriseClackNet(d["geom"], relu=c["relu"], device=DEV, smooth=(8.0, 24))
        with torch.no_grad():
            net.W.copy_(d.pop("W"))
        d["net"] = net
    return d


def run(state):
    d, c = state, state["c"]
    op = c["op"]
    if op == "recon":
        return api.reconstruct(d["geom"], d["g"], d["W"], c["store"], kahan=c["kahan"],
                               relu=c["relu"])
    if op == "filter":
        gF, scale = api.dc_filter(d["geom"], d["g"], d["W"], c["store"])
        return [gF, scale]
    if op == "backproject":
        return api.dc_backproject(d["geom"], d["gF"], d["scale"], kahan=c["kahan"],
                                  relu=c["relu"])
    if op == "backproject_adjoint":
        return api.dc_backproject_adjoint(d["geom"], d["grad"], d["vol"] if c["relu"] else None)
    if op == "filter_adjoint":
        return list(api.dc_filter_adjoint(d["geom"], d["grad"], None, d["W"], S=d["S"]))
    if op == "smooth":
        out = gauss_smooth(d["W"], 20.0, 60)
        grad, = torch.autograd.grad(out, d["W"], d["grad"])
        return [out.detach(), grad]
    if op == "crofton":
        return api.dc_crofton_weights(d["geom"])
    if op == "batch":
        d["batch"].run(d["g"], d["vols"])
        return d["vols"]
    if op == "train":
        vol = d["net"](d["g"])
        loss = torch.mean((vol - d["ref"]) ** 2)
        grad, = torch.autograd.grad(loss, d["net"].W)
        return {"loss": loss.detach(), "vol": vol.detach(), "grad_W": grad}
    raise ValueError(op)


# ---------------------------------------------------------------------- work
def _filter_flops(c):
    """A Joseph step: position, fraction, lerp, sum (7); a pixel-angle pair:
    position, fraction, two hat weights, two taps (13)."""
    px = 1.0 * c["batch"] * c["views"] * c["n_mu"] * c["rows"] * c["cols"]
    cover = min(1.0, c["n_s"] * c["ds"] / (c["pitch"] * math.hypot(c["rows"], c["cols"])) * 1.2)
    return 7.0 * 0.9 * px * cover * c["pitch"] / c["ds"], 13.0 * px


def work(case):
    c = case
    op = c["op"]
    if op == "batch":
        w = [work(dict(q, op="recon")) for q in _problems(c)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    img = 1.0 * c["batch"] * c["views"] * c["rows"] * c["cols"]
    vox = 1.0 * c["batch"] * c["nz"] * c["ny"] * c["nx"]
    wts = 1.0 * c["views"] * c["n_mu"] * c["n_s"]
    ls, bp2 = _filter_flops(c)
    px = {"f32": 4, "f32x2": 8, "bf16": 2, "f16": 2}[c["store"]]
    upd = 18.0 * vox * c["views"]
    if op == "recon":
        return {"bytes": 4 * img + 4 * vox + (4 * wts if c["weights"] else 0),
                "flops": ls + bp2 + upd}
    if op == "filter":
        return {"bytes": (4 + px) * img + (4 * wts if c["weights"] else 0), "flops": ls + bp2}
    if op == "backproject":
        return {"bytes": px * img + 4 * vox, "flops": upd}
    if op == "backproject_adjoint":
        return {"bytes": 4 * img + 4 * vox * (2 if c["relu"] else 1), "flops": upd}
    if op == "filter_adjoint":
        return {"bytes": 8 * img + 4 * wts * (c["batch"] + 2), "flops": ls + bp2}
    if op == "smooth":
        return {"bytes": 16 * wts, "flops": 2 * 2 * 2 * 121 * wts}
    if op == "crofton":                 # the sign test of every pair of views
        return {"bytes": 4 * wts, "flops": 6 * wts * c["views"]}
    if op == "train":
        return {"bytes": 4 * img + 8 * vox + 8 * wts, "flops": 2 * (ls + upd) + bp2}
    raise ValueError(op)


# --------------------------------------------------------------------- exact
def _angles(c):
    for m in range(c["n_mu"]):
        mu = m * math.pi / c["n_mu"]
        yield m, math.cos(mu), math.sin(mu), 4 * m <= c["n_mu"] or 4 * m >= 3 * c["n_mu"]


def _joseph(c, co, si, by_rows):
    """The Joseph weights of one angle: (line, pixel, weight), the scale p/|cos| included."""
    H, W, p = c["rows"], c["cols"], c["pitch"]
    cu, cv = (W - 1) / 2.0, (H - 1) / 2.0
    s = (torch.arange(c["n_s"], device=DEV, dtype=F64) - 0.5 * (c["n_s"] - 1)) * c["ds"]
    if by_rows:
        q = torch.arange(H, device=DEV)
        x = (s[:, None] - (q[None, :].to(F64) - cv) * (p * si)) / (co * p) + cu
        n, step, along, scale = W, 1, W, p / abs(co)
    else:
        q = torch.arange(W, device=DEV)
        x = (s[:, None] - (q[None, :].to(F64) - cu) * (p * co)) / (si * p) + cv
        n, step, along, scale = H, W, 1, p / abs(si)
    j = torch.floor(x)
    t = x - j
    j = j.long()
    k = torch.arange(c["n_s"], device=DEV)[:, None].expand_as(j)
    px = q[None, :] * along + j * step
    a, b = (j >= 0) & (j < n), (j >= -1) & (j < n - 1)
    return (torch.cat([k[a], k[b]]), torch.cat([px[a], px[b] + step]),
            torch.cat([(1.0 - t)[a], t[b]]) * scale)


def _times(rows, cols, vals, n_rows, x):
    """A sparse matrix given by its entries, times x."""
    order = torch.argsort(rows, stable=True)
    crow = torch.zeros(n_rows + 1, device=DEV, dtype=torch.long)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=n_rows), 0)
    A = torch.sparse_csr_tensor(crow, cols[order], vals[order], (n_rows, x.shape[0]))
    return A @ x


def _radon(c, img):
    """[N, H, W] images -> [n_mu, n_s, N] line sums."""
    x = img.reshape(img.shape[0], -1).t().contiguous()
    out = torch.empty((c["n_mu"], c["n_s"], x.shape[1]), device=DEV, dtype=F64)
    for m, co, si, br in _angles(c):
        k, px, w = _joseph(c, co, si, br)
        out[m] = _times(k, px, w, c["n_s"], x)
    return out


def _radon_T(c, R):
    """The transpose: [n_mu, n_s, N] -> [N, H, W]."""
    out = torch.zeros((c["rows"] * c["cols"], R.shape[2]), device=DEV, dtype=F64)
    for m, co, si, br in _angles(c):
        k, px, w = _joseph(c, co, si, br)
        out += _times(px, k, w, out.shape[0], R[m])
    return out.t().reshape(-1, c["rows"], c["cols"])


def _radii2(c):
    x = (torch.arange(c["cols"], device=DEV, dtype=F64) - (c["cols"] - 1) / 2.0) * c["pitch"]
    y = (torch.arange(c["rows"], device=DEV, dtype=F64) - (c["rows"] - 1) / 2.0) * c["pitch"]
    return x[None, :] ** 2 + y[:, None] ** 2 + SDD ** 2


def _half_grid(c):
    k = torch.arange(c["n_s"], device=DEV, dtype=F64)
    return (k - 0.5 * (c["n_s"] - 1) + 0.5) * c["ds"]


def _thetas(c, a):
    """Unit normals of the planes: components along l_x, l_y, l_z, [n_mu, n_s] each."""
    mu = torch.arange(c["n_mu"], device=DEV, dtype=F64)[:, None] * (math.pi / c["n_mu"])
    s = _half_grid(c)[None, :]
    n = torch.sqrt(s * s + SDD ** 2)
    return SDD * torch.cos(mu) / n, SDD * torch.sin(mu) / n, s / n


def _redundancy(c, a, v):
    """K [n_mu, n_s, V] of Eq. 10 (0 at the last entry)."""
    lx, ly, lz = _frames(a)
    tx, ty, tz = _thetas(c, a)
    dots = [torch.tensor((v * t).sum(1), device=DEV) for t in (lx, ly, lz)]
    vt = (tx[..., None] * dots[0] + ty[..., None] * dots[1] + tz[..., None] * dots[2]).abs_()
    n = torch.sqrt(_half_grid(c) ** 2 + SDD ** 2)
    K = vt.mul_(-1.0 / (4 * math.pi ** 2)).div_(n[None, :, None])
    K[:, -1] = 0.0
    return K


def _w_sino(c):
    return ((_half_grid(c) ** 2 + SDD ** 2) / SDD ** 2)[None, :, None]


def _shift_down(x):
    return torch.cat([torch.zeros_like(x[:, :1]), x[:, :-1]], 1)


def _filter64(c, g, W):
    """Eq. 11 on one batch item g [V, H, W]."""
    a, v, _ = _orbit(c["orbit"], c["views"])
    R = _radon(c, g * (SDD / torch.sqrt(_radii2(c))))
    S = torch.zeros_like(R)
    S[:, :-1] = (R[:, 1:] - R[:, :-1]) / c["ds"]
    del R
    S *= _w_sino(c)
    S *= _redundancy(c, a, v)
    S = S * (0.5 if W is None else W.permute(1, 2, 0))
    S = (S - _shift_down(S)) * (math.pi / c["n_mu"] / c["pitch"] ** 2)
    return _radon_T(c, S) * _radii2(c)


def _filter_adjoint64(c, G, S, W):
    """dL/dg and one batch item's dL/dW for G = dL/dg^F [V, H, W]."""
    a, v, _ = _orbit(c["orbit"], c["views"])
    P = _radon(c, G * _radii2(c)) * (math.pi / c["n_mu"] * c["ds"] / c["pitch"] ** 2)
    Q = torch.zeros_like(P)
    Q[:, :-1] = (P[:, :-1] - P[:, 1:]) / c["ds"]
    del P
    Q *= _redundancy(c, a, v)
    gW = (Q * S.permute(1, 2, 0)).permute(2, 0, 1)
    y = Q * W.permute(1, 2, 0) * _w_sino(c)
    gR = (_shift_down(y) - y) / c["ds"]
    gg = _radon_T(c, gR) * (SDD / torch.sqrt(_radii2(c)))
    return gg, gW


def _slabs(c, a, i, lx, ly, lz, B):
    """(z range, sampling grid, 1/|X - a|^2) of view i, slab by slab."""
    ax = [(torch.arange(n, device=DEV, dtype=F64) - (n - 1) / 2.0) * c["voxel"]
          for n in (c["nx"], c["ny"], c["nz"])]
    X, Y, Z = (t - a[i][k] for k, t in enumerate(ax))
    f, H, W = SDD / c["pitch"], c["rows"], c["cols"]
    depth = max(1, int(3e7 / (c["nx"] * c["ny"] * max(1, B // 2))))

    def dot(t, z):
        return (t[0] * X)[None, None, :] + (t[1] * Y)[None, :, None] + (t[2] * z)[:, None, None]

    for z0 in range(0, c["nz"], depth):
        z = Z[z0:z0 + depth]
        dep = -dot(lz[i], z)
        u = dot(lx[i], z) / dep * (2.0 * f / (W - 1))       # the principal point is the middle
        v = dot(ly[i], z) / dep * (2.0 * f / (H - 1))
        r2 = (X * X)[None, None, :] + (Y * Y)[None, :, None] + (z * z)[:, None, None]
        n = z.shape[0]
        grid = torch.stack([u, v], -1).reshape(1, n * c["ny"], c["nx"], 2)
        yield slice(z0, z0 + n), grid, 1.0 / r2


def _backproject64(c, gF):
    """Eq. 5: gF [B, V, H, W] -> [B, Z, Y, X]."""
    a, _, _ = _orbit(c["orbit"], c["views"])
    lx, ly, lz = _frames(a)
    B = gF.shape[0]
    out = torch.zeros((B, c["nz"], c["ny"], c["nx"]), device=DEV, dtype=F64)
    for i in range(c["views"]):
        for zs, grid, w in _slabs(c, a, i, lx, ly, lz, B):
            val = F.grid_sample(gF[:, i][None].to(F64), grid, align_corners=True)
            out[:, zs] += val.reshape(B, -1, c["ny"], c["nx"]) * w
    return out


def _backproject_adjoint64(c, grad):
    a, _, _ = _orbit(c["orbit"], c["views"])
    lx, ly, lz = _frames(a)
    B = grad.shape[0]
    out = torch.empty((B, c["views"], c["rows"], c["cols"]), device=DEV, dtype=F64)
    for i in range(c["views"]):
        img = torch.zeros((1, B, c["rows"], c["cols"]), device=DEV, dtype=F64, requires_grad=True)
        acc = torch.zeros_like(img)
        for zs, grid, w in _slabs(c, a, i, lx, ly, lz, B):
            val = F.grid_sample(img, grid, align_corners=True)
            acc = acc + torch.autograd.grad(val, img, (grad[:, zs] * w).reshape(val.shape))[0]
        out[:, i] = acc[0].detach()
    return out


def _smooth64(x, sigma, radius, transpose=False):
    """The Gaussian layer along mu and s of [V, n_mu, n_s] (mirror ends, unit
    sum, the last s entry untouched), or its transpose, as matrix products."""
    def matrix(n):
        t = torch.arange(-radius, radius + 1, device=DEV, dtype=F64)
        w = torch.exp(-0.5 * (t / sigma) ** 2)
        w /= w.sum()
        p = torch.arange(n, device=DEV)[:, None] + t.long()[None, :]
        T = max(1, 2 * (n - 1))
        p = p % T
        p = torch.where(p < n, p, T - p) if n > 1 else torch.zeros_like(p)
        A = torch.zeros((n, n), device=DEV, dtype=F64)
        A.scatter_add_(1, p, w[None, :].expand(n, -1).contiguous())
        return A.t() if transpose else A

    out = x.clone()
    y = torch.matmul(x[..., :-1], matrix(x.shape[2] - 1).t())
    out[..., :-1] = torch.matmul(matrix(x.shape[1]), y)
    return out


def _crofton64(c, phi):
    """Eq. 9 with m = 2 on a closed orbit (no taper there)."""
    a, v, _ = _orbit(c["orbit"], c["views"])
    a, v = _turned(a, phi), _turned(v, phi)
    lx, ly, lz = _frames(a)
    tx, ty, tz = _thetas(c, a)
    V = c["views"]
    A, Vd = torch.tensor(a, device=DEV), torch.tensor(v, device=DEV)
    out = torch.zeros((V, c["n_mu"], c["n_s"]), device=DEV, dtype=F64)
    ns = c["n_s"] - 1
    for i in range(V):
        th = sum(t[..., None] * torch.tensor(l[i], device=DEV)
                 for t, l in ((tx, lx), (ty, ly), (tz, lz)))[:, :ns].reshape(-1, 3)
        own = (th @ Vd[i]) ** 2
        f = th @ (A - A[i]).t()                              # [planes, V]
        j0, j1 = torch.arange(V, device=DEV), (torch.arange(V, device=DEV) + 1) % V
        keep = (j0 != i) & (j1 != i)
        f1 = f[:, j1]
        p, e = torch.nonzero(((f < 0) != (f1 < 0)) & keep, as_tuple=True)
        t = f[p, e] / (f[p, e] - f1[p, e])
        vt = Vd[e] + t[:, None] * (Vd[j1[e]] - Vd[e])
        s = own.clone().index_add_(0, p, (vt * th[p]).sum(1) ** 2)
        out[i, :, :ns] = torch.where(own > 0, own / s, torch.zeros_like(s)).reshape(-1, ns)
    return out


def _relu(c, f):
    return f.clamp(min=0.0) if c["relu"] else f


def _pairs(gF):
    return torch.stack([gF, F.pad(gF, (0, 1))[..., 1:] - gF], -1)


@torch.no_grad()
def exact(case, seed):
    c = case
    op = c["op"]
    d = _inputs(c, seed)
    if op == "batch":
        return [_relu(q, _backproject64(q, _filter64(q, g.to(F64), None)[None])[0])
                for q, g in zip(_problems(c), d["g"])]
    if op == "recon":
        W = None if d["W"] is None else d["W"].to(F64)
        gF = torch.stack([_filter64(c, g.to(F64), W) for g in d["g"]])
        return _relu(c, _backproject64(c, gF))
    if op == "filter":
        W = None if d["W"] is None else d["W"].to(F64)
        gF = torch.stack([_filter64(c, g.to(F64), W) for g in d["g"]])
        if c["store"] == "f32x2":
            return [_pairs(gF), None]
        if c["store"] == "f16":
            _, e = torch.frexp(gF.abs().amax((2, 3)))
            scale = torch.ldexp(torch.ones_like(gF[:, :, 0, 0]), e - 15)
            return [gF / scale[..., None, None], scale]
        return [gF, None]
    if op == "backproject":
        gF = d["gF"]
        if c["store"] == "f32x2":
            gF = gF[..., 0]
        elif c["store"] == "f16":
            gF = gF.to(F64) * d["scale"].to(F64)[..., None, None]
        return _relu(c, _backproject64(c, gF))
    if op == "backproject_adjoint":
        grad = d["grad"].to(F64)
        if c["relu"]:
            grad = grad * (d["vol"] > 0)
        with torch.enable_grad():
            return _backproject_adjoint64(c, grad)
    if op == "filter_adjoint":
        W, gW, gg = d["W"].to(F64), 0.0, []
        for G, S in zip(d["grad"], d["S"]):
            x, y = _filter_adjoint64(c, G.to(F64), S.to(F64), W)
            gg.append(x)
            gW = gW + y
        return [torch.stack(gg), gW]
    if op == "smooth":
        return [_smooth64(d["W"].to(F64), 20.0, 60),
                _smooth64(d["grad"].to(F64), 20.0, 60, transpose=True)]
    if op == "crofton":
        return _crofton64(c, d["turn"])
    if op == "train":
        W = _smooth64(d["W"].to(F64), 8.0, 24)
        a, _, _ = _orbit(c["orbit"], c["views"])
        g, ref = d["g"].to(F64), d["ref"].to(F64)
        vol = _relu(c, _backproject64(c, torch.stack([_filter64(c, x, W) for x in g])))
        loss = torch.mean((vol - ref) ** 2)
        gv = (vol - ref) * (2.0 / vol.numel())
        if c["relu"]:
            gv = gv * (vol > 0)
        with torch.enable_grad():
            gF = _backproject_adjoint64(c, gv)
        gW = 0.0
        for x, G in zip(g, gF):
            R = _radon(c, x * (SDD / torch.sqrt(_radii2(c))))
            S = torch.zeros_like(R)
            S[:, :-1] = (R[:, 1:] - R[:, :-1]) / c["ds"]
            S = (S * _w_sino(c)).permute(2, 0, 1)
            gW = gW + _filter_adjoint64(c, G, S, W)[1]
        return {"loss": loss, "vol": vol, "grad_W": _smooth64(gW, 8.0, 24, transpose=True)}
    return None
