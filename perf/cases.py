"""Work that programs built on this library have it do, as cases to time.

Each case goes through the package's public entry points, from the smallest
map to slices of the production lattice.  A case is a dict of plain values:
`kind` names the path, the other values its sizes.

  direct      one small map in FP64 by direct sum: create, shoot, read out
  map         one small mixed-precision map: create, shoot, mu, light curves
  step        a paper-scale map with the autotuned grid, host lenses to curves
  shard       a slice of the 1e13-ray production lattice on a kept field
  fold        the Table-1 fold field, kept and autotuned: clear, shoot, mu
  build       field creation at a given grid, and the trace of listed rays
  batch       many uneven maps replayed as one graph: mu, curves
  nearfar     the FP64 near/far mode on a kept field
  grad        one step of a gradient descent on a lens field (cloud in cell)
  curve_loss  the gradient of a light-curve loss through both autograd functions
  curves      light curves of extended sources from a map, and their transpose
  peaks       peak identification and statistics of a count map
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2308_14278_gb300 as ml
from paper_2308_14278_gb300 import autograd, inputs

MEAN_MASS = inputs.lognormal_mean(0.3, 0.5)
EDGES = np.concatenate([[0.0], np.geomspace(0.02, 45.0, 24)])


def listed():
    return [
        # The smallest problem: 100 lenses, a 2000 x 2000 ray grid, a 256 x 256
        # map, FP64 direct sum (the reference precision).
        {"name": "direct-small", "kind": "direct", "lenses": 100, "rays_x": 2000, "rays_y": 2000,
         "nx": 256, "ny": 256},
        # An interactive call: about 160 lenses and 1.8e6 rays, from the lens
        # arrays to mu and two light curves.  Latency and launches count.
        {"name": "map-small", "kind": "map", "kappa_star": 0.05, "nx": 200, "ny": 150, "n_av": 60.0,
         "tracks": 2, "samples": 500},
        # The paper-scale map: 13,000 lenses, 1e11 rays, 8192 x 8192, autotuned.
        {"name": "paper-step", "kind": "step", "lenses": 13000, "rays": 1e11, "nx": 8192, "ny": 8192},
        # One shard (1e11 consecutive rays) of the full production map: 13,000
        # lenses, 1e13 rays, 16384 x 16384, at a given grid.
        {"name": "production-shard", "kind": "shard", "lenses": 13000, "rays": 1e13, "slice": 1e11,
         "nx": 16384, "ny": 16384, "l2x": 40, "l2y": 20},
        # The Table-1 fold field at 1e11 rays, 2048 x 10240, autotuned.
        {"name": "fold-shoot", "kind": "fold", "rays": 1e11, "nx": 2048, "ny": 10240},
        # Its creation at the grid a tuned run reports, and 4096 traced rays.
        {"name": "fold-build", "kind": "build", "field": "fold", "lenses": 13745, "rays": 1e11,
         "nx": 2048, "ny": 10240, "l1x": 28.4, "l1y": 28.1, "l2x": 20, "l2y": 10, "trace": 4096},
        # 16 uneven maps (2,000-20,000 lenses, 1e9-1e10 rays, 4096 x 4096) with
        # ten light curves each, replayed as one graph.
        {"name": "batch-16", "kind": "batch", "maps": 16, "rays_lo": 1e9, "rays_hi": 1e10, "nx": 4096,
         "tracks": 10, "samples": 4096},
        # The FP64 near/far mode: 400 lenses, 1.2e7 rays, an odd map.
        {"name": "nearfar64", "kind": "nearfar", "kappa_star": 0.05, "nx": 401, "ny": 301, "n_av": 100.0},
        # The differentiable field: 1,000 lenses, 4e8 rays, a 1024 x 1024 map,
        # squared distance to a target map.
        {"name": "grad-1000", "kind": "grad", "lenses": 1000, "rays": 4e8, "nx": 1024, "l1": 2.5, "l2": 10},
        # Light-curve loss of a small field: 16 tracks, odd map, default grid.
        {"name": "curve-loss", "kind": "curve_loss", "kappa_star": 0.05, "nx": 301, "ny": 203, "n_av": 150.0,
         "tracks": 16, "samples": 1001, "sigma": 1.5},
        # 80 light curves of 4096 samples of a source of 4 pixels on an 8192 x
        # 4096 map, forward and transposed.
        {"name": "curves-wide", "kind": "curves", "nx": 8192, "ny": 4096, "tracks": 80, "samples": 4096,
         "sigma": 4.0},
        # Peaks of a Table-1 sized count map along both axes, with statistics.
        {"name": "peaks-table1", "kind": "peaks", "nx": 2048, "ny": 10240, "mean": 1000.0},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    """One more case: every size over the range from small programs up to the
    listed one of its kind."""
    kind = rng.choice(["direct", "map", "step", "shard", "fold", "build", "batch", "nearfar", "grad",
                       "curve_loss", "curves", "peaks"])
    if kind == "direct":
        return {"kind": kind, "lenses": int(_log(rng, 10, 200)), "rays_x": rng.randint(301, 2000),
                "rays_y": rng.randint(301, 2000), "nx": rng.randint(33, 400), "ny": rng.randint(33, 400)}
    if kind == "map":
        return {"kind": kind, "kappa_star": rng.choice([0.01, 0.02, 0.05]), "nx": rng.randint(50, 500),
                "ny": rng.randint(50, 500), "n_av": _log(rng, 4.0, 200.0), "tracks": rng.randint(1, 10),
                "samples": rng.randint(50, 1500)}
    if kind == "step":
        return {"kind": kind, "lenses": int(_log(rng, 2000, 13000)), "rays": _log(rng, 2e9, 1e11),
                "nx": rng.randint(1500, 8192), "ny": rng.randint(1500, 8192)}
    if kind == "shard":
        n = rng.randint(4001, 16384)
        return {"kind": kind, "lenses": int(_log(rng, 4000, 13000)), "rays": _log(rng, 2e3, 4e4) * n * n,
                "slice": _log(rng, 3e9, 1e11), "nx": n, "ny": n, "l2x": rng.choice([20, 40]), "l2y": 20}
    if kind == "fold":
        nx = rng.randint(401, 2048)
        return {"kind": kind, "rays": _log(rng, 300, 5000) * nx * 5 * nx, "nx": nx, "ny": 5 * nx}
    if kind == "build":
        if rng.random() < 0.5:
            l1 = rng.uniform(25.0, 56.0)
            return {"kind": kind, "field": "fold", "lenses": 13745, "rays": _log(rng, 1e10, 1e11), "nx": 1024,
                    "ny": 5120, "l1x": l1, "l1y": l1, "l2x": 20, "l2y": 10, "trace": rng.randint(100, 4096)}
        return {"kind": kind, "field": "linear", "lenses": int(_log(rng, 1000, 13000)),
                "rays": _log(rng, 1e9, 1e11), "nx": rng.randint(501, 4096), "ny": rng.randint(501, 4096),
                "l1x": 0.0, "l1y": 0.0, "l2x": rng.choice([20, 40, 80]), "l2y": rng.choice([10, 20]),
                "trace": rng.randint(100, 4096)}
    if kind == "batch":
        lo = _log(rng, 1e8, 1e9)
        return {"kind": kind, "maps": rng.randint(2, 14), "rays_lo": lo, "rays_hi": lo * _log(rng, 1.5, 10.0),
                "nx": rng.randint(801, 4096), "tracks": rng.randint(1, 10), "samples": rng.randint(500, 4096)}
    if kind == "nearfar":
        return {"kind": kind, "kappa_star": rng.choice([0.01, 0.02, 0.05]), "nx": rng.randint(100, 400),
                "ny": rng.randint(100, 300), "n_av": _log(rng, 10.0, 100.0)}
    if kind == "grad":
        n = rng.randint(151, 1024)
        return {"kind": kind, "lenses": int(_log(rng, 150, 1000)), "rays": _log(rng, 20.0, 380.0) * n * n,
                "nx": n, "l1": rng.uniform(2.0, 6.0), "l2": 10}
    if kind == "curve_loss":
        return {"kind": kind, "kappa_star": rng.choice([0.02, 0.05]), "nx": rng.randint(60, 400),
                "ny": rng.randint(60, 300), "n_av": _log(rng, 20.0, 150.0), "tracks": rng.randint(1, 16),
                "samples": rng.randint(100, 1500), "sigma": _log(rng, 0.5, 4.0)}
    if kind == "curves":
        return {"kind": kind, "nx": rng.randint(500, 8192), "ny": rng.randint(500, 4096),
                "tracks": rng.randint(1, 80), "samples": int(_log(rng, 100, 4096)),
                "sigma": _log(rng, 0.5, 4.0)}
    return {"kind": kind, "nx": rng.randint(300, 4096), "ny": rng.randint(300, 5120),
            "mean": _log(rng, 50.0, 3000.0)}


# ---- inputs --------------------------------------------------------------------

def _near_critical(n, rays, nx, ny, seed):
    """A field like the paper-scale one at another lens count: the lens disc is
    1.5 times the ray rectangle's half-diagonal (as inputs.batched_maps)."""
    ks, kappa, gamma = 0.005, 0.48, 0.50
    r = math.sqrt(n * MEAN_MASS / ks)
    lf = inputs.lens_disc(n, r, seed, "lognormal", 0.3, 0.5)
    lp = r / (0.75 * math.hypot(1.0 / (1.0 - kappa - gamma), 1.0 / (1.0 - kappa + gamma)))
    h = 0.5 * (lp - 20.0 * math.sqrt(ks))
    return inputs.Workload("near-critical", lf, kappa, gamma, ks, (0.0, 0.0, r), (-h, -h, h, h), (nx, ny),
                           n_av=rays / (nx * ny))


def _small(case, seed):
    """A consistent small field near the critical line (kappa 0.40, gamma 0.45),
    lattice fixed explicitly, the lens disc 1.5 times its half-diagonal."""
    ks, kappa, gamma = case["kappa_star"], 0.40, 0.45
    nx, ny = case["nx"], case["ny"]
    bx, by = 1.0, ny / nx
    band = 10.0 * math.sqrt(ks)
    hx, hy = (bx + band) / (1.0 - kappa - gamma), (by + band) / (1.0 - kappa + gamma)
    l3 = math.sqrt(4.0 * hx * hy / (case["n_av"] * nx * ny))
    r = 1.5 * math.hypot(hx, hy)
    n = max(1, int(round(ks * r * r / MEAN_MASS)))
    lf = inputs.lens_disc(n, r, seed, "lognormal")
    return inputs.Workload("small", lf, kappa, gamma, n * MEAN_MASS / r ** 2, (0.0, 0.0, r), (-bx, -by, bx, by),
                           (nx, ny), ray_box=(-hx, -hy, hx, hy),
                           ray_n=(max(1, round(2.0 * hx / l3)), max(1, round(2.0 * hy / l3))))


def _direct_map(case, seed):
    w = inputs.small_map(seed)
    w.lenses = inputs.lens_disc(case["lenses"], 15.0, seed, "unit")
    w.map_n = (case["nx"], case["ny"])
    w.ray_n = (case["rays_x"], case["rays_y"])
    return w


def _square_lattice(w, box, rays):
    """Fix the ray rectangle and a square lattice of about `rays` rays on it."""
    lx, ly = box[2] - box[0], box[3] - box[1]
    l3 = math.sqrt(lx * ly / rays)
    w.ray_box, w.ray_n = box, (max(1, round(lx / l3)), max(1, round(ly / l3)))
    return w


def _linear_box(w):
    """Pre-image of a map centred on the origin, widened by 10 sqrt(kappa_*)."""
    a, b, band = 1.0 - w.kappa - w.gamma, 1.0 - w.kappa + w.gamma, 10.0 * math.sqrt(w.kappa_star)
    hx, hy = (w.map_box[2] + band) / a, (w.map_box[3] + band) / b
    return (-hx, -hy, hx, hy)


def _fold_box(w):
    """Bounding box of the images of the fold map's widened source region."""
    _, k0, dx, dy = w.macro
    band = 10.0 * math.sqrt(w.kappa_star)
    ty = [(w.map_box[1] - band) / (2.0 * (1.0 - k0)), (w.map_box[3] + band) / (2.0 * (1.0 - k0))]
    ends = []
    for t in ty:
        s1 = math.sqrt(2.0 * (w.map_box[2] + band) / dx + (dy * t / dx) ** 2)
        ends += [-dy * t / dx - s1, -dy * t / dx + s1]
    return (min(ends), ty[0], max(ends), ty[1])


def _build_workload(case, seed):
    if case["field"] == "fold":
        w = inputs.fold_field(seed, n_rays=case["rays"], map_px=(case["nx"], case["ny"]))
        return _square_lattice(w, _fold_box(w), case["rays"])
    w = _near_critical(case["lenses"], case["rays"], case["nx"], case["ny"], seed)
    return _square_lattice(w, _linear_box(w), case["rays"])


def _grad_workload(case, seed):
    w = inputs.differentiable_field(seed, case["lenses"], case["rays"], case["nx"])
    w.l1, w.l2 = (case["l1"], case["l1"]), (case["l2"], case["l2"])
    return _square_lattice(w, _linear_box(w), case["rays"])


def _spec(w):
    s = {"sheet": w.sheet, "map_box": w.map_box, "map_n": w.map_n, "ray_box": w.ray_box, "ray_n": w.ray_n}
    if w.l1:
        s["l1"], s["l2_sub"] = w.l1, w.l2
    return s


def _parameters(w):
    """Lens tensors and macro parameters to differentiate by, on the GPU."""
    lens = [torch.as_tensor(v, dtype=torch.float64, device="cuda").requires_grad_(True)
            for v in (w.lenses.x, w.lenses.y, w.lenses.m)]
    macro = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (w.kappa, w.gamma, w.kappa_star)]
    return lens + macro


def _target(nx, ny, seed):
    """A smooth positive target map: what a coarser model of the sky predicts."""
    g = torch.Generator().manual_seed(seed)
    p = torch.rand(6, generator=g, dtype=torch.float64)
    y = torch.linspace(0, 1, ny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device="cuda")[None, :]
    t = 6.0 + (8.0 + 4.0 * p[0]) * (1.0 + torch.sin(6.0 * p[1] + 5.0 * x + (2.0 + 3.0 * p[2]) * y))
    return (t + 20.0 * p[3] * torch.exp(-((x - p[4]) ** 2 + (y - p[5]) ** 2) * 30.0)).float()


def _tracks(case, seed):
    margin = min(4.0 * case.get("sigma", 0.5) + 1.0, 0.4 * min(case["nx"], case.get("ny", case["nx"])))
    return inputs.tracks(case["tracks"], case["nx"], case.get("ny", case["nx"]), margin, seed)


def _count_map(case, seed):
    """Counts with the look of a shot map: Poisson noise of the given mean with
    caustic ridges across it."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ny, nx = case["ny"], case["nx"]
    y = torch.arange(ny, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(nx, device="cuda", dtype=torch.float32)[None, :]
    rate = torch.full((ny, nx), 0.6 * case["mean"], device="cuda")
    p = torch.rand((24, 4), generator=g, device="cuda").tolist()
    for a, b, c, d in p:
        s = (x - a * nx) * math.cos(6.28 * b) + (y - c * ny) * math.sin(6.28 * b)
        s = s + 0.02 * nx * torch.sin((x + y) * (0.002 + 0.01 * d))
        rate += case["mean"] * torch.rsqrt(1.0 + s.abs()) * (s > 0) * (0.3 + d)
    return torch.poisson(rate, generator=g).to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "direct":
        return {"kind": kind, "w": _direct_map(case, seed)}
    if kind == "map":
        return {"kind": kind, "w": _small(case, seed), "tracks": _tracks(case, seed), "samples": case["samples"]}
    if kind == "step":
        w = _near_critical(case["lenses"], case["rays"], case["nx"], case["ny"], seed)
        return {"kind": kind, "w": w, "tracks": inputs.tracks(10, case["nx"], case["ny"], 3.0, seed),
                "mu": torch.empty((case["ny"], case["nx"]), dtype=torch.float32, device="cuda")}
    if kind == "shard":
        w = _near_critical(case["lenses"], case["rays"], case["nx"], case["ny"], seed)
        f = ml.Field(w, l2_sub=(case["l2x"], case["l2y"]))
        n = min(f.n_rays, int(case["slice"]))
        return {"kind": kind, "field": f, "begin": (f.n_rays - n) // 2, "end": (f.n_rays - n) // 2 + n,
                "out": torch.empty((case["ny"], case["nx"]), dtype=torch.int32, device="cuda")}
    if kind == "fold":
        w = inputs.fold_field(seed, n_rays=case["rays"], map_px=(case["nx"], case["ny"]))
        return {"kind": kind, "field": ml.Field(w, tune=True),
                "mu": torch.empty((case["ny"], case["nx"]), dtype=torch.float32, device="cuda")}
    if kind == "build":
        w = _build_workload(case, seed)
        kw = {"l2_sub": (case["l2x"], case["l2y"])}
        if case["l1x"]:
            kw["l1"] = (case["l1x"], case["l1y"])
        idx = np.random.default_rng(seed).integers(0, w.ray_n[0] * w.ray_n[1], case["trace"])
        return {"kind": kind, "w": w, "kw": kw, "idx": torch.as_tensor(idx, device="cuda")}
    if kind == "batch":
        maps = inputs.batched_maps(case["maps"], seed % 100000, case["nx"], (case["rays_lo"], case["rays_hi"]),
                                   case["tracks"])
        tracks = np.stack([inputs.tracks(case["tracks"], case["nx"], case["nx"], 3.0, seed + i)
                           for i in range(len(maps))])
        b = ml.Batch([ml.make_desc(w, tune=True) for w in maps], tracks, case["samples"], 0.5)
        return {"kind": kind, "batch": b}
    if kind == "nearfar":
        f = ml.Field(_small(case, seed), precision=ml.PREC_NEARFAR64)
        return {"kind": kind, "field": f}
    if kind == "grad":
        w = _grad_workload(case, seed)
        return {"kind": kind, "par": _parameters(w), "spec": _spec(w), "target": _target(*w.map_n, seed)}
    if kind == "curve_loss":
        w = _small(case, seed)
        n = case["tracks"] * case["samples"]
        t = 20.0 + 10.0 * torch.sin(torch.arange(n, device="cuda", dtype=torch.float32) * (0.01 + 1e-3 * (seed % 7)))
        return {"kind": kind, "par": _parameters(w), "spec": _spec(w), "tracks": _tracks(case, seed),
                "samples": case["samples"], "sigma": case["sigma"], "target": t.view(case["tracks"], -1)}
    if kind == "curves":
        c = _count_map({"nx": case["nx"], "ny": case["ny"], "mean": 200.0}, seed)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        return {"kind": kind, "mu": c.float() * 0.05, "tracks": _tracks(case, seed), "samples": case["samples"],
                "sigma": case["sigma"],
                "grad": torch.randn((case["tracks"], case["samples"]), generator=g, device="cuda")}
    c = _count_map(case, seed)
    w = inputs.Workload("counts", inputs.LensField(np.zeros(0), np.zeros(0), np.zeros(0)), 0.25, 0.25, 0.0,
                        (0.0, 0.0, 1000.0), (0.0, 0.0, 40.0, 40.0 * case["ny"] / case["nx"]),
                        (case["nx"], case["ny"]), ray_box=(0.0, 0.0, 80.0, 80.0), ray_n=(8, 8))
    f = ml.Field(w, precision=ml.PREC_DIRECT64)
    ml.ml_field_set_counts(f.h, c)
    n = case["nx"] * case["ny"]
    return {"kind": "peaks", "field": f, "mask_x": torch.zeros(n + 4, dtype=torch.uint8, device="cuda"),
            "mask_y": torch.zeros(n + 4, dtype=torch.uint8, device="cuda")}


# ---- one pass --------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "direct":
        f = ml.Field(s["w"], precision=ml.PREC_DIRECT64)
        f.shoot()
        out = {"counts": f.counts(), "mu": f.mu("f64")}
        f.close()
        return out
    if kind == "map":
        f = ml.Field(s["w"])
        f.shoot()
        out = {"mu": f.mu(), "curves": f.light_curves(s["tracks"], s["samples"], 0.5)}
        f.close()
        return out
    if kind == "step":
        f = ml.Field(s["w"], tune=True)
        f.shoot()
        ml.ml_magnification_map(f.h, ml.MAP_MU_F32, s["mu"])
        curves = f.light_curves(s["tracks"], 4096, 0.5)
        dropped = f.stats()["rays_dropped"]
        f.close()
        return {"mu": s["mu"], "curves": curves, "dropped": dropped}
    if kind == "shard":
        f = s["field"]
        f.clear()
        f.shoot(s["begin"], s["end"])
        ml.ml_magnification_map(f.h, ml.MAP_COUNTS_U32, s["out"])
        return {"counts": s["out"]}
    if kind == "fold":
        f = s["field"]
        f.clear()
        f.shoot()
        ml.ml_magnification_map(f.h, ml.MAP_MU_F32, s["mu"])
        return {"mu": s["mu"]}
    if kind == "build":
        f = ml.Field(s["w"], **s["kw"])
        n = s["idx"].numel()
        beta = torch.empty((n, 2), dtype=torch.float64, device="cuda")
        pix = torch.empty((n, 2), dtype=torch.int32, device="cuda")
        ml.ml_trace_rays(f.h, s["idx"], beta, pix)
        f.close()
        return {"beta": beta, "pix": pix}
    if kind == "batch":
        b = s["batch"]
        b.run()
        return {"curves": b.curves(), "mu": [b.mu(i) for i in range(b.n)]}
    if kind == "nearfar":
        f = s["field"]
        f.clear()
        f.shoot()
        return {"counts": f.counts(), "mu": f.mu("f64")}
    if kind == "grad":
        for p in s["par"]:
            p.grad = None
        mu = autograd.CICMagnification.apply(*s["par"], s["spec"])
        ((mu - s["target"]) ** 2).sum().backward()
        return {"mu": mu.detach(), **_gradients(s["par"])}
    if kind == "curve_loss":
        for p in s["par"]:
            p.grad = None
        mu = autograd.CICMagnification.apply(*s["par"], s["spec"])
        c = autograd.LightCurves.apply(mu, s["tracks"], s["samples"], s["sigma"])
        ((c - s["target"]) ** 2).sum().backward()
        return {"mu": mu.detach(), "curves": c.detach(), **_gradients(s["par"])}
    if kind == "curves":
        mu = s["mu"].requires_grad_(True)
        mu.grad = None
        c = autograd.LightCurves.apply(mu, s["tracks"], s["samples"], s["sigma"])
        c.backward(s["grad"])
        return {"curves": c.detach(), "grad": mu.grad}
    h, out = s["field"].h, {}
    for name, along, mask in (("x", ml.ALONG_X, s["mask_x"]), ("y", ml.ALONG_Y, s["mask_y"])):
        n, _ = ml.ml_find_peaks(h, along, 5.0, mask, 1 << 20)
        out[name] = [n, mask, *(v.astype(np.int64) for v in ml.ml_peak_statistics(h, EDGES, along, 0.0, mask))]
    return out


def _gradients(par):
    return {"lens": [p.grad for p in par[:3]], "macro": torch.stack([p.grad for p in par[3:]])}


# ---- what a pass cannot do without -----------------------------------------------

def _runs(rays, nx, ny, slope):
    """Runs of rays that share a pixel along the lattice rows: a row of rays at
    macro slope `slope` crosses a pixel edge every (rays per pixel row) rays."""
    per = max(1.0, math.sqrt(rays / (nx * ny) / slope))
    return rays / per


def work(case):
    """Lenses read and maps written once.  Operations of a counted map: two
    evaluations (about 70 operations with the far series and the near lenses)
    per run of rays in one pixel, at the macro slope; of an FP64 direct sum: 12
    per ray and lens."""
    kind, nx, ny = case["kind"], case["nx"], case.get("ny", case["nx"])
    px = float(nx * ny)
    if kind == "direct":
        return {"bytes": 16.0 * px, "flops": 12.0 * case["rays_x"] * case["rays_y"] * case["lenses"]}
    if kind == "map":
        rays = case["n_av"] * px
        return {"bytes": 8.0 * px, "flops": 140.0 * _runs(rays, nx, ny, 0.15)}
    if kind == "step":
        return {"bytes": 24.0 * case["lenses"] + 8.0 * px, "flops": 140.0 * _runs(case["rays"], nx, ny, 0.02)}
    if kind == "shard":
        return {"bytes": 8.0 * px,
                "flops": 140.0 * _runs(case["rays"], nx, ny, 0.02) * min(1.0, case["slice"] / case["rays"])}
    if kind == "fold":
        return {"bytes": 8.0 * px, "flops": 140.0 * _runs(case["rays"], nx, ny, 0.2)}
    if kind == "build":
        return {"bytes": 24.0 * case["lenses"] + 4.0 * px + 48.0 * case["trace"],
                "flops": 12.0 * case["lenses"] * case["trace"]}
    if kind == "batch":
        rays = case["maps"] * math.sqrt(case["rays_lo"] * case["rays_hi"])
        return {"bytes": 8.0 * px * case["maps"] + 4.0 * case["maps"] * case["tracks"] * case["samples"],
                "flops": 140.0 * case["maps"] * _runs(rays / case["maps"], nx, ny, 0.03)}
    if kind == "nearfar":
        return {"bytes": 16.0 * px, "flops": 60.0 * case["n_av"] * px}
    if kind == "grad":
        return {"bytes": 16.0 * px + 48.0 * case["lenses"], "flops": 500.0 * _runs(case["rays"], nx, nx, 0.02)}
    if kind == "curve_loss":
        return {"bytes": 16.0 * px + 12.0 * case["tracks"] * case["samples"],
                "flops": 500.0 * _runs(case["n_av"] * px, nx, ny, 0.15)}
    if kind == "curves":
        h = 2 * math.floor(4.0 * case["sigma"]) + 2
        return {"bytes": 8.0 * px + 8.0 * case["tracks"] * case["samples"],
                "flops": 4.0 * h * h * case["tracks"] * case["samples"]}
    return {"bytes": 2.0 * 5.0 * px, "flops": 2.0 * 10.0 * px}


# How far two correct implementations may lie apart.  FP32 arithmetic on
# node-relative coordinates moves a ray by about 1e-7 of its deflection, which
# takes the rays within that distance of a pixel edge to the next pixel: about
# 1.5 in a million, measured against the direct sum and between level-1 grids.
# A map of n_av rays per pixel then differs by sqrt(3e-6 / n_av) in its 2-norm,
# in single counts of few pixels.  Four times that is stated, and at least the
# few rays of a small map.  Traced positions carry the series' truncation
# (at most 1e-7 Einstein radii).  The others are four times the largest error
# measured against exact(): FP64 sums in another order move no ray, traced
# positions agree to 7e-11 on the fold field, gradients to 2.4e-5 (FP32 pair terms of both
# signs), curves to 2.8e-8 and their transpose, FP32 atomics, to 2.8e-7.
def _flips(n_av, px):
    return {"rel": min(0.03, max(7e-3 / math.sqrt(n_av), 6.0 / (n_av * math.sqrt(px)))),
            "max": min(0.99, max(0.05, 4.0 / n_av)), "differ": 1e-3}


def tolerance(case):
    kind, px = case["kind"], float(case["nx"] * case.get("ny", case["nx"]))
    if kind in ("map",):
        return _flips(case["n_av"], px)
    if kind in ("step", "shard", "fold"):
        return _flips(case["rays"] / px, px)
    if kind == "batch":
        return _flips(case["rays_lo"] / px, px)
    return {"direct": {"rel": 1e-5, "differ": 1e-5},
            "nearfar": {"rel": 1e-4, "max": 0.3, "differ": 1e-3},
            "build": {"rel": 2e-8, "max": 4e-7, "differ": 1e-3},
            "grad": {"rel": 1e-4, "max": 4e-3},
            "curve_loss": {"rel": 1e-4, "max": 4e-3},
            "curves": {"rel": 1.2e-6, "max": 4e-5}}.get(kind, "exact")


# ---- the same results in 64 bits ---------------------------------------------------

PAIRS = 1.5e10          # ray-lens pairs that exact() takes on


def _rays(w, k):
    n3x, n3y = w.ray_n
    x0, y0, x1, y1 = w.ray_box
    tx = x0 + ((k % n3x).double() + 0.5) * ((x1 - x0) / n3x)
    ty = y0 + (torch.div(k, n3x, rounding_mode="floor").double() + 0.5) * ((y1 - y0) / n3y)
    return tx, ty


def _beta(w, lens, tx, ty):
    """Source positions by the direct sum over all lenses, and the pair terms."""
    x, y, m = lens
    dx, dy = tx[:, None] - x[None, :], ty[:, None] - y[None, :]
    inv = 1.0 / (dx * dx + dy * dy)
    ax, ay = (dx * inv) @ m, (dy * inv) @ m
    ux, uy = tx - w.sheet[0], ty - w.sheet[1]
    if len(w.sheet) > 3:
        sx, sy = torch.zeros_like(ux), -2.0 * w.kappa_star * uy.clamp(-w.sheet[2], w.sheet[2])
    else:
        s = -w.kappa_star * torch.clamp(w.sheet[2] ** 2 / (ux * ux + uy * uy), max=1.0)
        sx, sy = s * ux, s * uy
    if w.macro is not None:
        _, k0, d0, d1 = w.macro
        mx, my = 0.5 * d0 * tx * tx + d1 * tx * ty, 2.0 * (1.0 - k0) * ty
    else:
        mx, my = (1.0 - w.kappa - w.gamma) * tx, (1.0 - w.kappa + w.gamma) * ty
    return mx - ax - sx, my - ay - sy, dx, dy, inv


def _lens64(w):
    return [torch.as_tensor(v, dtype=torch.float64, device="cuda") for v in (w.lenses.x, w.lenses.y, w.lenses.m)]


def _chunks(w):
    n = w.ray_n[0] * w.ray_n[1]
    step = max(1, int(4e7 / max(1, w.lenses.n)))
    return [torch.arange(k, min(n, k + step), device="cuda") for k in range(0, n, step)]


def _pixel(w):
    x0, y0, x1, y1 = w.map_box
    return x0, y0, (x1 - x0) / w.map_n[0], (y1 - y0) / w.map_n[1]


def _scale(w):
    _, _, dpx, dpy = _pixel(w)
    x0, y0, x1, y1 = w.ray_box
    return ((x1 - x0) / w.ray_n[0]) * ((y1 - y0) / w.ray_n[1]) / (dpx * dpy)


def _mu64(w):
    lens, (nx, ny) = _lens64(w), w.map_n
    mx0, my0, dpx, dpy = _pixel(w)
    out = torch.zeros(nx * ny, dtype=torch.float64, device="cuda")
    for k in _chunks(w):
        bx, by = _beta(w, lens, *_rays(w, k))[:2]
        ix, iy = torch.floor((bx - mx0) / dpx), torch.floor((by - my0) / dpy)
        ok = (ix >= 0) & (ix < nx) & (iy >= 0) & (iy < ny)
        out += torch.bincount((iy[ok] * nx + ix[ok]).long(), minlength=nx * ny).double()
    return out.view(ny, nx) * _scale(w)


def _corners(w, bx, by):
    """The four pixels around each ray, their weights, and which lie in the map."""
    nx, ny = w.map_n
    mx0, my0, dpx, dpy = _pixel(w)
    fx, fy = (bx - mx0) / dpx - 0.5, (by - my0) / dpy - 0.5
    ix, iy = torch.floor(fx), torch.floor(fy)
    wx, wy = fx - ix, fy - iy
    for cx in (0, 1):
        for cy in (0, 1):
            px, py = ix + cx, iy + cy
            ok = (px >= 0) & (px < nx) & (py >= 0) & (py < ny)
            at = torch.where(ok, py * nx + px, 0.0).long()
            ox, oy = (wx if cx else 1.0 - wx), (wy if cy else 1.0 - wy)
            yield at, ok.double(), ox, oy, (1.0 if cx else -1.0) / dpx, (1.0 if cy else -1.0) / dpy


def _cic64(w):
    lens, (nx, ny) = _lens64(w), w.map_n
    out = torch.zeros(nx * ny, dtype=torch.float64, device="cuda")
    for k in _chunks(w):
        bx, by = _beta(w, lens, *_rays(w, k))[:2]
        for at, ok, ox, oy, _, _ in _corners(w, bx, by):
            out.index_add_(0, at, ok * ox * oy)
    return out.view(ny, nx) * _scale(w)


def _grad64(w, dM):
    """dLoss/d(x, y, m) and dLoss/d(kappa, gamma, kappa_*) from dLoss/dM."""
    lens = _lens64(w)
    G = dM.reshape(-1) * _scale(w)
    gl = [torch.zeros_like(v) for v in lens]
    gp = torch.zeros(3, dtype=torch.float64, device="cuda")
    for k in _chunks(w):
        tx, ty = _rays(w, k)
        bx, by, dx, dy, inv = _beta(w, lens, tx, ty)
        gx, gy = torch.zeros_like(bx), torch.zeros_like(by)
        for at, ok, ox, oy, sx, sy in _corners(w, bx, by):
            v = G[at] * ok
            gx += v * sx * oy
            gy += v * ox * sy
        t = (gx[:, None] * dx + gy[:, None] * dy) * inv
        gl[2] -= t.sum(0)
        gl[0] += lens[2] * ((gx[:, None] - 2.0 * t * dx) * inv).sum(0)
        gl[1] += lens[2] * ((gy[:, None] - 2.0 * t * dy) * inv).sum(0)
        gp += torch.stack([-(gx * tx + gy * ty).sum(), (gy * ty - gx * tx).sum(),
                           (gx * (tx - w.sheet[0]) + gy * (ty - w.sheet[1])).sum()])
    return {"lens": gl, "macro": gp.cpu()}


def _curves64(mu, tracks, samples, sigma):
    """Gaussian-source light curves sampled bilinearly, differentiable in mu."""
    ny, nx = mu.shape
    h = math.floor(4.0 * sigma)
    taps = torch.exp(-0.5 * (torch.arange(-h, h + 1, dtype=torch.float64, device="cuda") / sigma) ** 2)
    taps = (taps / taps.sum()).float().double()
    tr = torch.as_tensor(np.asarray(tracks), dtype=torch.float64, device="cuda")
    t = torch.arange(samples, dtype=torch.float64, device="cuda") / max(1, samples - 1)
    u = (tr[:, 0:1] + t * (tr[:, 2:3] - tr[:, 0:1]) - 0.5).reshape(-1)
    v = (tr[:, 1:2] + t * (tr[:, 3:4] - tr[:, 1:2]) - 0.5).reshape(-1)
    fu, fv = torch.floor(u), torch.floor(v)
    wx, wy = u - fu, v - fv
    zero = torch.zeros(1, dtype=torch.float64, device="cuda")
    off = torch.arange(-h, h + 2, dtype=torch.int64, device="cuda")
    pad = torch.cat([taps, zero]), torch.cat([zero, taps])
    out = []
    for a in range(0, u.numel(), 16384):
        sl = slice(a, a + 16384)
        kx = (1.0 - wx[sl, None]) * pad[0] + wx[sl, None] * pad[1]
        ky = (1.0 - wy[sl, None]) * pad[0] + wy[sl, None] * pad[1]
        # a corner pixel outside the map has no value; tracks keep clear of the rim
        px, py = fu[sl, None].long() + off, fv[sl, None].long() + off
        kx = kx * ((px >= 0) & (px < nx))
        ky = ky * ((py >= 0) & (py < ny))
        at = (py.clamp(0, ny - 1) * nx)[:, :, None] + px.clamp(0, nx - 1)[:, None, :]
        out.append(((mu.reshape(-1)[at] * kx[:, None, :]).sum(2) * ky).sum(1))
    return torch.cat(out).view(len(tracks), samples)


def exact(case, seed):
    kind = case["kind"]
    if kind == "direct":
        return {"counts": None, "mu": _mu64(_direct_map(case, seed))}
    if kind in ("map", "nearfar"):
        w = _small(case, seed)
        if w.ray_n[0] * w.ray_n[1] * w.lenses.n > PAIRS:
            return None
        mu = _mu64(w)
        if kind == "nearfar":
            return {"counts": None, "mu": mu}
        return {"mu": mu, "curves": _curves64(mu, _tracks(case, seed), case["samples"], 0.5)}
    if kind == "build":
        s = prepare(case, seed)
        w = s["w"]
        lens = _lens64(w)
        beta = [torch.stack(_beta(w, lens, *_rays(w, k))[:2], 1) for k in s["idx"].split(1024)]
        return {"beta": torch.cat(beta), "pix": None}
    if kind == "grad":
        w = _grad_workload(case, seed)
        if w.ray_n[0] * w.ray_n[1] * w.lenses.n > PAIRS:
            return None
        mu = _cic64(w)
        return {"mu": mu, **_grad64(w, 2.0 * (mu - _target(*w.map_n, seed).double()))}
    if kind == "curve_loss":
        w, s = _small(case, seed), prepare(case, seed)
        if w.ray_n[0] * w.ray_n[1] * w.lenses.n > PAIRS:
            return None
        mu = _cic64(w).requires_grad_(True)
        c = _curves64(mu, s["tracks"], s["samples"], s["sigma"])
        ((c - s["target"].double()) ** 2).sum().backward()
        return {"mu": mu.detach(), "curves": c.detach(), **_grad64(w, mu.grad)}
    if kind == "curves":
        s = prepare(case, seed)
        mu = s["mu"].double().requires_grad_(True)
        c = _curves64(mu, s["tracks"], s["samples"], s["sigma"])
        c.backward(s["grad"].double())
        return {"curves": c.detach(), "grad": mu.grad}
    return None
