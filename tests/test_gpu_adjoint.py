"""Cloud-in-cell map and its hand-written adjoint on the GPU.

The forward CIC map is checked against the FP64 oracle map; the adjoint
(ml_cic_backward) against the oracle's FP64 gradient on the same dLoss/dM,
and against central finite differences of the GPU forward itself through
the torch.autograd.Function.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2308_14278_gb300 import inputs

pytestmark = pytest.mark.gpu


def _case(seed=11, kappa=0.42, gamma=0.40, ks=0.05, map_n=(64, 48), n_av=150):
    """A consistent field (kappa_* = N <m> / R^2, disc 1.5 times the ray
    rectangle's half-diagonal) with the ray lattice fixed explicitly, so that
    it does not move with kappa and gamma."""
    box = (-1.0, -0.75, 1.0, 0.75)
    g0 = oracle.derive_geometry(kappa, gamma, ks, [], [], (0, 0, 1), box, map_n, n_av=n_av)
    r = 1.5 * math.hypot(max(abs(g0.rx0), abs(g0.rx1)), max(abs(g0.ry0), abs(g0.ry1)))
    n = int(round(ks * r * r / inputs.lognormal_mean(0.3, 0.5)))
    lf = inputs.lens_disc(n, r, seed, "lognormal")
    ks = n * inputs.lognormal_mean(0.3, 0.5) / r ** 2
    return inputs.Workload("cic", lf, kappa, gamma, ks, (0.0, 0.0, r), box, map_n,
                           ray_box=(g0.rx0, g0.ry0, g0.rx1, g0.ry1), ray_n=(g0.n3x, g0.n3y))


def _target(w, seed=12):
    """A smooth positive target map (a tilted plane plus a bump)."""
    ny, nx = w.map_n[1], w.map_n[0]
    yy, xx = np.mgrid[0:ny, 0:nx]
    return 2.0 + 0.5 * xx / nx - 0.3 * yy / ny + np.exp(-((xx - nx / 2) ** 2 + (yy - ny / 3) ** 2) / 50.0)


def _field(ml, w, **kw):
    return ml.Field(w, precision=ml.PREC_MIXED, deposit=ml.DEPOSIT_CIC, **kw)


def test_cic_map_matches_oracle(ml):
    w = _case()
    f = _field(ml, w)
    info = f.info
    g = oracle.geometry_of(w, p=info["taylor_p"], l2_sub=info["l2_sub_x"], l2_sub_y=info["l2_sub_y"])
    f.shoot()
    st = f.stats()
    mu = f.mu("f32").cpu().numpy().astype(np.float64)
    ref = oracle.cic_mu_scale(g) * oracle.cic_forward(g, w.lenses.x, w.lenses.y, w.lenses.m)
    assert st["rays_dropped"] == 0
    err = np.abs(mu - ref)
    assert err.max() <= 1e-4 * ref.mean(), err.max() / ref.mean()
    assert err.sum() / ref.sum() <= 1e-5
    # the one-call differentiable forward clears, reshoots and scales the same map
    import torch
    again = torch.empty(w.map_n[::-1], dtype=torch.float32, device="cuda")
    ml.ml_cic_forward(f.h, again)
    assert np.allclose(again.cpu().numpy(), mu, rtol=1e-5, atol=1e-6 * mu.max())
    f.close()


@pytest.mark.parametrize("method", ["nearfar", "direct"])
def test_cic_adjoint_matches_oracle_gradient(ml, method):
    import torch
    w = _case()
    f = _field(ml, w)
    info = f.info
    assert info["far_bound"] <= 1e-7
    g = oracle.geometry_of(w, p=info["taylor_p"], l2_sub=info["l2_sub_x"], l2_sub_y=info["l2_sub_y"])
    T = _target(w)
    gl_ref, gp_ref = oracle.cic_grad(g, w.lenses.x, w.lenses.y, w.lenses.m, T)
    _, M = oracle.cic_loss(g, w.lenses.x, w.lenses.y, w.lenses.m, T)
    G = torch.as_tensor(2.0 * (M - T), dtype=torch.float32).cuda().contiguous()
    f.shoot()
    glens = torch.full((w.lenses.n, 3), 7.0, dtype=torch.float64, device="cuda")   # overwritten
    gpar = torch.full((3,), 7.0, dtype=torch.float64, device="cuda")
    ml.ml_cic_backward(f.h, G, glens, gpar,
                       method=ml.ADJOINT_NEARFAR if method == "nearfar" else ml.ADJOINT_DIRECT)
    gl, gp = glens.cpu().numpy(), gpar.cpu().numpy()
    for c in range(3):
        scale = np.abs(gl_ref[:, c]).max()
        assert np.abs(gl[:, c] - gl_ref[:, c]).max() <= 1e-4 * scale, (c, np.abs(gl[:, c] - gl_ref[:, c]).max() / scale)
    assert np.all(np.abs(gp - gp_ref) <= 1e-4 * np.abs(gp_ref)), (gp, gp_ref)
    f.close()


def test_cic_backward_rejects_ngp_field(ml):
    import torch
    w = _case()
    f = ml.Field(w, precision=ml.PREC_MIXED)
    G = torch.zeros(w.map_n[::-1], dtype=torch.float32, device="cuda")
    glens = torch.zeros((w.lenses.n, 3), dtype=torch.float64, device="cuda")
    gpar = torch.zeros(3, dtype=torch.float64, device="cuda")
    with pytest.raises(ml.MLError):
        ml.ml_cic_backward(f.h, G, glens, gpar)
    f.close()


def test_autograd_function_matches_finite_differences(ml):
    """Gradient of L = sum (M - T)^2 through CICMagnification.backward against
    central differences of the GPU forward.  A ray at distance r from a lens
    moves by m h / r^2, so for a lens among the rays the difference quotient
    converges only once that is well below a pixel: for the dominant lens
    here the FP64 oracle's quotient is -1579, -5154, -5561, -5695.6 at
    h = 1e-3, 3e-4, 1e-4, 3e-5 against the exact -5695.9.  The difference
    check therefore takes the lenses with the largest position gradients
    among those at least 0.3 from the ray rectangle, at h = 3e-4: there the
    oracle's own quotient is within 0.11% of its exact gradient for positions,
    0.2% for kappa and gamma and 1.2% for masses (a mass moves every ray, and
    the CIC weights have kinks at pixel centres).  A smaller h would meet the
    FP32 resolution of the forward's lens offsets and Taylor coefficients.
    The tolerance adds the measured run-to-run spread of L (FP32 atomic
    order).  With the sheet centred on the origin, dL/dkappa = -dL/dkappa_*
    exactly."""
    import torch
    from paper_2308_14278_gb300.autograd import CICMagnification
    w = _case(n_av=400)
    T = torch.as_tensor(_target(w), dtype=torch.float64).cuda()
    probe = _field(ml, w)
    spec = dict(sheet=w.sheet, map_box=w.map_box, map_n=w.map_n, ray_box=w.ray_box, ray_n=w.ray_n,
                taylor_p=probe.info["taylor_p"],
                l1=(probe.info["n1x"] * probe.info["l3x"], probe.info["n1y"] * probe.info["l3y"]),
                l2_sub=(probe.info["l2_sub_x"], probe.info["l2_sub_y"]))
    probe.close()
    x = torch.tensor(w.lenses.x, requires_grad=True)
    y = torch.tensor(w.lenses.y, requires_grad=True)
    m = torch.tensor(w.lenses.m, requires_grad=True)
    par = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
           for v in (w.kappa, w.gamma, w.kappa_star)]

    def loss(xv, yv, mv, kv, gv, sv):
        M = CICMagnification.apply(xv, yv, mv, kv, gv, sv, spec)
        return ((M.double() - T) ** 2).sum()

    L = loss(x, y, m, *par)
    L.backward()
    assert all(t.grad is not None and t.grad.shape == t.shape for t in (x, y, m, *par))
    base = [loss(x.detach(), y.detach(), m.detach(), *[p.detach() for p in par]).item()
            for _ in range(4)]
    h = 3e-4
    spread = (max(base) - min(base)) / (2 * h)         # quotient noise from FP32 accumulation
    x0, y0, x1, y1 = w.ray_box
    dist = np.hypot(np.maximum(np.maximum(x0 - w.lenses.x, w.lenses.x - x1), 0),
                    np.maximum(np.maximum(y0 - w.lenses.y, w.lenses.y - y1), 0))
    score = np.where(dist > 0.3, np.abs(x.grad.numpy()) + np.abs(y.grad.numpy()), -1.0)
    ranked = np.argsort(-score)[:3]
    assert np.all(score[ranked] > 0)
    for k in ranked:
        for c, t in enumerate((x, y, m)):
            arrs = [x.detach().clone(), y.detach().clone(), m.detach().clone()]
            arrs[c][k] += h
            lp = loss(*arrs, *[p.detach() for p in par]).item()
            arrs[c][k] -= 2 * h
            lm = loss(*arrs, *[p.detach() for p in par]).item()
            fd = (lp - lm) / (2 * h)
            ad = t.grad[k].item()
            tol = (0.025 if c == 2 else 0.01) * abs(ad) + 4 * spread
            assert abs(fd - ad) <= tol, (k, c, fd, ad, spread)
    for q in range(3):
        pv = [p.detach().clone() for p in par]
        pv[q] += h
        lp = loss(x.detach(), y.detach(), m.detach(), *pv).item()
        pv[q] -= 2 * h
        lm = loss(x.detach(), y.detach(), m.detach(), *pv).item()
        fd = (lp - lm) / (2 * h)
        ad = par[q].grad.item()
        assert abs(fd - ad) <= 0.01 * abs(ad) + 4 * spread, (q, fd, ad, spread)
    assert abs(par[0].grad.item() + par[2].grad.item()) <= 1e-6 * abs(par[0].grad.item())


def test_cic_stripe_of_the_differentiable_field_matches_oracle(ml):
    """The differentiable field (1,000 lenses, 4e8-ray lattice, 2.5 theta_E
    level-1 cells: most near lists empty, some with one lens) shot on a stripe
    of 64 lattice rows from a ragged start, so that the forward's pair walk
    runs in every form (empty and short near lists, uniform and ragged lane
    ranges), against the oracle's CIC map of the same rays."""
    w = inputs.differentiable_field(0)
    f = _field(ml, w)
    info = f.info
    g = oracle.geometry_of(w, p=info["taylor_p"], l2_sub=info["l2_sub_x"], l2_sub_y=info["l2_sub_y"],
                           l1=(info["n1x"] * info["l3x"], info["n1y"] * info["l3y"]))
    r0 = (g.n3y // 2) * g.n3x + 777
    r1 = r0 + 64 * g.n3x
    f.shoot(r0, r1)
    st = f.stats()
    assert st["rays_in"] + st["rays_out"] + st["rays_dropped"] == r1 - r0
    assert 0.02 < st["near_pairs"] / (r1 - r0) < 0.5
    mu = f.mu("f32").cpu().numpy().astype(np.float64)
    ref = oracle.cic_mu_scale(g) * oracle.cic_forward(g, w.lenses.x, w.lenses.y, w.lenses.m, r0, r1)
    err = np.abs(mu - ref)
    assert err.max() <= 1e-4 * ref.max(), err.max() / ref.max()
    assert err.sum() / ref.sum() <= 1e-5
    f.close()


def test_cic_adjoint_on_a_stripe_of_the_differentiable_field_matches_oracle(ml):
    """ml_cic_backward (near/far and direct) against the oracle's FP64
    gradient on a field whose lattice is 64 rows of the differentiable
    field's, starting on a level-1 row boundary, with the same level-1 cells
    (2.5 theta_E) and level-2 subdivisions (10, 10): nine tasks in ten have
    no near lens, so the adjoint's zero- and one-lens pair walks run as they
    do on the full field."""
    import dataclasses
    import torch
    full = inputs.differentiable_field(0)
    f0 = _field(ml, full)
    fi = f0.info
    f0.close()
    rows = 64
    j0 = fi["n1y"] * (fi["N1y"] // 2)
    ry0 = fi["ray_y0"] + j0 * fi["l3y"]
    w = dataclasses.replace(full, ray_box=(fi["ray_x0"], ry0, fi["ray_x1"], ry0 + rows * fi["l3y"]),
                            ray_n=(fi["n_rays_x"], rows), n_av=0.0,
                            l1=(fi["n1x"] * fi["l3x"], fi["n1y"] * fi["l3y"]))
    f = _field(ml, w)
    info = f.info
    for k in ("n1x", "n1y", "n2x", "n2y", "l2_sub_x", "l2_sub_y"):
        assert info[k] == fi[k], k
    assert info["far_bound"] <= 1e-7
    g = oracle.geometry_of(w, p=info["taylor_p"], l2_sub=info["l2_sub_x"], l2_sub_y=info["l2_sub_y"])
    assert (g.n1x, g.n1y, g.n2x, g.n2y) == (info["n1x"], info["n1y"], info["n2x"], info["n2y"])
    f.shoot()
    st = f.stats()
    assert st["rays_dropped"] == 0 and st["rays_in"] > 0.5 * f.n_rays
    assert 0.02 < st["near_pairs"] / f.n_rays < 0.5
    # a smooth dL/dM: a ray's dL/dbeta then changes little when its FP32
    # source position and the oracle's FP64 one fall on either side of a pixel
    # centre (with an uncorrelated dL/dM one such ray moves a column's sum by
    # about 1/sqrt(rays) of its size)
    ny, nx = w.map_n[1], w.map_n[0]
    yy, xx = np.mgrid[0:ny, 0:nx]
    Gn = (np.cos(2 * np.pi * xx / 97.0) + np.sin(2 * np.pi * yy / 61.0) +
          0.5 * np.exp(-((xx - 0.4 * nx) ** 2 + (yy - 0.5 * ny) ** 2) / 2000.0)).astype(np.float32)
    G = torch.from_numpy(Gn)
    gl_ref, gp_ref = oracle.cic_grad_dM(g, w.lenses.x, w.lenses.y, w.lenses.m, Gn.astype(np.float64))
    Gd = G.cuda().contiguous()
    for method in (ml.ADJOINT_NEARFAR, ml.ADJOINT_DIRECT):
        gl = torch.empty((w.lenses.n, 3), dtype=torch.float64, device="cuda")
        gp = torch.empty(3, dtype=torch.float64, device="cuda")
        ml.ml_cic_backward(f.h, Gd, gl, gp, method=method)
        gl, gp = gl.cpu().numpy(), gp.cpu().numpy()
        for c in range(3):
            scale = np.abs(gl_ref[:, c]).max()
            err = np.abs(gl[:, c] - gl_ref[:, c]).max() / scale
            assert err <= 1e-4, (method, c, err)
        assert np.all(np.abs(gp - gp_ref) <= 1e-4 * np.abs(gp_ref)), (method, gp, gp_ref)
    f.close()


def test_nearfar_adjoint_agrees_with_direct_at_full_size(ml):
    """1,000 lenses, 4e8 rays, 1024^2 CIC: the moment-based adjoint (far
    lenses through the node series) against every ray times every lens with
    the exact derivatives; they differ by the series truncation only."""
    import torch
    w = inputs.differentiable_field(0)
    f = _field(ml, w)
    assert f.info["far_bound"] <= 1e-7
    G = torch.randn(w.map_n[::-1], generator=torch.Generator().manual_seed(3)).cuda()
    out = {}
    for method in (ml.ADJOINT_NEARFAR, ml.ADJOINT_DIRECT):
        gl = torch.empty((w.lenses.n, 3), dtype=torch.float64, device="cuda")
        gp = torch.empty(3, dtype=torch.float64, device="cuda")
        ml.ml_cic_backward(f.h, G, gl, gp, method=method)
        out[method] = (gl.cpu().numpy(), gp.cpu().numpy())
    (a, pa), (b, pb) = out[ml.ADJOINT_NEARFAR], out[ml.ADJOINT_DIRECT]
    for c in range(3):
        scale = np.abs(b[:, c]).max()
        assert np.abs(a[:, c] - b[:, c]).max() <= 1e-4 * scale, (c, np.abs(a[:, c] - b[:, c]).max() / scale)
    assert np.all(np.abs(pa - pb) <= 1e-5 * np.abs(pb))
    # the sheet is centred on the origin: dL/dkappa = -dL/dkappa_*
    assert abs(pa[0] + pa[2]) <= 1e-9 * abs(pa[0])
    f.close()


# -- light-curve loss ---------------------------------------------------------

def _lc_case(seed=21, nx=40, ny=30, n_tracks=5, n_samples=60, sigma=0.8):
    rng = np.random.default_rng(seed)
    mu = rng.uniform(0.5, 3.0, (ny, nx))
    tracks = np.column_stack([rng.uniform(-2, nx + 1, n_tracks), rng.uniform(-2, ny + 1, n_tracks),
                              rng.uniform(-2, nx + 1, n_tracks), rng.uniform(-2, ny + 1, n_tracks)])
    return mu, tracks, n_samples, sigma


def test_map_light_curves_match_oracle(ml):
    import torch
    mu, tracks, ns, sigma = _lc_case()
    out = torch.empty((len(tracks), ns), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves(torch.as_tensor(mu, dtype=torch.float32).cuda(), tracks, ns, sigma, out)
    ref = oracle.light_curves(mu.astype(np.float32).astype(np.float64), tracks, ns, sigma)
    assert np.allclose(out.cpu().numpy(), ref, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("l2", [(10, 10), (3, 2), (1, 1)])
@pytest.mark.parametrize("px", [(64, 48), (301, 7), (5, 4)])
def test_cic_runs_by_quadrature_match_the_rays_one_by_one(ml, l2, px):
    """Columns without near lenses sum a quad's rays by quadrature; the per-ray
    walk evaluates each.  Long columns on short quads, quads longer than a column
    and a few rays wide, on a sparse field: the same rays in and out of the map,
    and every pixel within the FP32 sums' rounding, 2^-24 of the pixel's sum per
    quad added (some hundred), and weights of 2e-7 a ray."""
    w = _case()
    w.map_n = px
    n_rays = w.ray_n[0] * w.ray_n[1]
    kw = dict(l1=(2.0, 1.5), l2_sub=l2)
    fq, fr = _field(ml, w, **kw), _field(ml, w, walk=ml.WALK_PER_RAY, **kw)
    for r0, r1 in ((0, n_rays), (n_rays // 3 + 5, n_rays // 2 + 1)):
        out = []
        for f in (fq, fr):
            f.clear()
            f.shoot(r0, r1)
            out.append((f.mu().cpu().numpy().astype(np.float64), f.stats()))
        (a, sa), (b, sb) = out
        for k in ("rays_in", "rays_out", "rays_dropped", "near_pairs"):
            assert sa[k] == sb[k], k
        assert np.abs(a - b).max() <= 2e-5 * b.max(), np.abs(a - b).max() / b.max()
        assert abs(a.sum() - b.sum()) <= 1e-6 * b.sum()
    fq.close()
    fr.close()


@pytest.mark.parametrize("cells", [4, 5, 6, 7])
def test_cic_quadrature_on_level1_cells_a_few_rays_wide(ml, cells):
    """Cells a few rays wide, where far lenses come as near as that: a piece of four
    rays there would carry up to 9e-6 of the map's largest value from the
    quadrature; pieces of three are the rays themselves.  Against the rays one by
    one: a pixel sums some 200 rays of weights rounded to 2^-24 of the sum at most,
    16 x 2^-24 being several times their rms."""
    w = _case()
    w.map_n, w.ray_n = (30, 22), (400, 300)
    lx, ly = (w.ray_box[2] - w.ray_box[0]) / 400, (w.ray_box[3] - w.ray_box[1]) / 300
    kw = dict(l1=(cells * lx, 20 * ly), l2_sub=(1, 1), taylor_p=16)
    out = []
    for walk in (ml.WALK_CERTIFIED, ml.WALK_PER_RAY):
        f = _field(ml, w, walk=walk, **kw)
        assert f.info["n1x"] == cells
        f.shoot()
        out.append(f.mu().cpu().numpy().astype(np.float64))
        f.close()
    assert np.abs(out[0] - out[1]).max() <= 16 * 2.0 ** -24 * out[1].max(), np.abs(out[0] - out[1]).max() / out[1].max()


@pytest.mark.parametrize("px,same", [((400, 300), True), ((42, 31), True), ((20, 15), False)])
def test_sparse_cic_lattices_go_ray_by_ray(ml, px, same):
    """Lattices of fewer than four rays a quad take the rays one by one (the runs'
    quadrature would cost more than they do): with one lane adding to a pixel at
    most, the map is the per-ray walk's; longer runs are summed, and differ in the
    last bits."""
    w = _case()
    w.map_n, w.ray_n = px, (500, 1)
    w.lenses, w.kappa_star = inputs.LensField(np.zeros(0), np.zeros(0), np.zeros(0)), 0.0
    out = []
    for walk in (ml.WALK_CERTIFIED, ml.WALK_PER_RAY):
        f = _field(ml, w, walk=walk, l1=(20.0, 1.0), l2_sub=(2, 2))
        f.shoot()
        out.append(f.mu().cpu().numpy())
        f.close()
    assert np.array_equal(out[0], out[1]) == same


def _corner_sums(mu, tracks, ns, sigma):
    """Light curves corner by corner and tap by tap in FP64 with float taps, as
    the library documents them: corners outside the map or of weight zero and
    taps outside the map are left out (so infinities elsewhere stay there)."""
    ny, nx = mu.shape
    h = int(np.floor(4 * sigma))
    t = np.exp(-0.5 * (np.arange(-h, h + 1) / sigma) ** 2)
    taps = (t / t.sum()).astype(np.float32).astype(np.float64)
    out = np.zeros((len(tracks), ns))
    for i, (x0, y0, x1, y1) in enumerate(tracks):
        for k in range(ns):
            f = k / (ns - 1) if ns > 1 else 0.0
            u, v = x0 + f * (x1 - x0) - 0.5, y0 + f * (y1 - y0) - 0.5
            i0, j0 = int(np.floor(u)), int(np.floor(v))
            for c in range(4):
                pi, pj = i0 + (c & 1), j0 + (c >> 1)
                w = (u - i0 if c & 1 else 1 - (u - i0)) * (v - j0 if c >> 1 else 1 - (v - j0))
                if not (0 <= pi < nx and 0 <= pj < ny) or w == 0:
                    continue
                xs, ys = np.arange(max(0, pi - h), min(nx, pi + h + 1)), np.arange(max(0, pj - h), min(ny, pj + h + 1))
                with np.errstate(invalid="ignore", over="ignore"):
                    rows = (mu[np.ix_(ys, xs)] * taps[xs - pi + h]).sum(1)
                    out[i, k] += w * (rows * taps[ys - pj + h]).sum()
    return out


@pytest.mark.parametrize("sigma", [0.2, 0.5, 1.9, 16.0])
@pytest.mark.parametrize("ns", [1, 3, 33])
def test_light_curves_and_transpose_over_sources_and_spacings(ml, sigma, ns):
    """Windows of 2 to 130 pixels on a 37 x 29 map, samples far apart and close
    together (33: a chunk and one more), tracks in, across and beyond the rim.
    The sums carry about 46 bits, so a curve lies within the rounding of its
    float (2^-24) and of the sums' 1e-12; the transpose is FP32: per pixel at
    most ns + 3 roundings of terms that add up to J^T |w|."""
    import torch
    rng = np.random.default_rng(3)
    mu = rng.uniform(-1.0, 3.0, (29, 37)).astype(np.float32)
    tracks = np.array([[3.0, 4.0, 30.0, 20.0], [-40.0, 5.5, 80.0, 9.5], [12.25, -3.0, 12.25, 31.0],
                       [36.9, 28.9, 37.4, 29.4], [500.0, 500.0, 501.0, 900.0], [5.5, 6.5, 7.5, 6.5]])
    m = torch.as_tensor(mu).cuda()
    out = torch.empty((len(tracks), ns), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves(m, tracks, ns, sigma, out)
    ref = _corner_sums(mu.astype(np.float64), tracks, ns, sigma)
    mag = _corner_sums(np.abs(mu).astype(np.float64), tracks, ns, sigma)
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 2.0 ** -24 * np.abs(ref) + 1e-12 * mag + 1e-45)
    w = rng.standard_normal((len(tracks), ns)).astype(np.float32)
    w[0, 0] = 0.0
    g = torch.empty((29, 37), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves_backward(torch.as_tensor(w).cuda(), tracks, ns, sigma, g)
    for _ in range(6):
        # <J e, w> = <e, J^T w> on maps of a few random pixels
        e = np.zeros((29, 37))
        at = rng.integers(0, 29), rng.integers(0, 37)
        e[at] = 1.0
        col = _corner_sums(e, tracks, ns, sigma)
        assert abs(g.cpu().numpy()[at] - (col * w).sum()) <= 2.0 ** -24 * (w.size + 3) * (col * np.abs(w)).sum() + 1e-45


@pytest.mark.parametrize("sigma", [0.74, 0.75, 2.74, 2.75])
def test_light_curves_at_the_widths_where_lanes_change(ml, sigma):
    """Windows of 6 and 8, 22 and 24 pixels: one, four and eight lanes a sample."""
    test_light_curves_and_transpose_over_sources_and_spacings(ml, sigma, 33)


@pytest.mark.parametrize("sigma,left", [(0.5, 1e-6), (4.0, 1e-6), (4.0, 1e-9)])
def test_light_curves_of_maps_that_cancel(ml, sigma, left):
    """Maps of both signs whose curves are far smaller than their values: 60 windows
    of random pixels of 1000, each with one pixel set so that the sum in 64 bits
    comes to about `left`.  The sums are those in FP64: within the rounding of the
    float they are returned in and 2^-49 of the pixels (weights add up to one, and
    FP64 sums of a thousand terms round to a few times 2^-53 of them)."""
    import torch
    rng = np.random.default_rng(4)
    h, cell, nx, ny = int(4 * sigma), 40, 10, 6
    mu = (rng.choice([-1000.0, 1000.0], (ny * cell, nx * cell))).astype(np.float32)
    at = np.array([(cell * i + 20 + rng.uniform(-1, 1), cell * j + 20 + rng.uniform(-1, 1))
                   for j in range(ny) for i in range(nx)])
    tracks = np.concatenate([at, at], 1)
    wide = mu.astype(np.float64)
    for k, (x, y) in enumerate(at):
        i, j = int(x - 0.5), int(y - 0.5)
        for px in ((i, j), (i + 1, j), (i - h, j)):
            one = np.zeros_like(wide)
            one[px[1], px[0]] = 1.0
            w = _corner_sums(one, tracks[k:k + 1], 1, sigma)[0, 0]
            wide[px[1], px[0]] = 0.0
            rest = _corner_sums(wide, tracks[k:k + 1], 1, sigma)[0, 0]
            wide[px[1], px[0]] = np.float32((left - rest) / w)
    mu = wide.astype(np.float32)
    ref = _corner_sums(wide, tracks, 1, sigma)
    assert np.abs(ref).max() < 2 * left
    out = torch.empty((len(at), 1), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves(torch.as_tensor(mu).cuda(), tracks, 1, sigma, out)
    err = np.abs(out.cpu().numpy() - ref)
    assert np.all(err <= 2.0 ** -24 * np.abs(ref) + 2.0 ** -49 * 1000.0), err.max()


def test_light_curves_of_large_counts_and_unusual_maps(ml):
    """Counts up to 2^32 - 1 (beyond 2^24 a float drops bits), and infinities,
    NaN and values near the FP32 range's ends in a float map: as the corner
    sums in FP64 give them."""
    import torch
    rng = np.random.default_rng(8)
    tracks = np.array([[2.0, 2.0, 18.0, 14.0], [10.5, 1.5, 10.5, 14.5]])
    w = inputs.Workload("counts", inputs.LensField(np.zeros(0), np.zeros(0), np.zeros(0)), 0.25, 0.25, 0.0,
                        (0.0, 0.0, 100.0), (-1.0, -1.0, 1.0, 1.0), (20, 16), ray_box=(-2.0, -1.5, 2.0, 1.5),
                        ray_n=(64, 48))
    f = ml.Field(w, precision=ml.PREC_DIRECT64)
    n = rng.integers(0, 2 ** 32, (16, 20)).astype(np.uint32)
    n[5:9, 5:9] = rng.integers(0, 1 << 23, (4, 4))
    ml.ml_field_set_counts(f.h, torch.as_tensor(n.view(np.int32)).cuda())
    got = f.light_curves(tracks, 30, 0.7).cpu().numpy()
    ref = _corner_sums(n.astype(np.float64), tracks, 30, 0.7) * f.info["mu_per_count"]
    assert np.all(np.abs(got - ref) <= 2.0 ** -23 * np.abs(ref))
    f.close()
    for value in (np.inf, -np.inf, np.nan, 3e38, 1e-40, 2e-38):
        mu = np.full((16, 20), value if abs(value) < 1e-30 else 1.0, np.float32)
        mu[7, 10] = value
        out = torch.empty((2, 30), dtype=torch.float32, device="cuda")
        ml.ml_map_light_curves(torch.as_tensor(mu).cuda(), tracks, 30, 0.7, out)
        with np.errstate(over="ignore"):
            ref = _corner_sums(mu.astype(np.float64), tracks, 30, 0.7).astype(np.float32)
        assert np.allclose(out.cpu().numpy(), ref, rtol=2.0 ** -22, atol=3e-45, equal_nan=True), value


@pytest.mark.parametrize("sigma,spacing", [(0.2, 0.3), (0.5, 60.0), (1.0, 0.1), (1.0, 9.0), (4.0, 0.5), (4.0, 17.0), (4.0, 60.0)])
@pytest.mark.parametrize("along", [(1.0, 0.001), (0.002, 1.0), (0.6, 0.8)])
def test_light_curve_transpose_gathers_or_scatters(ml, sigma, spacing, along):
    """Chunks of samples that share most of their pixels and chunks that share
    none, along and across the rows, partly outside the map: the outer products of
    each sample's weights, added up in FP64.  FP32 sums of n samples' products:
    (n + 4) 2^-24 of the sum of their sizes."""
    import torch
    rng = np.random.default_rng(6)
    ny, nx, ns, h = 700, 900, 37, int(4 * sigma)
    a = rng.uniform(-20, 200, (3, 2))
    tracks = np.concatenate([a, a + spacing * (ns - 1) * np.array(along)], 1)
    w = rng.standard_normal((3, ns)).astype(np.float32)
    t = np.exp(-0.5 * (np.arange(-h, h + 1) / sigma) ** 2)
    taps = (t / t.sum()).astype(np.float32).astype(np.float64)
    ref, size, hits = np.zeros((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx))

    def axis(c, n):
        i = int(np.floor(c))
        out = np.zeros(n + 2 * h + 4)
        for j, f in ((i, 1.0 - (c - i)), (i + 1, c - i)):
            if 0 <= j < n:
                out[j: j + 2 * h + 1] += f * taps
        return out[h: h + n]

    for k in range(3):
        for q in range(ns):
            f = q / (ns - 1)
            u = tracks[k, 0] + f * (tracks[k, 2] - tracks[k, 0]) - 0.5
            v = tracks[k, 1] + f * (tracks[k, 3] - tracks[k, 1]) - 0.5
            wy, wx = axis(v, ny), axis(u, nx)
            y, x = np.flatnonzero(wy), np.flatnonzero(wx)
            if len(y) and len(x):
                at = np.ix_(y, x)
                p = np.outer(wy[y], wx[x])
                ref[at] += float(w[k, q]) * p
                size[at] += abs(float(w[k, q])) * p
                hits[at] += 1
    g = torch.empty((ny, nx), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves_backward(torch.as_tensor(w).cuda(), tracks, ns, sigma, g)
    got = g.cpu().numpy()
    assert np.all(np.abs(got - ref) <= (hits + 4) * 2.0 ** -24 * size + 1e-45)
    assert np.all(got[hits == 0] == 0.0)


def test_light_curve_adjoint_is_the_transpose_of_the_oracle_operator(ml):
    """Brute force: the oracle's light-curve operator J (samples x pixels),
    column by column on unit maps; the GPU backward must return J^T w."""
    import torch
    mu, tracks, ns, sigma = _lc_case(nx=20, ny=14, n_tracks=3, n_samples=25)
    ny, nx = mu.shape
    J = np.zeros((len(tracks) * ns, ny * nx))
    for p in range(ny * nx):
        e = np.zeros(ny * nx)
        e[p] = 1.0
        J[:, p] = oracle.light_curves(e.reshape(ny, nx), tracks, ns, sigma).ravel()
    w = np.random.default_rng(4).standard_normal(len(tracks) * ns)
    g = torch.empty((ny, nx), dtype=torch.float32, device="cuda")
    ml.ml_map_light_curves_backward(torch.as_tensor(w.reshape(len(tracks), ns), dtype=torch.float32).cuda(),
                                    tracks, ns, sigma, g)
    ref = (J.T @ w).reshape(ny, nx)
    assert np.abs(g.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
    assert np.count_nonzero(ref) > 0


def test_light_curve_loss_gradient_matches_oracle(ml):
    """L = sum (curves - c_target)^2 with curves = LightCurves(CICMagnification):
    the autograd gradient (GPU light-curve transpose, GPU near/far adjoint)
    against the oracle's FP64 CIC gradient of the same dL/dM, where dL/dM is the
    oracle operator's transpose applied to dL/dcurves."""
    import torch
    from paper_2308_14278_gb300.autograd import CICMagnification, LightCurves
    w = _case()
    probe = _field(ml, w)
    info = probe.info
    spec = dict(sheet=w.sheet, map_box=w.map_box, map_n=w.map_n, ray_box=w.ray_box, ray_n=w.ray_n,
                taylor_p=info["taylor_p"], l1=(info["n1x"] * info["l3x"], info["n1y"] * info["l3y"]),
                l2_sub=(info["l2_sub_x"], info["l2_sub_y"]))
    probe.close()
    g = oracle.geometry_of(w, p=info["taylor_p"], l1=spec["l1"], l2_sub=info["l2_sub_x"],
                           l2_sub_y=info["l2_sub_y"])
    nx, ny = w.map_n
    rng = np.random.default_rng(9)
    tracks = np.column_stack([rng.uniform(3, nx - 3, 6), rng.uniform(3, ny - 3, 6),
                              rng.uniform(3, nx - 3, 6), rng.uniform(3, ny - 3, 6)])
    ns, sigma = 80, 0.7
    target = rng.uniform(1.0, 3.0, (6, ns))
    x = torch.tensor(w.lenses.x, requires_grad=True)
    y = torch.tensor(w.lenses.y, requires_grad=True)
    m = torch.tensor(w.lenses.m, requires_grad=True)
    par = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
           for v in (w.kappa, w.gamma, w.kappa_star)]
    mu = CICMagnification.apply(x, y, m, *par, spec)
    curves = LightCurves.apply(mu, tracks, ns, sigma)
    loss = ((curves.double() - torch.as_tensor(target).cuda()) ** 2).sum()
    loss.backward()
    # oracle: M, curves, dL/dcurves, J^T, FP64 CIC gradient
    M = oracle.cic_mu_scale(g) * oracle.cic_forward(g, w.lenses.x, w.lenses.y, w.lenses.m)
    c_ref = oracle.light_curves(M, tracks, ns, sigma)
    assert np.abs(curves.detach().cpu().numpy() - c_ref).max() <= 1e-4 * np.abs(c_ref).max()
    dl = 2.0 * (c_ref - target)
    J = np.zeros((6 * ns, ny * nx))
    for p in range(ny * nx):
        e = np.zeros(ny * nx)
        e[p] = 1.0
        J[:, p] = oracle.light_curves(e.reshape(ny, nx), tracks, ns, sigma).ravel()
    dM = (J.T @ dl.ravel()).reshape(ny, nx)
    gl, gp = oracle.cic_grad_dM(g, w.lenses.x, w.lenses.y, w.lenses.m, dM)
    got = np.column_stack([x.grad.numpy(), y.grad.numpy(), m.grad.numpy()])
    for c in range(3):
        scale = np.abs(gl[:, c]).max()
        assert np.abs(got[:, c] - gl[:, c]).max() <= 1e-3 * scale, (c, np.abs(got[:, c] - gl[:, c]).max() / scale)
    gpar = np.array([p_.grad.item() for p_ in par])
    assert np.all(np.abs(gpar - gp) <= 1e-3 * np.abs(gp)), (gpar, gp)
