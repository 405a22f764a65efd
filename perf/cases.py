"""The work a user of this library has it do, as measurable cases.

Every case goes through the public Python entry points (``LensFMM`` and its
methods, ``multiplane_ipm_map``, ``map_source`` and the autograd wrappers).  A
program that makes magnification maps draws a star field, builds a plan over
it and maps it once, so the map, halo and gradient cases build the plan inside
the pass; a program that asks one lens many questions keeps its plan, so the
ray and potential cases build it beforehand.  Fields have the shapes of
``paper_2211_00354_gb300/synth.py``, drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_00354_gb300 import autograd, lens, synth

F64 = torch.float64


# ---- the cases ---------------------------------------------------------------

def _window(npix, h=0.063, half=None):
    """Stars and sizes of a window of the high-magnification map, as
    synth.c2_window takes them."""
    half = 0.05 * npix if half is None else half
    g = synth.shooting_grid(0.45, 0.45, half, h, margin_frac=0.03,
                            margin_min=max(10.0 * h, 0.1 * half))
    rc = math.hypot(0.5 * g.nx * h, 0.5 * g.ny * h)
    return int(math.ceil(0.45 * (1.25 * rc) ** 2))


def listed():
    return [
        # The smallest whole map: 1e3 stars, 500^2 cells, 100^2 pixels (synth.c1_plain).
        # What a first script or a parameter scan of small maps runs: latency, launches.
        dict(name="plain map", kind="map", field="uniform", n=1000, kstar=0.4, ks=0.0, g=0.0,
             masses="equal", half=5.0, npix=100, h=0.04, ext=10.0, p=24, leaf=8, cap=0, refine=0,
             prec="f32"),
        # An ordinary map: 200^2 pixels of the high-magnification field (synth.c2_window),
        # the cells over the cap refined once instead of dropped.
        dict(name="map window, refined", kind="map", field="uniform", n=_window(200), kstar=0.45,
             ks=0.0, g=0.45, masses="equal", half=10.0, npix=200, h=0.063, ext=0.0, p=16, leaf=8,
             cap=64, refine=1, prec="f32"),
        # The headline workload of bench.py: 1.5e6 stars, 2000^2 pixels, 1.14e8 cells.
        dict(name="high magnification map", kind="map", field="uniform", n=1_500_000, kstar=0.45,
             ks=0.0, g=0.45, masses="equal", half=100.0, npix=2000, h=0.063, ext=0.0, p=16, leaf=8,
             cap=64, refine=0, prec="f32"),
        # Clustered lenses, masses spread over decades (bench.py --workload clustered): the
        # adaptive lists, rays few per pixel.
        dict(name="clustered map", kind="map", field="clustered", n=1_000_000, per=1000, ks=0.3,
             g=0.3, half=50.0, npix=4096, h=0.0244, p=16, leaf=64, cap=64, refine=0, prec="f32"),
        # Next to a critical curve (bench.py --workload critical): 2.2e10 cells in chunks, few
        # stars; the largest pass.
        dict(name="critical curve map", kind="map", field="critical", n=200_000, half=1.0,
             npix=8192, h=2.44e-4, p=16, leaf=4, cap=64, refine=0, prec="f32"),
        # A simulated halo: 1e7 particles, deflections on a 4096^2 grid (bench.py --workload nfw).
        dict(name="halo deflections", kind="halo", n=10_000_000, grid=4096, p=12, leaf=128,
             prec="f32"),
        # Fitting a light curve: forward and backward of the squared loss with respect to stars,
        # masses and smooth field (bench.py --workload differentiation).
        dict(name="gradient step", kind="grad", n=100_000, e1=30.0, e2=2.5, h=0.01, ns=2048,
             length=5.0, sigma=0.05, p=24, leaf=16, prec="f32"),
        # The same at the autograd wrapper's defaults: everything in float64.
        dict(name="gradient step, float64", kind="grad", n=20_000, e1=10.0, e2=1.25, h=0.02,
             ns=512, length=2.0, sigma=0.05, p=24, leaf=16, prec="f64"),
        # Ray bundles with Jacobians through a plan that is kept (image positions, shear).
        dict(name="rays with jacobian", kind="rays", n=10_000, m=20_011, kstar=0.4, ks=0.1, g=0.2,
             masses="range", p=16, leaf=16, jac=True, prec="f32"),
        # Potential (time delays) at many rays of a kept plan, float64.
        dict(name="potential", kind="potential", n=100_000, m=262_144, kstar=0.45, ks=0.0, g=0.45,
             masses="equal", p=16, leaf=8, prec="f32"),
        # Sources of finite size on a finished map (bench.py --next-rows).
        dict(name="finite source", kind="source", nx=2000, ny=2000, sigma=5.0, trunc=6.0),
        # Three lens planes (bench.py --next-rows), on the window of the second case.
        dict(name="three plane map", kind="planes", planes=3, n=_window(200), half=10.0, npix=200,
             h=0.063, p=16, leaf=8, cap=64, prec="f32"),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["plain", "window", "clustered", "critical", "halo", "grad", "rays", "potential",
                       "source", "planes"])
    if kind == "plain":
        half, npix = rng.uniform(2.0, 6.0), rng.randint(40, 250)
        return dict(kind="map", field="uniform", n=logint(300, 3000), kstar=0.4, ks=0.0, g=0.0,
                    masses=rng.choice(["equal", "range"]), half=half, npix=npix,
                    h=0.8 * half / npix * rng.uniform(0.5, 1.0), ext=2.0 * half, p=24,
                    leaf=rng.randint(6, 16), cap=0, refine=0, prec=rng.choice(["f32", "f32", "f64"]))
    if kind == "window":
        npix = logint(50, 1200)
        f64 = npix < 250 and rng.random() < 0.3
        h = rng.uniform(0.05, 0.1)
        half = 0.05 * npix
        return dict(kind="map", field="uniform", n=_window(npix, h, half), kstar=0.45, ks=0.0,
                    g=0.45, masses=rng.choice(["equal", "range"]), half=half, npix=npix, h=h,
                    ext=0.0, p=32 if f64 else rng.choice([16, 16, 20, 24]), leaf=rng.randint(4, 16),
                    cap=64, refine=rng.choice([0, 0, 0, 1]), prec="f64" if f64 else "f32")
    if kind == "clustered":
        k, per = logint(20, 1000), logint(100, 1000)
        npix = logint(300, 4096)
        return dict(kind="map", field="clustered", n=k * per, per=per, ks=0.3, g=0.3,
                    half=50.0 * npix / 4096, npix=npix, h=0.0244, p=16,
                    leaf=rng.choice([16, 32, 64]), cap=64, refine=rng.choice([0, 0, 1]), prec="f32")
    if kind == "critical":
        # like the listed one, a cell of about one pixel's side; a window much smaller than
        # this would be missed by rays that its stars deflect by ~0.3
        npix, half = logint(256, 3000), rng.uniform(0.7, 1.0)
        return dict(kind="map", field="critical", n=logint(20_000, 200_000), half=half, npix=npix,
                    h=2.0 * half / npix * rng.uniform(1.0, 2.0), p=16, leaf=rng.choice([4, 8]),
                    cap=64, refine=0, prec="f32")
    if kind == "halo":
        return dict(kind="halo", n=logint(50_000, 10_000_000), grid=logint(200, 4096),
                    p=rng.choice([12, 12, 16]), leaf=rng.choice([32, 64, 128]), prec="f32")
    if kind == "grad":
        f64 = rng.random() < 0.4
        e1 = rng.uniform(4.0, 12.0) if f64 else rng.uniform(6.0, 30.0)
        return dict(kind="grad", n=logint(2000, 20_000 if f64 else 100_000), e1=e1,
                    e2=rng.uniform(0.8, 1.25 if f64 else 2.5), h=rng.uniform(0.02, 0.03) if f64
                    else rng.uniform(0.01, 0.02), ns=logint(64, 512 if f64 else 2048),
                    length=rng.uniform(1.0, 2.0), sigma=rng.uniform(0.03, 0.1),
                    p=rng.choice([24, 24, 32]), leaf=rng.choice([8, 16, 24]),
                    prec="f64" if f64 else "f32")
    if kind == "rays":
        return dict(kind="rays", n=logint(500, 300_000), m=logint(100, 1_000_000), kstar=0.4,
                    ks=0.1, g=0.2, masses=rng.choice(["equal", "range"]),
                    p=rng.choice([16, 20, 24, 32]), leaf=rng.randint(8, 32),
                    jac=rng.random() < 0.5, prec=rng.choice(["f32", "f32", "f64"]))
    if kind == "potential":
        return dict(kind="potential", n=logint(2000, 300_000), m=logint(1000, 500_000), kstar=0.45,
                    ks=0.0, g=0.45, masses=rng.choice(["equal", "range"]), p=16,
                    leaf=rng.randint(8, 16), prec=rng.choice(["f32", "f64"]))
    if kind == "source":
        return dict(kind="source", nx=logint(150, 2500), ny=logint(150, 1600),
                    sigma=math.exp(rng.uniform(math.log(0.6), math.log(6.0))),
                    trunc=rng.uniform(4.0, 6.0))
    npix = logint(60, 300)
    return dict(kind="planes", planes=rng.randint(2, 4), n=_window(npix), half=0.05 * npix,
                npix=npix, h=0.063, p=16, leaf=rng.randint(6, 16), cap=64, prec="f32")


# ---- inputs ------------------------------------------------------------------

def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, dtype=F64, device="cuda")


def _polar(r, t):
    return torch.stack([r * torch.cos(t), r * torch.sin(t)], dim=1)


def _disk(gen, n, radius):
    return _polar(radius * torch.sqrt(_rand(gen, n)), 2.0 * math.pi * _rand(gen, n))


def _uniform(gen, n, kstar, masses, lo=0.5, hi=1.5):
    m = (torch.ones(n, dtype=F64, device="cuda") if masses == "equal"
         else lo + (hi - lo) * _rand(gen, n))
    mean = 1.0 if masses == "equal" else 0.5 * (lo + hi)
    return _disk(gen, n, math.sqrt(n * mean / kstar)), m


def _clustered(gen, n, per, a=0.5, trunc=20.0, kstar=0.2):
    m = torch.exp(torch.randn(n, generator=gen, dtype=F64, device="cuda"))
    centres = _disk(gen, n // per, math.sqrt(n * math.exp(0.5) / kstar))
    u = _rand(gen, n) * (trunc * trunc / (1.0 + trunc * trunc))
    return (centres.repeat_interleave(per, dim=0)
            + _polar(a * torch.sqrt(u / (1.0 - u)), 2.0 * math.pi * _rand(gen, n))), m


def _halo(gen, n, q=0.7, c=10.0):
    """Elliptical NFW halo (synth.nfw_halo): radii by interpolating the
    inverse of the enclosed-mass profile."""
    tab = torch.linspace(0.0, 1.0, 1 << 20, dtype=F64, device="cuda") ** 2 * c
    cdf = torch.log1p(tab) - tab / (1.0 + tab)
    t = _rand(gen, n) * cdf[-1]
    i = torch.searchsorted(cdf, t).clamp_(1, cdf.numel() - 1)
    r = tab[i - 1] + (t - cdf[i - 1]) / (cdf[i] - cdf[i - 1]) * (tab[i] - tab[i - 1])
    cz, ph = 2.0 * _rand(gen, n) - 1.0, 2.0 * math.pi * _rand(gen, n)
    xy = _polar(r * torch.sqrt(1.0 - cz * cz), ph)
    xy[:, 1] *= q
    inside = ((xy.abs() <= 2.0).all(dim=1)).to(F64).mean()
    return xy, (16.0 / math.pi / inside / n).repeat(n).contiguous()


def _grid(case):
    if case["kind"] == "planes" or case["field"] == "uniform":
        if case.get("ext"):
            return synth.shooting_grid(0.0, 0.0, case["half"], case["h"],
                                       half_extent=(case["ext"], case["ext"]))
        return synth.shooting_grid(0.45, 0.45, case["half"], case["h"], margin_frac=0.03,
                                   margin_min=max(10.0 * case["h"], 0.1 * case["half"]))
    if case["field"] == "clustered":
        return synth.shooting_grid(0.5, 0.3, case["half"], case["h"], margin_frac=0.03,
                                   margin_min=5.0)
    return synth.shooting_grid(0.82, 0.17, case["half"], case["h"], margin_frac=0.03,
                               margin_min=0.3)


def _target(g):
    return (g.x0, g.x0 + g.nx * g.h, g.y0, g.y0 + g.ny * g.h)


def _smooth(case):
    return (0.81, 0.17) if case.get("field") == "critical" else (case["ks"], case["g"])


def _map_field(case, seed):
    gen = _gen(seed)
    if case["field"] == "clustered":
        return _clustered(gen, case["n"], case["per"])
    if case["field"] == "critical":
        return _uniform(gen, case["n"], 0.01, "range", 0.1, 1.0)
    return _uniform(gen, case["n"], case["kstar"], case["masses"])


def _plane_set(case, seed):
    """The window's stars dealt to the planes, the shear on the nearest; the
    distance ratios grow with the separation of the planes."""
    stars, masses = _uniform(_gen(seed), case["n"], 0.45, "equal")
    K = case["planes"]
    beta = [[0.2 * (j - i) * (1.0 - 0.06 * (j - i)) if j > i else 0.0 for j in range(K)]
            for i in range(K)]
    return [(stars[k::K].contiguous(), masses[k::K].contiguous(), 0.0, 0.45 if k == 0 else 0.0)
            for k in range(K)], beta


def _region(case):
    """Rays of the kept-plan cases lie in the inner half of the star disk."""
    r = 0.5 * math.sqrt(case["n"] / case["kstar"])
    return (-r, r, -0.5 * r, 0.5 * r)


def _ray_inputs(case, seed):
    gen = _gen(seed)
    stars, masses = _uniform(gen, case["n"], case["kstar"], case["masses"])
    t = _region(case)
    u = _rand(gen, case["m"], 2)
    lo = torch.tensor([t[0], t[2]], dtype=F64, device="cuda")
    hi = torch.tensor([t[1], t[3]], dtype=F64, device="cuda")
    return stars, masses, lo + (hi - lo) * u


def _grad_inputs(case, seed):
    """Stars, masses, grid rays, track samples and the observed curve."""
    gen = _gen(seed)
    stars, masses = _uniform(gen, case["n"], 0.3, "range")
    h = case["h"]
    nx, ny = int(round(2 * case["e1"] / h)), int(round(2 * case["e2"] / h))
    x = -case["e1"] + h * torch.arange(nx + 1, dtype=F64, device="cuda")
    y = -case["e2"] + h * torch.arange(ny + 1, dtype=F64, device="cuda")
    rays = torch.stack([x[None, :].expand(ny + 1, -1), y[:, None].expand(-1, nx + 1)],
                       dim=2).reshape(-1, 2).contiguous()
    track = torch.tensor(synth.light_curve_track(case["ns"], length=case["length"]), device="cuda")
    s = torch.linspace(0.0, 1.0, case["ns"], dtype=F64, device="cuda")
    ph = 2.0 * math.pi * _rand(gen, 2)
    target = 4.0 * (1.0 + 0.4 * torch.sin(9.0 * s + ph[0]) + 0.2 * torch.sin(31.0 * s + ph[1]))
    box = (-case["e1"], float(x[-1]), -case["e2"], float(y[-1]))
    return stars, masses, rays, track, target, box


def _image(case, seed):
    """A map like a caustic network: positive, smooth on a few pixels with a long tail."""
    gen = _gen(seed)
    a = torch.randn((case["ny"], case["nx"]), generator=gen, dtype=F64, device="cuda")
    for d in (0, 1):
        a = a + a.roll(1, d) + a.roll(2, d) + a.roll(3, d)
    return 5.0 * torch.exp(0.25 * a)


_PREC = {"f32": lens.FP32_BULK, "f64": lens.FP64}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "map":
        stars, masses = _map_field(case, seed)
        return dict(case=case, stars=stars, masses=masses, grid=_grid(case))
    if kind == "halo":
        stars, masses = _halo(_gen(seed), case["n"])
        k = case["grid"]
        return dict(case=case, stars=stars, masses=masses,
                    grid=synth.Grid(x0=-2.0, y0=-2.0, h=4.0 / k, nx=k - 1, ny=k - 1))
    if kind == "grad":
        return dict(case=case, data=_grad_inputs(case, seed))
    if kind in ("rays", "potential"):
        stars, masses, rays = _ray_inputs(case, seed)
        plan = lens.LensFMM(stars, masses, case["ks"], case["g"], p=case["p"],
                            leaf_size=case["leaf"], prec=_PREC[case["prec"]],
                            target_box=_region(case))
        return dict(case=case, plan=plan, rays=rays)
    if kind == "source":
        return dict(case=case, map=_image(case, seed))
    planes, beta = _plane_set(case, seed)
    return dict(case=case, planes=planes, beta=beta, grid=_grid(case))


# ---- one pass ----------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "map":
        ks, g = _smooth(case)
        grid, half = state["grid"], case["half"]
        with lens.LensFMM(state["stars"], state["masses"], ks, g, p=case["p"],
                          leaf_size=case["leaf"], prec=_PREC[case["prec"]],
                          target_box=_target(grid)) as plan:
            mp, _ = plan.ipm_map(grid, (-half, half, -half, half), case["npix"], case["npix"],
                                 bbox_cap=case["cap"], refine_levels=case["refine"])
        return mp
    if kind == "halo":
        grid = state["grid"]
        with lens.LensFMM(state["stars"], state["masses"], 0.0, 0.0, p=case["p"],
                          leaf_size=case["leaf"], prec=_PREC[case["prec"]],
                          target_box=_target(grid)) as plan:
            return plan.deflect_grid(grid)
    if kind == "grad":
        stars, masses, rays, track, target, box = state["data"]
        stars = stars.detach().requires_grad_(True)
        masses = masses.detach().requires_grad_(True)
        y = autograd.deflect(stars, masses, 0.2, 0.4, rays, p=case["p"], leaf_size=case["leaf"],
                             prec=_PREC[case["prec"]], target_box=box)
        F = autograd.light_curve(y, case["h"] ** 2, track, case["sigma"])
        ((F - target) ** 2).sum().backward()
        return [F.detach(), stars.grad, masses.grad]
    if kind == "rays":
        if case["jac"]:
            return list(state["plan"].deflect(state["rays"], jacobian=True))
        return [state["plan"].deflect(state["rays"])]
    if kind == "potential":
        return state["plan"].potential(state["rays"])
    if kind == "source":
        return lens.map_source(state["map"], case["sigma"], case["trunc"])
    half = case["half"]
    mp, _ = lens.multiplane_ipm_map(state["planes"], state["beta"], state["grid"],
                                    (-half, half, -half, half), case["npix"], case["npix"],
                                    p=case["p"], leaf_size=case["leaf"],
                                    prec=_PREC[case["prec"]], bbox_cap=case["cap"])
    return mp


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Bytes: inputs once, outputs once.  Flops: per ray an order-p local
    expansion (8 (p+1)) and about nine leaves of half-full near stars (10 a
    pair), per cell about 60 for its polygon, per star 8 (p+1) for its
    multipole; the other kinds beside their formulas."""
    kind = case["kind"]
    if kind == "source":
        npix = case["nx"] * case["ny"]
        return {"bytes": 16.0 * npix,
                "flops": 2.0 * math.pi * (case["trunc"] * case["sigma"]) ** 2 * npix}
    n, p, leaf = case["n"], case["p"], case["leaf"]
    per_ray = 8.0 * (p + 1) + 10.0 * min(n, 4.5 * leaf)
    tree = 8.0 * (p + 1) * n
    if kind in ("map", "planes"):
        g = _grid(case)
        K = case.get("planes", 1)
        return {"bytes": 24.0 * n + 8.0 * case["npix"] ** 2,
                "flops": tree + g.n_rays * per_ray * K + 60.0 * g.n_cells}
    if kind == "halo":
        rays = case["grid"] ** 2
        return {"bytes": 24.0 * n + 16.0 * rays, "flops": tree + rays * per_ray}
    if kind == "grad":
        rays = (2 * case["e1"] / case["h"] + 1) * (2 * case["e2"] / case["h"] + 1)
        # forward and the transposed pass; stars, masses, rays in, curve and gradients out
        return {"bytes": 48.0 * n + 16.0 * rays + 32.0 * case["ns"],
                "flops": 2.0 * tree + 2.5 * rays * per_ray}
    m = case["m"]
    out = 8.0 if kind == "potential" else 48.0 if case["jac"] else 16.0
    return {"bytes": (16.0 + out) * m, "flops": m * per_ray * (2.0 if case.get("jac") else 1.0)}


# ---- the same in 64 bits -----------------------------------------------------

_PAIRS = 1 << 25  # ray-star pairs at a time


def _chunks(m, n):
    step = max(1, _PAIRS // max(n, 1))
    return [(a, min(m, a + step)) for a in range(0, m, step)]


def _star_sum(x, stars, masses, jac=False):
    """sum_i m_i d / |d|^2 at every ray (a star exactly at a ray adds nothing)
    and its derivatives (S11, S12; S22 = -S11)."""
    out = torch.empty_like(x)
    J = torch.empty_like(x) if jac else None
    for a, b in _chunks(x.shape[0], stars.shape[0]):
        d1 = x[a:b, 0, None] - stars[None, :, 0]
        d2 = x[a:b, 1, None] - stars[None, :, 1]
        r2 = d1 * d1 + d2 * d2
        inv = torch.where(r2 > 0, 1.0 / r2, torch.zeros_like(r2))
        w = masses * inv
        out[a:b, 0] = (w * d1).sum(1)
        out[a:b, 1] = (w * d2).sum(1)
        if jac:
            w = w * inv
            J[a:b, 0] = (w * (d2 - d1) * (d2 + d1)).sum(1)
            J[a:b, 1] = (-2.0 * w * d1 * d2).sum(1)
    return (out, J) if jac else out


def _lens_equation(x, stars, masses, ks, g):
    al = _star_sum(x, stars, masses)
    return torch.stack([(1.0 - ks - g) * x[:, 0] - al[:, 0], (1.0 - ks + g) * x[:, 1] - al[:, 1]], 1)


def _overlaps(mp, q, weight, area):
    """Adds cells q (k, 4, 2) in pixel units to the map: weight * (signed
    area in the pixel) / (signed area), by Green's theorem per edge."""
    ny, nx = mp.shape
    A = 0.5 * ((q[:, 2, 0] - q[:, 0, 0]) * (q[:, 3, 1] - q[:, 1, 1])
               - (q[:, 3, 0] - q[:, 1, 0]) * (q[:, 2, 1] - q[:, 0, 1]))
    lo, hi = torch.floor(q.amin(1)).long(), torch.floor(q.amax(1)).long()
    x0, x1 = lo[:, 0].clamp(min=0), hi[:, 0].clamp(max=nx - 1)
    y0, y1 = lo[:, 1].clamp(min=0), hi[:, 1].clamp(max=ny - 1)
    wd = x1 - x0 + 1
    npx = wd.clamp(min=0) * (y1 - y0 + 1).clamp(min=0)
    npx = torch.where(A.abs() > 1e-14 * area, npx, torch.zeros_like(npx))
    keep = (npx > 0).nonzero()[:, 0]
    q, A, x0, y0, wd, npx = q[keep], A[keep], x0[keep], y0[keep], wd[keep], npx[keep]
    ends = npx.cumsum(0)
    a = 0
    while a < q.shape[0]:
        base = int(ends[a - 1]) if a else 0
        b = max(a + 1, int(torch.searchsorted(ends, base + (1 << 22))))
        cell = torch.repeat_interleave(torch.arange(a, b, device=q.device), npx[a:b])
        k = torch.arange(cell.numel(), device=q.device) - (ends[cell] - npx[cell] - base)
        px, py = x0[cell] + k % wd[cell], y0[cell] + k // wd[cell]
        s = torch.zeros_like(A[cell])
        for e in range(4):
            e0, e1 = q[cell, e], q[cell, (e + 1) & 3]
            ey = e1[:, 1] - e0[:, 1]
            slope = torch.where(ey != 0, (e1[:, 0] - e0[:, 0]) / torch.where(ey != 0, ey, torch.ones_like(ey)),
                                torch.zeros_like(ey))
            ya = torch.minimum(torch.maximum(e0[:, 1], py.to(F64)), py + 1.0)
            yb = torch.minimum(torch.maximum(e1[:, 1], py.to(F64)), py + 1.0)
            xa = e0[:, 0] + (ya - e0[:, 1]) * slope - px
            xb = e0[:, 0] + (yb - e0[:, 1]) * slope - px
            u, v = torch.minimum(xa, xb), torch.maximum(xa, xb)
            uc, vc = u.clamp(0.0, 1.0), v.clamp(0.0, 1.0)
            num = 0.5 * (vc - uc) * (vc + uc) + (v - v.clamp(max=1.0)) - (u - u.clamp(max=1.0))
            flat = v - u < 1e-12
            mean = torch.where(flat, (0.5 * (u + v)).clamp(0.0, 1.0),
                               num / torch.where(flat, torch.ones_like(u), v - u))
            s = s + (yb - ya) * mean
        mp.view(-1).index_add_(0, py * nx + px, weight * s / A[cell])
        a = b


def _map_exact(stars, masses, ks, g, grid, half, npix):
    """First-order IPM of the grid, no cell dropped."""
    pix = 2.0 * half / npix
    mp = torch.zeros((npix, npix), dtype=F64, device="cuda")
    c = torch.tensor(grid.corners().reshape(-1, 2), device="cuda")
    y = (_lens_equation(c, stars, masses, ks, g).reshape(grid.ny + 1, grid.nx + 1, 2) + half) / pix
    q = torch.stack([y[:-1, :-1], y[:-1, 1:], y[1:, 1:], y[1:, :-1]], 2).reshape(-1, 4, 2)
    meets = ((q.amax(1) >= 0) & (torch.floor(q.amin(1)) <= npix - 1)).all(1)
    area = (grid.h / pix) ** 2
    _overlaps(mp, q[meets], area, area)
    return mp


def exact(case, seed):
    kind = case["kind"]
    if kind == "planes" or kind == "map" and not case.get("ext"):
        # A first-order map divides by the signed area of nearly folded cells: at high
        # magnification a few such pixels hold most of the norm, and the rounding of the
        # corners decides them.  The plain map is free of that.
        return None
    if kind == "map":
        stars, masses = _map_field(case, seed)
        return _map_exact(stars, masses, case["ks"], case["g"], _grid(case), case["half"],
                          case["npix"])
    if kind == "halo":
        if case["n"] * float(case["grid"]) ** 2 > 3e10:
            return None
        stars, masses = _halo(_gen(seed), case["n"])
        k = case["grid"]
        x = torch.tensor(synth.Grid(-2.0, -2.0, 4.0 / k, k - 1, k - 1).corners().reshape(-1, 2),
                         device="cuda")
        return _lens_equation(x, stars, masses, 0.0, 0.0).reshape(k, k, 2)
    if kind == "grad":
        stars, masses, rays, track, target, _ = _grad_inputs(case, seed)
        if stars.shape[0] * float(rays.shape[0]) > 3e10:
            return None
        y = _lens_equation(rays, stars, masses, 0.2, 0.4)
        s2, cut = case["sigma"] ** 2, (6.0 * case["sigma"]) ** 2
        norm = case["h"] ** 2 / (2.0 * math.pi * s2)
        F = torch.zeros_like(target)
        gy = torch.zeros_like(y)
        for second in (False, True):  # the curve, then dL/dy
            for a, b in _chunks(y.shape[0], track.shape[0]):
                d = y[a:b, None, :] - track[None]
                q = (d * d).sum(2)
                G = torch.where(q <= cut, norm * torch.exp(-q / (2.0 * s2)), torch.zeros_like(q))
                if second:
                    gy[a:b] = ((2.0 * (F - target) * G)[..., None] * (-d / s2)).sum(1)
                else:
                    F += G.sum(0)
        # dL/dm_i = -sum_r g.d/|d|^2, dL/dx_i = sum_r m_i (g/|d|^2 - 2 d (g.d)/|d|^4)
        gs, gm = torch.zeros_like(stars), torch.zeros_like(masses)
        for a, b in _chunks(rays.shape[0], stars.shape[0]):
            d1 = rays[a:b, 0, None] - stars[None, :, 0]
            d2 = rays[a:b, 1, None] - stars[None, :, 1]
            r2 = d1 * d1 + d2 * d2
            inv = torch.where(r2 > 0, 1.0 / r2, torch.zeros_like(r2))
            g1, g2 = gy[a:b, 0, None], gy[a:b, 1, None]
            gd = (g1 * d1 + g2 * d2) * inv
            gm -= gd.sum(0)
            gs[:, 0] += ((g1 - 2.0 * d1 * gd) * inv).sum(0)
            gs[:, 1] += ((g2 - 2.0 * d2 * gd) * inv).sum(0)
        return [F, gs * masses[:, None], gm]
    if kind in ("rays", "potential"):
        if case["n"] * float(case["m"]) > 5e10:
            return None
        stars, masses, x = _ray_inputs(case, seed)
        ks, g = case["ks"], case["g"]
        if kind == "potential":
            psi = 0.5 * ks * (x * x).sum(1) + 0.5 * g * (x[:, 0] ** 2 - x[:, 1] ** 2)
            for a, b in _chunks(x.shape[0], stars.shape[0]):
                r2 = ((x[a:b, 0, None] - stars[None, :, 0]) ** 2
                      + (x[a:b, 1, None] - stars[None, :, 1]) ** 2)
                psi[a:b] += (masses * torch.where(r2 > 0, 0.5 * torch.log(r2),
                                                  torch.zeros_like(r2))).sum(1)
            return psi
        y = _lens_equation(x, stars, masses, ks, g)
        if not case["jac"]:
            return [y]
        _, S = _star_sum(x, stars, masses, jac=True)
        a, b = 1.0 - ks - g, 1.0 - ks + g
        return [y, torch.stack([a - S[:, 0], -S[:, 1], -S[:, 1], b + S[:, 0]], 1).reshape(-1, 2, 2)]
    # the disk |d| <= trunc sigma of the Gaussian, renormalised inside the map
    m, sig = _image(case, seed), case["sigma"]
    R = int(math.floor(case["trunc"] * sig))
    cut = case["trunc"] * case["trunc"] * sig * sig
    num, den = torch.zeros_like(m), torch.zeros_like(m)
    ny, nx = m.shape
    for dy in range(-R, R + 1):
        for dx in range(-R, R + 1):
            if dx * dx + dy * dy > cut or abs(dy) >= ny or abs(dx) >= nx:
                continue
            w = math.exp(-(dx * dx + dy * dy) / (2.0 * sig * sig))
            ys, xs = slice(max(0, -dy), ny - max(0, dy)), slice(max(0, -dx), nx - max(0, dx))
            yd, xd = slice(max(0, dy), ny - max(0, -dy)), slice(max(0, dx), nx - max(0, -dx))
            num[ys, xs] += w * m[yd, xd]
            den[ys, xs] += w
    return num / den
