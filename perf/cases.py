"""Timed cases of the library: what its users have it do, through its public
entry points.

A case is a sky scene (sources, exposures, patches) and one call on it:

* ``derivatives``  ELBO, gradient and Hessian of every source (elbo_grad_hess)
* ``newton``       one trust-region pass over the colour classes (newton_step)
* ``gradient``     the autograd objective: value, then backward
* ``loglik``       a round of the sampler: all chains' log-likelihoods
* ``render``       own moments and neighbour backgrounds of every patch
* ``field_elbo``   the ELBO of whole images
* ``fit``          a region fit to convergence
* ``steps``        trust-region subproblems of independent sources

Scenes are drawn on the GPU with the distributions of ``fields`` (fluxes,
shapes, PSFs, skies, patch sizes).  Layouts: ``field``, one set of images with
sources at uniform positions; ``blends``, groups of 1..11 sources inside each
other's patches, every group with its own exposures; ``cutout``, a source in
images no larger than its patch.
"""
import dataclasses
import math

import numpy as np
import torch

import fields
from paper_1803_00113_gb300 import celeste as cel
from paper_1803_00113_gb300.autograd import SourceObjective
from paper_1803_00113_gb300.mcmc import GpuLogLik

BANDS = fields.N_BANDS
NT = fields.N_THETA


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one detection re-evaluated on its cutouts (interactive use, unit of latency)
        dict(name="cutout_derivatives", call="derivatives", layout="cutout", sources=1, side=41,
             per_band=1),
        # the same source's Newton iteration: the smallest step of a fit
        dict(name="cutout_newton", call="newton", layout="cutout", sources=1, side=41, per_band=1),
        # a small request of the fitting service, from start to converged catalogue
        dict(name="request_fit", call="fit", layout="field", sources=8, height=120, width=120,
             per_band=2),
        # a large request: many classes, several exposures a band
        dict(name="region_fit", call="fit", layout="field", sources=56, height=419, width=419,
             per_band=3, cache=True),
        # the field's sources in one Newton pass (neighbours rendered again)
        dict(name="field_newton", call="newton", layout="field", sources=600, height=2048,
             width=1489, per_band=1),
        # an optimiser of the user's own on the autograd objective
        dict(name="field_gradient", call="gradient", layout="field", sources=1024, height=2048,
             width=1489, per_band=1),
        # convergence check of a field: every pixel of every image
        dict(name="field_elbo", call="field_elbo", layout="field", sources=600, height=2048,
             width=1489, per_band=1),
        # posterior curvatures (uncertainties) of blended sources
        dict(name="blend_derivatives", call="derivatives", layout="blends", sources=300,
             per_band=6),
        # model images for residual plots and masks
        dict(name="blend_render", call="render", layout="blends", sources=500, per_band=4),
        # one round of the sampler: 16 sources, 25 chains for each of two types
        dict(name="chains_loglik", call="loglik", layout="field", sources=200, height=1024,
             width=745, per_band=1, sampled=16, chains=50),
        # the trust-region solver on a user's own quadratic models
        dict(name="steps", call="steps", problems=4096),
        # the survey's bulk work: thousands of blended sources, cached renders
        dict(name="batched_newton", call="newton", layout="blends", sources=8192, per_band=6,
             cache=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def odd(lo, hi):
        return log_int(lo, hi) | 1

    call = rng.choice(["derivatives", "newton", "newton", "gradient", "loglik", "render",
                       "field_elbo", "fit", "steps"])
    if call == "steps":
        return dict(call=call, problems=log_int(1, 8192))
    case = dict(call=call)
    layout = {"field_elbo": ["field"], "fit": ["field"], "loglik": ["field"],
              "gradient": ["field", "blends"]}.get(call, ["field", "blends", "cutout"])
    case["layout"] = rng.choice(layout)
    if call == "fit":
        side = log_int(32, 512)
        case.update(sources=log_int(1, 64), height=side, width=side, per_band=rng.randint(1, 4),
                    cache=rng.random() < 0.5)
    elif case["layout"] == "cutout":
        case.update(sources=1, side=odd(15, 101), per_band=rng.randint(1, 6))
    elif case["layout"] == "field":
        case.update(sources=log_int(20, 1200), height=log_int(256, 2048), width=log_int(256, 1489),
                    per_band=rng.randint(1, 2))
    else:
        case.update(sources=log_int(12, 2500 if call == "newton" else 500),
                    per_band=rng.randint(1, 6))
    if call == "newton" and case["layout"] == "blends":
        case["cache"] = rng.random() < 0.7
    if call == "loglik":
        case.update(sampled=min(rng.randint(1, 24), case["sources"]), chains=2 * rng.randint(4, 40))
    if rng.random() < 0.2:
        # shorter galaxy mixtures
        case.update(n_exp=rng.randint(3, 8), n_dev=rng.randint(3, 8))
    return case


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------

def _model(case):
    m = fields.make_model()
    for key, a, t in (("n_exp", "alpha_exp", "tau_exp"), ("n_dev", "alpha_dev", "tau_dev")):
        n = case.get(key)
        if n and n < len(getattr(m, a)):
            alpha = getattr(m, a)[-n:]
            m = dataclasses.replace(m, **{a: alpha / alpha.sum(), t: getattr(m, t)[-n:]})
    return m


def _spread(counts):
    """(owner, index within the owner) of counts[i] items per owner i."""
    owner = np.repeat(np.arange(len(counts)), counts)
    first = np.cumsum(counts) - counts
    return owner, np.arange(len(owner)) - first[owner]


_SEL = np.array([[-1, -1, 0, 0], [0, -1, 0, 0], [0, 0, 0, 0], [0, 0, 1, 0], [0, 0, 1, 1]], float)


def _rot(phi):
    c, s = np.cos(phi), np.sin(phi)
    return np.stack([np.stack([c, -s], -1), np.stack([s, c], -1)], -2)


def _geometry(case, seed):
    """Everything of a scene but its pixels; a fields.Problem and the truth."""
    rng = np.random.default_rng([int(seed), 1803])
    model = _model(case)
    n = case["sources"]
    layout, mx = case["layout"], case["per_band"]
    # the case alone fixes the sizes (patches, groups, exposures): shape
    shape = np.random.default_rng([n, mx, 13])
    logr = shape.normal(math.log(5.0), 1.2, n)
    star = shape.uniform(size=n) < 0.3
    colors = np.where(star[:, None], [0.9, 0.4, 0.15, 0.08], [1.2, 0.6, 0.35, 0.3]) \
        + shape.normal(0, 0.25, (n, 4))
    radius = np.exp(shape.normal(math.log(1.5), 0.5, n))
    axis, angle = rng.uniform(0.2, 1.0, n), rng.uniform(0, math.pi, n)
    prof = rng.uniform(0.02, 0.98, n)
    var = np.where(star, 0.0, radius ** 2 / (2 * math.log(2.0)))
    Rs = _rot(angle)
    D = np.zeros((n, 2, 2))
    D[:, 0, 0], D[:, 1, 1] = var, var * axis ** 2
    cov = np.swapaxes(Rs, 1, 2) @ D @ Rs
    flux = np.exp(logr[:, None] + colors @ _SEL.T)                     # [n, band]
    # patch sides, groups, positions
    if layout == "blends":
        sizes = []
        while sum(sizes) < n:
            sizes.append(min(int(shape.integers(1, 12)), n - sum(sizes)))
        sizes = np.array(sizes)
        group, _ = _spread(sizes)
        side = np.minimum(np.round(np.exp(shape.uniform(math.log(15), math.log(101), n))).astype(int) | 1, 101)
        lo = np.minimum.reduceat(side, np.cumsum(sizes) - sizes)
        hi = np.maximum.reduceat(side, np.cumsum(sizes) - sizes)
        spread = 0.35 * lo
        gh = gw = hi + (2 * spread).astype(int) + 8
        pos = (gh / 2.0)[group][:, None] + spread[group][:, None] * rng.uniform(-1, 1, (n, 2))
        counts = shape.integers(1, mx + 1, (len(sizes), BANDS))
    else:
        sizes, group = np.array([n]), np.zeros(n, int)
        if layout == "cutout":
            side = np.full(n, case["side"])
            gh = gw = np.array([case["side"]])
            pos = (case["side"] - 1) / 2.0 + rng.uniform(-0.5, 0.5, (n, 2))
        else:
            gh, gw = np.array([case["height"]]), np.array([case["width"]])
            pos = np.column_stack([rng.uniform(3, gw[0] - 4, n), rng.uniform(3, gh[0] - 4, n)])
            # odd side covering where the noiseless source exceeds 0.2 sqrt(sky)
            sig2 = 16.0 + var
            peak = 220.0 * flux.max(1) / (2 * math.pi * sig2) / (0.2 * math.sqrt(50.0))
            reach = np.sqrt(2 * sig2 * np.log(np.maximum(peak, 1.0)))
            side = np.clip(2 * np.ceil(reach).astype(int) + 1, 15, 101)
        counts = np.full((1, BANDS), mx)
    # images, group by group and band by band
    ig, _ = _spread(counts.sum(1))
    band = np.concatenate([np.repeat(np.arange(BANDS), c) for c in counts])
    ni = len(ig)
    ih, iw = gh[ig], gw[ig]
    A = _rot(rng.uniform(-0.004, 0.004, ni)) * (1 + rng.uniform(-0.002, 0.002, (ni, 1, 2)))
    t = rng.uniform(-1.5, 1.5, (ni, 2))
    if layout == "cutout":                       # the cutout is centred on the source
        t = pos[0] - A @ pos[0]
    psf = np.zeros((ni, 3, 6))
    psf[:, :, 0] = -np.sort(-rng.dirichlet([4.0, 2.0, 1.0], ni), 1)
    sig = rng.uniform([1.0, 1.6, 2.5], [1.6, 2.5, 4.0], (ni, 3))
    ell, phi = rng.uniform(0, 0.08, (ni, 3)), rng.uniform(0, math.pi, (ni, 3))
    E = np.zeros((ni, 3, 2, 2))
    E[..., 0, 0], E[..., 1, 1] = (sig * (1 + ell)) ** 2, (sig * (1 - ell)) ** 2
    C = _rot(phi) @ E @ np.swapaxes(_rot(phi), -1, -2)
    psf[:, :, 3], psf[:, :, 4], psf[:, :, 5] = C[..., 0, 0], C[..., 0, 1], C[..., 1, 1]
    ky, kx = (4, 3) if layout == "field" and max(gh[0], gw[0]) > 512 else (1, 1)
    sky = rng.uniform(50, 200, (ni, 1, 1)) * (1 + (rng.uniform(-0.05, 0.05, (ni, ky, kx)) if ky > 1 else 0))
    # patches, source by source, one per image of the source's group
    m = counts.sum(1)
    first = np.cumsum(m) - m
    ps, k = _spread(m[group])
    pimg = first[group[ps]] + k
    c = np.einsum("pij,pj->pi", A[pimg], pos[ps]) + t[pimg]
    w, h = np.minimum(side[ps], iw[pimg]), np.minimum(side[ps], ih[pimg])
    x0 = np.clip(np.round(c[:, 0]).astype(int) - w // 2, 0, iw[pimg] - w)
    y0 = np.clip(np.round(c[:, 1]).astype(int) - h // 2, 0, ih[pimg] - h)
    ptr = np.concatenate([[0], np.cumsum(m[group])])
    # neighbours: sources of a group whose patches overlap in one of its images
    g0 = np.cumsum(sizes) - sizes
    a, j = _spread(sizes[group])
    b = g0[group[a]] + j
    pair, kk = _spread(m[group[a]])
    pa, pb = ptr[a[pair]] + kk, ptr[b[pair]] + kk
    hit = (x0[pa] < x0[pb] + w[pb]) & (x0[pb] < x0[pa] + w[pa]) & \
          (y0[pa] < y0[pb] + h[pb]) & (y0[pb] < y0[pa] + h[pa])
    near = np.zeros(len(a), bool)
    np.logical_or.at(near, pair[hit], True)
    near &= a != b
    nptr = np.concatenate([[0], np.cumsum(np.bincount(a[near], minlength=n))])
    theta = np.zeros((n, NT))

    def logit(p):
        return np.log(p / (1 - p))

    theta[:, 0] = logit(np.where(star, 0.8, 0.2)) + rng.normal(0, 0.3, n)
    for i in (0, 1):
        theta[:, 1 + 2 * i] = logr + rng.normal(0, 0.15, n)
        theta[:, 2 + 2 * i] = math.log(0.02) + rng.normal(0, 0.3, n)
        theta[:, 5 + 4 * i:9 + 4 * i] = colors + rng.normal(0, 0.08, (n, 4))
        theta[:, 13 + 4 * i:17 + 4 * i] = math.log(0.01) + rng.normal(0, 0.3, (n, 4))
    theta[:, 21:23] = pos + rng.uniform(-0.3, 0.3, (n, 2))
    theta[:, 23] = angle + rng.normal(0, 0.1, n)
    theta[:, 24] = np.log(radius) + rng.normal(0, 0.1, n)
    theta[:, 25] = logit(np.clip(axis, 0.05, 0.95)) + rng.normal(0, 0.2, n)
    theta[:, 26] = logit(np.clip(prof, 0.05, 0.95)) + rng.normal(0, 0.2, n)
    npix = ih * iw
    i32 = lambda v: np.ascontiguousarray(v, dtype=np.int32)  # noqa: E731
    p = fields.Problem(
        model=model, pixels=None, sky=sky.astype(np.float32).ravel(), img_band=i32(band),
        img_h=i32(ih), img_w=i32(iw), img_stride=i32(iw),
        img_pix_off=(np.cumsum(npix) - npix).astype(np.int64),
        img_sky_off=np.arange(ni, dtype=np.int64) * (ky * kx), img_sky_ny=np.full(ni, ky, np.int32),
        img_sky_nx=np.full(ni, kx, np.int32), img_calib=200.0 * rng.uniform(0.9, 1.1, ni), img_A=A,
        img_t=t, img_psf=psf, theta=theta, patch_ptr=i32(ptr), patch_img=i32(pimg), patch_x0=i32(x0),
        patch_y0=i32(y0), patch_w=i32(w), patch_h=i32(h), nbr_ptr=i32(nptr), nbr_idx=i32(b[near]))
    return p, dict(flux=flux, cov=cov, pos=pos)


def _per_pixel(area, most=1 << 24):
    """Chunks (owner, index) of the pixels of patches with the given areas."""
    end = np.cumsum(area)
    lo = 0
    while lo < len(area):
        base = end[lo - 1] if lo else 0
        hi = max(lo + 1, int(np.searchsorted(end, base + most, side="right")))
        dev = _device()
        a = torch.as_tensor(area[lo:hi], device=dev)
        owner = torch.repeat_interleave(torch.arange(hi - lo, device=dev), a)
        yield slice(lo, hi), owner, torch.arange(len(owner), device=dev) - (torch.cumsum(a, 0) - a)[owner]
        lo = hi


def _device():
    return torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def _sky(p, i, y, x, dtype):
    """Sky at rows y and columns x of images i (tensors), between the knots."""
    dev = y.device
    ny, nx = int(p.img_sky_ny[0]), int(p.img_sky_nx[0])
    k = torch.as_tensor(p.sky, device=dev).to(dtype).view(-1, ny, nx)
    if ny == 1 and nx == 1:
        return k[i, 0, 0]
    hw = torch.as_tensor(np.stack([p.img_h, p.img_w]), device=dev)
    gy, gx = y.to(dtype) * (ny - 1) / (hw[0][i] - 1), x.to(dtype) * (nx - 1) / (hw[1][i] - 1)
    iy, ix = gy.floor().clamp(0, ny - 2).long(), gx.floor().clamp(0, nx - 2).long()
    fy, fx = gy - iy, gx - ix
    return (1 - fy) * ((1 - fx) * k[i, iy, ix] + fx * k[i, iy, ix + 1]) \
        + fy * ((1 - fx) * k[i, iy + 1, ix] + fx * k[i, iy + 1, ix + 1])


def _scene(case, seed):
    """A fields.Problem with photon counts: sky plus, for every source, one
    Gaussian per PSF component, with Poisson noise (rounded normal)."""
    p, truth = _geometry(case, seed)
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    ps = np.repeat(np.arange(p.n_sources), np.diff(p.patch_ptr))
    im = p.patch_img
    mu = np.einsum("pij,pj->pi", p.img_A[im], truth["pos"][ps]) + p.img_t[im]
    G = p.img_A[im] @ truth["cov"][ps] @ np.swapaxes(p.img_A[im], 1, 2)
    C = p.img_psf[im][:, :, 3:] + np.stack([G[:, 0, 0], G[:, 0, 1], G[:, 1, 1]], -1)[:, None]
    det = C[..., 0] * C[..., 2] - C[..., 1] ** 2
    amp = (truth["flux"][ps, p.img_band[im]] * p.img_calib[im])[:, None] \
        * p.img_psf[im][:, :, 0] / (2 * math.pi * np.sqrt(det))
    f32 = lambda v: torch.as_tensor(v, dtype=torch.float32, device=dev)  # noqa: E731
    q = f32(np.stack([amp, -0.5 * C[..., 2] / det, C[..., 1] / det, -0.5 * C[..., 0] / det], -1))
    off = f32(mu - np.stack([p.patch_x0, p.patch_y0], 1))
    start = torch.as_tensor(p.img_pix_off[im] + p.patch_y0.astype(np.int64) * p.img_stride[im]
                            + p.patch_x0, device=dev)
    width = torch.as_tensor(np.stack([p.patch_w, p.img_stride[im]]), device=dev).long()
    total = int((p.img_h.astype(np.int64) * p.img_stride).sum())
    lam = torch.zeros(total, dtype=torch.int64, device=dev)    # 2^-20 counts: sums in any order
    area = p.patch_w.astype(np.int64) * p.patch_h
    for sl, own, k in _per_pixel(area):
        ly, lx = k // width[0][sl][own], k % width[0][sl][own]
        dx, dy = lx - off[sl][own, 0], ly - off[sl][own, 1]
        v = torch.zeros_like(dx)
        for c in range(3):
            e = q[sl, c][own]
            v += e[:, 0] * torch.exp(e[:, 1] * dx * dx + e[:, 2] * dx * dy + e[:, 3] * dy * dy)
        lam.index_add_(0, start[sl][own] + ly * width[1][sl][own] + lx, (v * 2.0 ** 20).long())
    pixels = torch.empty(total, dtype=torch.float32, device=dev)
    for sl, own, k in _per_pixel(p.img_h.astype(np.int64) * p.img_w):
        w = torch.as_tensor(p.img_w, device=dev)[sl][own]
        lo = int(p.img_pix_off[sl.start])
        s = _sky(p, own + sl.start, k // w, k % w, torch.float32) \
            + lam[lo:lo + len(own)].float() * 2.0 ** -20
        z = torch.randn(len(own), generator=gen, device=dev)
        pixels[lo:lo + len(own)] = (s + s.sqrt() * z).round().clamp_min(0)
    p.pixels = pixels.cpu().numpy()
    return p


# ---------------------------------------------------------------------------
# states and passes
# ---------------------------------------------------------------------------

def _steps_inputs(case, seed):
    """Gradients, Hessians (mostly concave) and radii of quadratic models."""
    rng = np.random.default_rng([int(seed), 27])
    n = case["problems"]
    Q, _ = np.linalg.qr(rng.standard_normal((n, NT, NT)))
    lam = np.exp(rng.uniform(math.log(0.05), math.log(2e4), (n, NT)))
    lam *= np.where(rng.uniform(size=(n, NT)) < 0.02, -0.01, 1.0)
    H = -(Q * lam[:, None, :]) @ np.swapaxes(Q, 1, 2)
    g = np.exp(rng.uniform(math.log(0.1), math.log(300.0), (n, 1))) * rng.standard_normal((n, NT))
    d = np.exp(rng.uniform(math.log(0.02), math.log(8.0), n))
    return [torch.as_tensor(v, device=_device()) for v in (g, 0.5 * (H + np.swapaxes(H, 1, 2)), d)]


def _chain_thetas(case, p, seed):
    """The sampled sources (brightest first) and their chains' point values."""
    rng = np.random.default_rng([int(seed), 50])
    order = np.argsort(-p.theta[:, 1])[:case["sampled"]]
    th = np.repeat(p.theta[order], case["chains"], 0)
    th[:, 1:27] += rng.normal(0, 0.2, (len(th), 26)) * (np.arange(1, 27) != 23)
    kind = np.tile(np.arange(case["chains"]) * 2 // case["chains"], len(order))
    th[:, 0] = np.where(kind == 1, 40.0, -40.0)           # a point value of the type
    th[:, 2] = th[:, 4] = -40.0
    th[:, 13:21] = -40.0
    return [int(s) for s in order], th


def prepare(case, seed):
    call = case["call"]
    if call == "steps":
        g, H, d = _steps_inputs(case, seed)
        return dict(call=call, ctx=cel.Context(fields.make_model()), g=g, H=H, d=d)
    p = _scene(case, seed)
    if call == "loglik":
        sources, th = _chain_thetas(case, p, seed)
        return dict(call=call, ev=GpuLogLik(p, sources, case["chains"]), th=th)
    ctx = cel.Context(p.model)
    dp = cel.DeviceProblem(p, render_cache=bool(case.get("cache")))
    st = dict(call=call, ctx=ctx, dp=dp, theta0=dp.theta.clone())
    every = list(range(p.n_sources))
    # the tiles that autotune() picks for such scenes (pixels per item by patch area)
    tiles = (256, 256, 512, 0) if case["layout"] == "blends" and case.get("cache") else None
    if call == "newton":
        st["plans"] = [cel.Plan(ctx, dp, c, ppi_bucket=tiles) for c in cel.color_classes(p)]
        st["delta"], st["status"] = cel.newton_state(dp)
        if dp.cache is not None:
            for plan in st["plans"]:
                cel.render_cache(plan)
    elif call == "fit":
        st["fit"] = cel.Fit(ctx, dp, every)
    elif call == "field_elbo":
        st["field"] = cel.FieldElbo(ctx, dp)
    else:
        st["plan"] = cel.Plan(ctx, dp, every)
        if call == "gradient":
            st["objective"] = SourceObjective(st["plan"])
    return st


def run(state):
    call = state["call"]
    if call == "steps":
        return cel.tr_subproblem(state["ctx"], state["g"], state["H"], state["d"])
    if call == "loglik":
        return state["ev"](state["th"])
    dp = state["dp"]
    if call == "derivatives":
        return cel.elbo_grad_hess(state["plan"])
    if call == "newton":
        # a pass from the starting parameters (the cache's first half holds
        # their renders: a pass writes trial renders into the other)
        dp.theta.copy_(state["theta0"])
        state["delta"].fill_(1.0)
        state["status"].zero_()
        if dp.cache_half is not None:
            dp.cache_half.zero_()
        for plan in state["plans"]:
            cel.newton_step(plan, state["delta"], state["status"])
        return dp.theta, state["delta"], state["status"]
    if call == "gradient":
        theta = state["theta0"].detach().clone().requires_grad_(True)
        value = state["objective"](theta)
        value.sum().backward()
        return value.detach(), theta.grad
    if call == "render":
        return cel.render(state["plan"]) + cel.background(state["plan"])
    if call == "field_elbo":
        return state["field"]()
    dp.theta.copy_(state["theta0"])
    passes, gains = state["fit"].run()
    gains = np.array(gains + [0.0] * (5 - passes))         # 5: the most passes of a fit
    return (passes, gains, dp.theta) + state["fit"].results()


def work(case):
    """Bytes: each input and output once.  FLOPs: 4,200 a source-pixel visit
    with gradient and Hessian, 1,700 with the gradient, 400 for a value."""
    if case["call"] == "steps":
        n = case["problems"]
        return dict(bytes=8.0 * n * (NT * NT + 2 * NT + 2), flops=n * (NT ** 3 * 2.0))
    p, _ = _geometry(case, 0)
    area = p.patch_w.astype(np.int64) * p.patch_h
    visits, n = float(area.sum()), p.n_sources
    pixels = float((p.img_h.astype(np.int64) * p.img_w).sum())
    call = case["call"]
    if call == "derivatives":
        return dict(bytes=4 * min(pixels, visits) + 8.0 * n * (NT * NT + 2 * NT + 2), flops=4200 * visits)
    if call == "newton":
        return dict(bytes=4 * min(pixels, visits) + 16.0 * n * (NT + 1)
                    + (16 * visits if case.get("cache") else 0), flops=4600 * visits)
    if call == "gradient":
        return dict(bytes=4 * min(pixels, visits) + 8.0 * n * (2 * NT + 1), flops=2100 * visits)
    if call == "loglik":
        order = np.argsort(-p.theta[:, 1])[:case["sampled"]]
        per = sum(float(area[p.patch_ptr[s]:p.patch_ptr[s + 1]].sum()) for s in order)
        return dict(bytes=4 * per + 8.0 * case["sampled"] * case["chains"] * (NT + 1),
                    flops=400 * per * case["chains"])
    if call == "render":
        return dict(bytes=16 * visits + 8.0 * n * NT, flops=800 * visits)
    if call == "field_elbo":
        return dict(bytes=4 * pixels + 8.0 * n * NT, flops=400 * visits + 20 * pixels)
    # a fit: about 20 iterations a source in each of about 3 passes
    return dict(bytes=4 * pixels + 16.0 * n * NT, flops=60 * 4600 * visits)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

class _Exact:
    """The objective of a scene in float64 (plain torch)."""

    def __init__(self, p):
        self.p, self.dev = p, _device()
        d = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=self.dev)  # noqa: E731
        self.d = d
        self.theta = d(p.theta)
        self.A, self.t, self.psf = d(p.img_A), d(p.img_t), d(p.img_psf)
        self.calib, self.sel = d(p.img_calib), d(_SEL)[torch.as_tensor(p.img_band, device=self.dev).long()]
        self.img = torch.as_tensor(p.patch_img, device=self.dev).long()
        m = p.model
        self.tau = d(np.concatenate([m.tau_exp, m.tau_dev]))
        self.alpha, self.ne = d(np.concatenate([m.alpha_exp, m.alpha_dev])), len(m.tau_exp)
        self.rect = torch.as_tensor(np.stack([p.patch_x0, p.patch_y0, p.patch_w, p.patch_h]), device=self.dev).long()
        self.area = p.patch_w.astype(np.int64) * p.patch_h
        self.counts = torch.as_tensor(p.pixels, device=self.dev)

    def moments(self, th, patch, own, x, y):
        """E and V of E_q[l f] at pixels (x, y) of their patches' images:
        patch[k] with parameters th[k], pixel i belonging to row own[i]."""
        im = self.img[patch]
        A, psf, cal, sel = self.A[im], self.psf[im], self.calib[im], self.sel[im]
        mu = (A @ th[:, 21:23, None])[..., 0] + self.t[im]
        c, s = th[:, 23].cos(), th[:, 23].sin()
        r2 = (2 * th[:, 24]).exp()
        d2 = r2 * th[:, 25].sigmoid() ** 2
        S = torch.stack([c * c * r2 + s * s * d2, c * s * (d2 - r2), c * s * (d2 - r2),
                         s * s * r2 + c * c * d2], -1).view(-1, 2, 2)
        G = A @ S @ A.transpose(1, 2)
        Gv = torch.stack([G[:, 0, 0], G[:, 0, 1], G[:, 1, 1]], -1)
        rho = th[:, 26].sigmoid()
        pw = torch.cat([rho[:, None] * self.alpha[:self.ne], (1 - rho)[:, None] * self.alpha[self.ne:]], 1)

        def density(cov, wt, off):                         # [K, J, 3], [K, J], [K, J, 2]
            det = cov[..., 0] * cov[..., 2] - cov[..., 1] ** 2
            lw = torch.log(wt) - 0.5 * torch.log(det) - math.log(2 * math.pi)
            dx, dy = x[:, None] - (mu[:, None, 0] + off[..., 0])[own], y[:, None] - (mu[:, None, 1] + off[..., 1])[own]
            qx, qy, qz = (cov[..., 2] / det)[own], (cov[..., 1] / det)[own], (cov[..., 0] / det)[own]
            return torch.exp(lw[own] - 0.5 * (qx * dx * dx - 2 * qy * dx * dy + qz * dy * dy)).sum(1)

        J = len(self.tau)
        Fs = density(psf[:, :, 3:], psf[:, :, 0], psf[:, :, 1:3])
        cov = psf[:, :, None, 3:] + self.tau[None, None, :, None] * Gv[:, None, None]
        Fg = density(cov.reshape(-1, 3 * J, 3), (psf[:, :, 0, None] * pw[:, None]).reshape(-1, 3 * J),
                     psf[:, :, None, 1:3].expand(-1, -1, J, -1).reshape(-1, 3 * J, 2))
        q = torch.stack([(-th[:, 0]).sigmoid(), th[:, 0].sigmoid()], 1)
        m = torch.stack([th[:, 1 + 2 * i] + (sel * th[:, 5 + 4 * i:9 + 4 * i]).sum(1) for i in (0, 1)], 1)
        v = torch.stack([th[:, 2 + 2 * i].exp() + (sel * sel * th[:, 13 + 4 * i:17 + 4 * i].exp()).sum(1)
                         for i in (0, 1)], 1)
        e1 = cal[:, None] * (m + 0.5 * v).exp()
        F = torch.stack([Fg, Fs], 1)
        kF = e1[own] * F
        E = (q[own] * kF).sum(1)
        V = (q[own] * torch.expm1(v)[own] * kF ** 2).sum(1) + q[own, 0] * q[own, 1] * (kF[:, 0] - kF[:, 1]) ** 2
        return E, V

    def pixels(self, patches):
        """(row, x, y, count, sky) of the pixels of the listed patches."""
        area = self.area[patches]
        own = torch.repeat_interleave(torch.arange(len(patches), device=self.dev),
                                      torch.as_tensor(area, device=self.dev))
        first = torch.as_tensor(np.cumsum(area) - area, device=self.dev)
        k = torch.arange(len(own), device=self.dev) - first[own]
        pt = torch.as_tensor(patches, device=self.dev).long()
        x0, y0, w, _ = self.rect[:, pt]
        x, y = x0[own] + k % w[own], y0[own] + k // w[own]
        im = self.img[pt][own]
        p = self.p
        at = torch.as_tensor(p.img_pix_off, device=self.dev)[im] \
            + y * torch.as_tensor(p.img_stride, device=self.dev).long()[im] + x
        return own, x.double(), y.double(), self.counts[at].double(), _sky(p, im, y, x, torch.float64), first

    def background(self, sources, patches, sky, first, theta):
        """Sky and zero plus the neighbours' moments at those pixels."""
        p = self.p
        E, V = sky.clone(), torch.zeros_like(sky)
        nb = np.diff(p.nbr_ptr)[sources]
        a, k = _spread(nb)
        t = p.nbr_idx[p.nbr_ptr[np.asarray(sources)][a] + k]
        m = np.diff(p.patch_ptr)[sources]
        row0 = np.cumsum(m) - m
        pair, i = _spread(m[a])
        row, q = row0[a[pair]] + i, p.patch_ptr[t[pair]] + i
        P = np.asarray(patches)[row]
        x0, y0 = np.maximum(p.patch_x0[P], p.patch_x0[q]), np.maximum(p.patch_y0[P], p.patch_y0[q])
        x1 = np.minimum(p.patch_x0[P] + p.patch_w[P], p.patch_x0[q] + p.patch_w[q])
        y1 = np.minimum(p.patch_y0[P] + p.patch_h[P], p.patch_y0[q] + p.patch_h[q])
        keep = (x1 > x0) & (y1 > y0)
        row, q, P, t = row[keep], q[keep], P[keep], t[pair][keep]
        x0, y0, x1, y1 = x0[keep], y0[keep], x1[keep], y1[keep]
        T = lambda v: torch.as_tensor(np.asarray(v), device=self.dev).long()  # noqa: E731
        for sl, own, j in _per_pixel((x1 - x0).astype(np.int64) * (y1 - y0), 1 << 20):
            w = T(x1 - x0)[sl][own]
            x, y = T(x0)[sl][own] + j % w, T(y0)[sl][own] + j // w
            e, v = self.moments(theta[T(t[sl])], T(q[sl]), own, x.double(), y.double())
            at = first[T(row)[sl][own]] + (y - T(p.patch_y0[P])[sl][own]) * T(p.patch_w[P])[sl][own] \
                + x - T(p.patch_x0[P])[sl][own]
            E.index_add_(0, at, e)
            V.index_add_(0, at, v)
        return E, V

    def kl(self, th):
        m, d = self.p.model, self.d
        a = th[:, 0].sigmoid()
        la, lb = torch.nn.functional.logsigmoid(th[:, 0]), torch.nn.functional.logsigmoid(-th[:, 0])
        kl = a * (la - math.log(m.prior_a)) + (1 - a) * (lb - math.log1p(-m.prior_a))
        for i, q in ((0, 1 - a), (1, a)):
            R1, R2 = (float(v) for v in m.prior_r[i])
            lv = th[:, 2 + 2 * i]
            klr = 0.5 * (math.log(R2) - lv + (lv.exp() + (th[:, 1 + 2 * i] - R1) ** 2) / R2 - 1)
            cm, lc = th[:, 5 + 4 * i:9 + 4 * i], th[:, 13 + 4 * i:17 + 4 * i]
            P = torch.linalg.inv(d(m.color_cov[i]))
            dd = cm[:, None] - d(m.color_mean[i])
            K = 0.5 * ((torch.diagonal(P, dim1=1, dim2=2)[None] * lc.exp()[:, None]).sum(-1)
                       + torch.einsum("njk,jkl,njl->nj", dd, P, dd) - 4
                       + torch.logdet(d(m.color_cov[i]))[None] - lc.sum(1, keepdim=True))
            kl = kl + q * (klr - torch.logsumexp(d(np.log(m.color_w[i]))[None] - K, 1))
        e1, e2 = (float(v) for v in m.e_radius)
        kl = kl + th[:, 24] + 0.5 * math.log(2 * math.pi * e2) + (th[:, 24] - e1) ** 2 / (2 * e2)
        for k, (b1, b2) in ((25, m.e_axis), (26, m.e_profile)):
            ls = torch.nn.functional.logsigmoid
            kl = kl - (b1 - 1) * ls(th[:, k]) - (b2 - 1) * ls(-th[:, k]) \
                + math.lgamma(b1) + math.lgamma(b2) - math.lgamma(b1 + b2)
        return kl

    def objective(self, sources, theta=None, most=1 << 20):
        """Chunks (sources, function of their [k, 27] parameters giving the
        per-source pixel sums relative to absence, base sums)."""
        p = self.p
        theta = self.theta if theta is None else theta
        vis = np.array([self.area[p.patch_ptr[s]:p.patch_ptr[s + 1]].sum() for s in sources])
        chunk = np.cumsum(vis) // most
        for c in np.unique(chunk):
            some = np.asarray(sources)[chunk == c]
            patches = np.concatenate([np.arange(p.patch_ptr[s], p.patch_ptr[s + 1]) for s in some])
            rows = torch.as_tensor(np.repeat(np.arange(len(some)), np.diff(p.patch_ptr)[some]), device=self.dev)
            own, x, y, cnt, sky, first = self.pixels(patches)
            bE, bV = self.background(some, patches, sky, first, theta)
            base_px = -bE + cnt * (torch.log(bE) - bV / (2 * bE ** 2))
            src, pt = rows[own], torch.as_tensor(patches, device=self.dev).long()
            zero = torch.zeros(len(some), dtype=torch.float64, device=self.dev)

            def rel(th, rows=rows, pt=pt, own=own, x=x, y=y, cnt=cnt, bE=bE, bV=bV, src=src, zero=zero):
                e, v = self.moments(th[rows], pt, own, x, y)
                E, V = bE + e, bV + v
                term = -e + cnt * (torch.log1p(e / bE) - V / (2 * E ** 2) + bV / (2 * bE ** 2))
                return zero.index_add(0, src, term)

            yield some, rel, zero.index_add(0, src, base_px)

    def derivatives(self, sources, theta=None, hess=True, value_only=False):
        theta = self.theta if theta is None else theta
        out = []
        for some, rel, base in self.objective(sources, theta, 1 << (20 if hess else 21)):
            th = theta[torch.as_tensor(some, device=self.dev).long()].detach().requires_grad_(not value_only)
            r = rel(th) - self.kl(th)
            row = [(r + base).detach(), r.detach()]
            if not value_only:
                (g,) = torch.autograd.grad(r.sum(), th, create_graph=hess)
                row.append(g.detach())
                if hess:
                    row.append(torch.stack([torch.autograd.grad(g[:, k].sum(), th, retain_graph=True)[0]
                                            for k in range(NT)], 2).detach())
            out.append(row)
        return [torch.cat(v) for v in zip(*out)]


def _exact_steps(g, H, delta):
    """The trust-region steps by eigendecomposition and bisection, and the
    predicted gains."""
    lam, Q = torch.linalg.eigh(-0.5 * (H + H.transpose(1, 2)))
    gh = (Q.transpose(1, 2) @ g[..., None])[..., 0]
    lo = (-lam[:, 0]).clamp_min(0)
    hi = lo + g.norm(dim=1) / delta
    inside = (lam[:, 0] > 0) & ((gh / lam).norm(dim=1) <= delta)
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        big = (gh / (lam + mid[:, None])).norm(dim=1) > delta
        lo, hi = torch.where(big, mid, lo), torch.where(big, hi, mid)
    y = gh / (lam + torch.where(inside, torch.zeros_like(hi), hi)[:, None])
    return (Q @ y[..., None])[..., 0], (gh * y).sum(1) - 0.5 * (lam * y * y).sum(1)


def _exact_newton(case, p):
    ex = _Exact(p)
    theta, n = ex.theta.clone(), p.n_sources
    delta = torch.ones(n, dtype=torch.float64, device=ex.dev)
    status = torch.zeros(n, dtype=torch.int32, device=ex.dev)
    color = -np.ones(n, dtype=int)
    for s in range(n):                                     # greedy, ascending
        used = set(color[p.nbr_idx[p.nbr_ptr[s]:p.nbr_ptr[s + 1]]])
        color[s] = next(c for c in range(n + 1) if c not in used)
    for c in range(int(color.max()) + 1):
        cls = np.flatnonzero(color == c)
        i = torch.as_tensor(cls, device=ex.dev)
        _, rel, g, H = ex.derivatives(cls, theta)
        step, pred = _exact_steps(g, H, delta[i])
        stop = pred <= 1e-9 * (1 + rel.abs())
        trial = theta.clone()
        trial[i] += step
        got = torch.cat([f(trial[torch.as_tensor(some, device=ex.dev)])
                         - ex.kl(trial[torch.as_tensor(some, device=ex.dev)])
                         for some, f, _ in ex.objective(cls, theta, 1 << 21)])
        rho, size = (got - rel) / pred, step.norm(dim=1)
        acc = (rho > 0.1) & got.isfinite() & ~stop
        new = torch.where(~(rho >= 0.25), 0.25 * size,
                          torch.where((rho > 0.75) & (size >= 0.99 * delta[i]),
                                      (2 * delta[i]).clamp_max(100.0), delta[i]))
        delta[i] = torch.where(stop, delta[i], new)
        status[i] = torch.where(stop, cel.ST_CONVERGED,
                                torch.where(acc, cel.ST_ACCEPTED, cel.ST_REJECTED)).int()
        theta[i] = torch.where(acc[:, None], trial[i], theta[i])
    # radii follow from which steps were accepted: no 64-bit value of their own
    return theta, None, None


def exact(case, seed):
    call = case["call"]
    if call == "steps":
        return _exact_steps(*_steps_inputs(case, seed))
    if call == "fit" or case["sources"] > 1200 or (case["layout"] == "blends" and case["sources"] > 300
                                                   and call == "newton"):
        return None                                        # minutes in 64 bits
    p = _scene(case, seed)
    with torch.no_grad() if call in ("loglik", "render", "field_elbo") else torch.enable_grad():
        if call == "newton":
            return _exact_newton(case, p)
        ex = _Exact(p)
        every = np.arange(p.n_sources)
        if call == "derivatives":
            return tuple(ex.derivatives(every))
        if call == "gradient":
            e, _, g = ex.derivatives(every, hess=False)
            return e, g
        if call == "loglik":
            sources, th = _chain_thetas(case, p, seed)
            th = ex.d(th).view(len(sources), case["chains"], NT)
            out = torch.empty(len(sources), case["chains"], dtype=torch.float64, device=ex.dev)
            for k, s in enumerate(sources):
                for _, rel, _ in ex.objective([s]):
                    for c in range(case["chains"]):
                        out[k, c] = rel(th[k, c][None])[0]
            return out.reshape(-1).cpu().numpy()
        if call == "render":
            E, V, bE, bV = [], [], [], []
            for sl in np.array_split(every, max(1, len(every) // 16)):
                patches = np.arange(p.patch_ptr[sl[0]], p.patch_ptr[sl[-1] + 1])
                own, x, y, _, sky, first = ex.pixels(patches)
                src = torch.as_tensor(np.repeat(sl, np.diff(p.patch_ptr)[sl]), device=ex.dev)
                pt = torch.as_tensor(patches, device=ex.dev)
                for k in range(0, len(own), 1 << 20):      # rows of consecutive patches
                    o = own[k:k + (1 << 20)]
                    e, v = ex.moments(ex.theta[src], pt, o, x[k:k + (1 << 20)], y[k:k + (1 << 20)])
                    E.append(e)
                    V.append(v)
                be, bv = ex.background(sl, patches, sky, first, ex.theta)
                bE.append(be)
                bV.append(bv)
            return tuple(torch.cat(v) for v in (E, V, bE, bV))
        # field_elbo: every source's moments added into the images
        kl = ex.kl(ex.theta).sum()
        E = torch.zeros(len(p.pixels), dtype=torch.float64, device=ex.dev)
        V = torch.zeros_like(E)
        for sl, own, k in _per_pixel(p.img_h.astype(np.int64) * p.img_w):
            w = torch.as_tensor(p.img_w, device=ex.dev).long()[sl][own]
            lo = int(p.img_pix_off[sl.start])
            E[lo:lo + len(own)] = _sky(p, own + sl.start, k // w, k % w, torch.float64)
        ps = np.repeat(every, np.diff(p.patch_ptr))
        for sl, own, k in _per_pixel(ex.area, 1 << 20):
            pt = torch.arange(sl.start, sl.stop, device=ex.dev)
            x0, y0, w, _ = ex.rect[:, pt]
            x, y = x0[own] + k % w[own], y0[own] + k // w[own]
            e, v = ex.moments(ex.theta[torch.as_tensor(ps[sl], device=ex.dev)], pt, own, x.double(), y.double())
            im = ex.img[pt][own]
            at = torch.as_tensor(p.img_pix_off, device=ex.dev)[im] \
                + y * torch.as_tensor(p.img_stride, device=ex.dev).long()[im] + x
            E.index_add_(0, at, e)
            V.index_add_(0, at, v)
        px = (-E + ex.counts.double() * (torch.log(E) - V / (2 * E ** 2))).sum()
        return torch.stack([px - kl, px, kl])
