"""Performance cases of libfse: the calls a survey pipeline makes, at the sizes it makes them.

    listed()            the named cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs on the GPU (host memory for the host-buffer call), from the seed alone
    run(state)          one pass through the public entry points, and everything it computes
    work(case)          bytes and operations one pass cannot do without
    exact(case, seed)   the same results in 64 bits, in plain torch, where they have such a value

A case is a dict: "kind" names the call, the rest its sizes and options.

Inputs follow the recipes of the synthetic workloads: Sersic galaxies and stars
point-sampled on the pixel grid, noise N(0, 1) on zero sky.  The fits and the
moment stages end on iteration caps, bounds and failed steps for some noisy
stamps, whose records have no value apart from the iteration's own; those calls
therefore have no exact() value.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1203_0571_gb300 import autograd as A
from paper_1203_0571_gb300 import binding as B

K = math.sqrt(2.0 * math.log(2.0))          # half-light radius / sigma of a Gaussian
RECORD = (("x0", 0), ("y0", 1), ("e1", 2), ("e2", 3), ("I0", 4), ("re", 5), ("n", 6), ("flux", 7),
          ("sigma_w", 14), ("r50", 15))     # float words of the 64-byte result record
RECORD_INT = (("npix", 10), ("it_mom", 11), ("it_fit", 12), ("status", 13))
STAR = (("size", 0), ("beta", 1), ("I0", 2), ("flux", 3), ("r50", 4))
STAR_INT = (("iters", 5), ("status", 6))


def listed():
    return [
        # A user tries the library, or measures one small field: 256 stamps, the default options.
        dict(name="fit-256x32", kind="fit", count=256, h=32, w=32, dtype="f32", ivar=False, defaults=True,
             supersample=1),
        # The benchmark: a survey tile of 100,000 galaxies and stars, 48x48, resident in GPU memory.
        dict(name="fit-100k-48", kind="fit", count=100_000, h=48, w=48, dtype="f32", ivar=False, defaults=False,
             supersample=1),
        # A batch as an exposure yields it: stamps sized by their objects, 16 to 128 px, any order.
        dict(name="ragged-40k-16-128", kind="ragged", count=40_000, lo=16, hi=128, sides="object", dtype="f32",
             ivar=False),
        # An archive of compressed stamps: bf16 pixels with a scale per stamp, 32 to 64 px.
        dict(name="ragged-50k-bf16", kind="ragged", count=50_000, lo=32, hi=64, sides="square", dtype="bf16",
             ivar=False),
        # The service form: pinned host buffers in, records out, copies included.
        dict(name="host-40k-48", kind="host", count=40_000, h=48, w=48, dtype="f32", ivar=False),
        # The profile fit alone, with a weight map, at centres and ellipticities measured before; odd stamps.
        dict(name="sersic-8k-47x45-ivar", kind="sersic", count=8_000, h=47, w=45, dtype="f32", ivar=True,
             supersample=1),
        # A training step through the measured shapes: moments forward, pixel gradient backward.
        dict(name="shape-step-20k-48", kind="shape", count=20_000, h=48, w=48, ellip=True),
        # A training step through chi^2: 65,536 stamps of 64x64, gradients to parameters and pixels.
        dict(name="chi2-step-65k-64", kind="chi2", count=65_536, h=64, w=64, dtype="f32", ivar=False, dpix=True),
        # PSF measurement on the stars of a field: Gaussian profile, 32x32.
        dict(name="star-gauss-50k-32", kind="star", count=50_000, h=32, w=32, dtype="f32", profile="gauss"),
        # The same with the Moffat profile, 48x48.
        dict(name="star-moffat-20k-48", kind="star", count=20_000, h=48, w=48, dtype="f32", profile="moffat"),
        # The cut-out of each object from its 512x512 image, before anything is measured, into a buffer
        # the pipeline keeps (room for the largest square of every image).
        dict(name="cutout-500x512", kind="cutout", count=500, h=512, w=512, dtype="f32"),
        # Forward-mode propagation of a pixel perturbation (a calibration error) to the shapes.
        dict(name="jvp-50k-48", kind="jvp", count=50_000, h=48, w=48),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ranges: any size between, odd and non-square stamps among them."""
    kind = rng.choice(["fit", "fit", "ragged", "ragged", "host", "sersic", "shape", "chi2", "star", "star", "cutout",
                       "jvp"])
    h = rng.randint(24, 64)
    w = h if rng.random() < 0.5 else max(20, h + rng.randint(-7, 7))
    area = h * w
    dtype = "bf16" if rng.random() < 0.3 else "f32"
    ivar = rng.random() < 0.3
    if kind == "fit":
        defaults = rng.random() < 0.25
        ss = 2 if not defaults and rng.random() < 0.15 else 1
        top = 4_000 if defaults or ss > 1 else min(60_000, 120_000_000 // area)
        return dict(kind=kind, count=_logint(rng, 200, top), h=h, w=w, dtype=dtype, ivar=ivar, defaults=defaults,
                    supersample=ss)
    if kind == "ragged":
        lo, hi = rng.choice([(16, 128), (32, 64), (12, 40), (20, 90)])
        sides = rng.choice(["object", "square", "any"])
        return dict(kind=kind, count=_logint(rng, 500, min(50_000, 110_000_000 // (((lo + hi) // 2) ** 2))), lo=lo,
                    hi=hi, sides=sides, dtype=dtype, ivar=ivar)
    if kind == "host":
        return dict(kind=kind, count=_logint(rng, 500, min(40_000, 90_000_000 // area)), h=h, w=w, dtype=dtype,
                    ivar=ivar)
    if kind == "sersic":
        return dict(kind=kind, count=_logint(rng, 300, 8_000), h=h, w=w, dtype=dtype, ivar=ivar,
                    supersample=2 if rng.random() < 0.15 else 1)
    if kind == "shape":
        return dict(kind=kind, count=_logint(rng, 300, 20_000), h=h, w=w, ellip=rng.random() < 0.8)
    if kind == "chi2":
        return dict(kind=kind, count=_logint(rng, 1_000, 65_000), h=h, w=w, dtype=dtype, ivar=ivar,
                    dpix=dtype == "f32" and rng.random() < 0.7)
    if kind == "star":
        return dict(kind=kind, count=_logint(rng, 500, min(45_000, 45_000_000 // area)), h=h, w=w, dtype=dtype,
                    profile=rng.choice(["gauss", "moffat"]))
    if kind == "cutout":
        h = rng.randint(200, 600)
        w = h if rng.random() < 0.5 else rng.randint(200, 600)
        return dict(kind=kind, count=_logint(rng, 20, 130_000_000 // (h * w)), h=h, w=w, dtype=dtype)
    return dict(kind=kind, count=_logint(rng, 500, min(50_000, 115_000_000 // area)), h=h, w=w)


# ------------------------------------------------------------------ inputs
_ctx = None


def _context():
    """One context per process, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = B.Context(0)
    return _ctx


def _b_of_n(n):
    """b(n) of the Sersic profile by the expansion of Ciotti & Bertin (1999)."""
    return 2 * n - 1 / 3 + 4 / (405 * n) + 46 / (25515 * n * n)


def _sizes(case, r):
    n = case["count"]
    if "lo" not in case:
        return np.full(n, case["h"]), np.full(n, case["w"]), None
    lo, hi = case["lo"], case["hi"]
    if case["sides"] == "object":           # a stamp eight half-light radii wide, r_e spread in the logarithm
        re = np.exp(r.uniform(math.log(lo / 16), math.log(hi / 8), n))
        side = np.clip(np.rint(8 * re), lo, hi).astype(np.int64)
        return side, side, re
    h = r.integers(lo, hi + 1, n)
    return h, (h if case["sides"] == "square" else r.integers(lo, hi + 1, n)), None


def _objects(case, r):
    """Sizes and generating parameters of the objects (numpy, float64)."""
    n = case["count"]
    h, w, re = _sizes(case, r)
    kind = case["kind"]
    p = dict(n=r.uniform(0.5, 6.0 if kind == "chi2" else 4.0, n), re=r.uniform(1.5, 5.0, n) if re is None else re,
             beta=np.zeros(n))
    gabs, phi = r.uniform(0, 0.5, n), r.uniform(0, math.pi, n)
    snr = r.uniform(15, 200, n)
    off = 20.0 if kind == "cutout" else 1.0
    dx, dy = r.uniform(-off, off, n), r.uniform(-off, off, n)
    if kind == "star":
        r50, gabs, snr = r.uniform(1.5, 2.5, n), r.uniform(0, 0.25, n), np.full(n, 300.0)
        p["n"], p["re"] = np.full(n, 0.5), r50
        if case["profile"] == "moffat":     # re holds r_d
            p["beta"] = r.uniform(3, 5, n)
            p["re"] = r50 / np.sqrt(2 ** (1 / (p["beta"] - 1)) - 1)
    elif re is None and kind != "cutout":   # a fifth of a tile's objects are stars
        star = r.random(n) < 0.2
        p["n"] = np.where(star, 0.5, p["n"])
        p["re"] = np.where(star, r.uniform(1, 2, n), p["re"])
        gabs = np.where(star, r.uniform(0, 0.05, n), gabs)
    q = (1 - gabs) / (1 + gabs)
    b = _b_of_n(p["n"])
    # amplitude from the matched-filter signal-to-noise ratio: sum m^2 = SNR^2
    s2 = np.where(p["beta"] > 0, math.pi * q * p["re"] ** 2 / np.maximum(2 * p["beta"] - 1, 1),
                  2 * math.pi * p["n"] * q * p["re"] ** 2 *
                  np.exp(np.vectorize(math.lgamma)(2 * p["n"]) - 2 * p["n"] * np.log(2 * b)))
    p.update(b=b, gabs=gabs, g1=gabs * np.cos(2 * phi), g2=gabs * np.sin(2 * phi), xc=(w - 1) / 2 + dx,
             yc=(h - 1) / 2 + dy, I0=snr / np.sqrt(s2))
    return h, w, p


def _pixels(h, w, p, gen, dtype):
    """Flat pixel buffer (stamps back to back), offsets and, for bf16, the per-stamp scale."""
    area = h * w
    offset = np.concatenate([[0], np.cumsum(area)[:-1]]).astype(np.int64)
    total = int(area.sum())
    pix = torch.empty(total, dtype=torch.float32, device="cuda")
    scale = torch.empty(len(h), dtype=torch.float32, device="cuda")
    cols = torch.as_tensor(np.stack([p["xc"], p["yc"], p["g1"], p["g2"], (1 - p["gabs"]) * p["re"], 1 / p["n"], p["b"],
                                     p["I0"], p["beta"], w], axis=1).astype(np.float32)).cuda()
    areas = torch.as_tensor(area).cuda()
    i0 = 0
    while i0 < len(h):
        i1 = max(i0 + 1, int(np.searchsorted(offset, offset[i0] + (1 << 24))))
        m = int(area[i0:i1].sum())
        o0 = int(offset[i0])
        sid = torch.repeat_interleave(torch.arange(i1 - i0, device="cuda"), areas[i0:i1], output_size=m)
        start = torch.as_tensor(offset[i0:i1] - o0).cuda()
        local = (torch.arange(m, device="cuda") - start[sid]).to(torch.int32)
        xc, yc, g1, g2, rq, inv_n, b, I0, beta, wf = cols[i0:i1][sid].unbind(1)
        row = torch.div(local, wf.to(torch.int32), rounding_mode="floor")
        d1, d2 = (local - row * wf.to(torch.int32)) - xc, row - yc
        R2 = ((1 - g1) ** 2 + g2 ** 2) * d1 * d1 + ((1 + g1) ** 2 + g2 ** 2) * d2 * d2 - 4 * g2 * d1 * d2
        x = R2.clamp_(min=1e-12).sqrt_() / rq
        img = I0 * torch.exp(-b * x ** inv_n)
        if bool((p["beta"][i0:i1] > 0).any()):
            img = torch.where(beta > 0, I0 * (1 + x * x) ** (-beta), img)
        img += torch.randn(m, generator=gen, device="cuda")
        if dtype == "bf16":
            mx = torch.zeros(i1 - i0, device="cuda").scatter_reduce(0, sid, img.abs(), reduce="amax")
            scale[i0:i1] = mx
            img = img / mx[sid]
        pix[o0:o0 + m] = img
        i0 = i1
    return (pix.to(torch.bfloat16), offset, scale) if dtype == "bf16" else (pix, offset, None)


def _record(**cols):
    """Result records a previous call left: the given float columns, moments converged."""
    n = len(next(iter(cols.values())))
    f = torch.zeros((n, 16), dtype=torch.float32)
    at = dict(RECORD)
    for k, v in cols.items():
        f[:, at[k]] = torch.as_tensor(np.asarray(v, dtype=np.float32))
    f.view(torch.int32)[:, 13] = B.ST["MOM_CONVERGED"]
    return f.cuda().view(torch.uint8)


def prepare(case, seed):
    r = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, n = case["kind"], case["count"]
    ctx = _context()
    h, w, p = _objects(case, r)
    pix, offset, scale = _pixels(h, w, p, gen, case.get("dtype", "f32"))
    idx = B.make_index(offset, h, w)
    s = dict(kind=kind, ctx=ctx, pix=pix, idx=idx, scale=scale, ivar=None, h=int(h[0]), w=int(w[0]))
    if case.get("ivar"):                    # a weight map: the sky's variance varies across the field
        s["ivar"] = torch.rand(pix.numel(), generator=gen, device="cuda") * 0.6 + 0.7
    max_pix = int((h * w).max())
    if kind == "fit":
        s["opts"] = None if case["defaults"] else B.default_opts(max_pix=max_pix, supersample=case["supersample"])
        s["out"] = torch.zeros((n, 64), dtype=torch.uint8, device="cuda")
    elif kind == "ragged":
        s["out"] = torch.zeros((n, 64), dtype=torch.uint8, device="cuda")
    elif kind == "host":
        s["pix"], s["idx"] = pix.cpu().pin_memory(), idx.cpu().pin_memory()
        s["scale"] = None if scale is None else scale.cpu().pin_memory()
        s["ivar"] = None if s["ivar"] is None else s["ivar"].cpu().pin_memory()
        s["out"] = torch.zeros((n, 64), dtype=torch.uint8).pin_memory()
    elif kind == "sersic":
        # centres and ellipticities as a moment stage measures them, sigma_w from the growth curve
        s["opts"] = B.default_opts(max_pix=max_pix, supersample=case["supersample"])
        e = r.normal(0, 0.004, (2, n))
        s["start"] = _record(x0=p["xc"] + r.normal(0, 0.02, n), y0=p["yc"] + r.normal(0, 0.02, n), e1=p["g1"] + e[0],
                             e2=p["g2"] + e[1], sigma_w=np.clip(p["re"] / K * r.uniform(0.85, 1.05, n), 0.5, 12),
                             r50=p["re"])
        s["out"] = torch.empty_like(s["start"])
    elif kind == "star":
        s["opts"] = B.default_opts(max_pix=max_pix)
        r50 = p["re"] * np.sqrt(np.where(p["beta"] > 0, 2 ** (1 / np.maximum(p["beta"] - 1, 0.1)) - 1, 1.0))
        s["moments"] = _record(x0=p["xc"] + r.normal(0, 0.005, n), y0=p["yc"] + r.normal(0, 0.005, n),
                               e1=p["g1"] + r.normal(0, 0.002, n), e2=p["g2"] + r.normal(0, 0.002, n),
                               sigma_w=r50 / K * r.uniform(0.95, 1.05, n), r50=r50)
        s["profile"] = case["profile"]
        s["out"] = torch.zeros((n, 32), dtype=torch.uint8, device="cuda")
    elif kind == "shape":
        s["opts"], s["ellip"] = B.default_opts(max_pix=max_pix), case["ellip"]
        s["pix"].requires_grad_(True)
        s["gout"] = torch.randn((n, 5), generator=gen, device="cuda")
    elif kind == "chi2":
        # parameters near the optimum, as during training
        q = np.stack([p["xc"] + r.normal(0, 0.05, n), p["yc"] + r.normal(0, 0.05, n), 0.95 * p["g1"], 0.95 * p["g2"],
                      p["I0"] * r.uniform(0.9, 1.1, n), p["re"] * r.uniform(0.9, 1.1, n),
                      p["n"] * r.uniform(0.95, 1.05, n)], axis=1)
        s["params"] = torch.as_tensor(q.astype(np.float32)).cuda().requires_grad_(True)
        s["pix"].requires_grad_(case["dpix"])
        s["gout"] = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) + 0.5
    elif kind == "cutout":
        s["out"] = torch.zeros(n * 128 * 128, dtype=pix.dtype, device="cuda")
    elif kind == "jvp":
        opts = B.default_opts(max_pix=max_pix)
        s["moments"] = ctx.centroid(pix, idx, opts=opts)
        ctx.ellipticity(pix, idx, s["moments"], opts=opts)
        s["tangent"] = torch.randn(pix.numel(), generator=gen, device="cuda")
        s["status"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    return s


# ------------------------------------------------------------------ one pass
def _fields(out, names, ints, chi2=False):
    """The columns of a record tensor, each in its own type (views)."""
    f, i = out.view(torch.float32).unbind(1), out.view(torch.int32).unbind(1)
    d = {k: f[c] for k, c in names}
    d.update((k, i[c]) for k, c in ints)
    if chi2:
        d["chi2"] = out.view(torch.float64).select(1, 4)
    return d


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "fit":
        out = ctx.fit_batch(s["pix"], s["idx"], scale=s["scale"], inv_var=s["ivar"], opts=s["opts"], out=s["out"])
        return _fields(out, RECORD, RECORD_INT, chi2=True)
    if kind == "ragged":
        out = ctx.fit_batch_ragged(s["pix"], s["idx"], scale=s["scale"], inv_var=s["ivar"], out=s["out"])
        return _fields(out, RECORD, RECORD_INT, chi2=True)
    if kind == "host":
        out = ctx.fit_batch_host(s["pix"], s["idx"], scale=s["scale"], inv_var=s["ivar"], out=s["out"])
        return _fields(out, RECORD, RECORD_INT, chi2=True)
    if kind == "sersic":
        out = s["out"].copy_(s["start"])
        ctx.sersic_fit(s["pix"], s["idx"], out, scale=s["scale"], inv_var=s["ivar"], opts=s["opts"])
        return _fields(out, RECORD, RECORD_INT, chi2=True)
    if kind == "star":
        out = ctx.star_fit(s["pix"], s["idx"], s["moments"], profile=s["profile"], scale=s["scale"], opts=s["opts"],
                           out=s["out"])
        return _fields(out, STAR, STAR_INT)
    if kind == "shape":
        s["pix"].grad = None
        theta = A.moment_shape(s["pix"], s["idx"], ctx, opts=s["opts"], ellip=s["ellip"])
        theta.backward(s["gout"])
        return {"theta": theta.detach(), "dpix": s["pix"].grad}
    if kind == "chi2":
        s["params"].grad = s["pix"].grad = None
        chi2 = A.sersic_chi2(s["params"], s["pix"], s["idx"], ctx, scale=s["scale"], inv_var=s["ivar"])
        chi2.backward(s["gout"])
        d = {"chi2": chi2.detach(), "dparams": s["params"].grad}
        if s["pix"].grad is not None:
            d["dpix"] = s["pix"].grad
        return d
    if kind == "cutout":
        pix, idx, info = ctx.cutout(s["pix"], s["idx"], scale=s["scale"], out=s["out"])
        i = info.view(torch.int32)
        return {"pix": pix, "index": idx, "square": i[:, :4], "r50": info.view(torch.float32)[:, 4],
                "status": i[:, 5]}
    out = ctx.moment_jvp(s["pix"], s["idx"], s["moments"], s["tangent"], status=s["status"])
    return {"dtheta": out, "status": s["status"]}


def work(case):
    """Every pixel read once (and its gradient written once), the records written once; operations
    per pixel of the method: 31 per moment-kind pass and 33 per fit-kind pass over a typical
    object's passes, 40 per pixel for chi^2 and its gradient, 20 for the gradients of the moments."""
    n = case["count"]
    if "lo" in case:
        lo, hi = case["lo"], case["hi"]
        if case["sides"] == "object":
            u = np.clip(8 * np.exp(np.linspace(math.log(lo / 16), math.log(hi / 8), 2001)), lo, hi)
            area = float((u * u).mean())
        else:
            m = (lo + hi) / 2
            area = m * m + ((hi - lo) ** 2 / 12 if case["sides"] == "square" else 0)
    else:
        area = case["h"] * case["w"]
    px = n * area
    e = 2 if case.get("dtype") == "bf16" else 4
    read = px * (e + (4 if case.get("ivar") else 0)) + 16 * n
    kind, ss = case["kind"], case.get("supersample", 1) ** 2
    if kind in ("fit", "ragged", "host"):
        return {"bytes": read + 64 * n, "flops": px * (12 + 9 * 31 + 8.5 * 33 * ss)}
    if kind == "sersic":
        return {"bytes": read + 128 * n, "flops": px * 8.5 * 33 * ss}
    if kind == "star":
        return {"bytes": read + 96 * n, "flops": px * 15 * (6 if case["profile"] == "gauss" else 9)}
    if kind == "shape":
        return {"bytes": 2 * read, "flops": px * (12 + 9 * 31 + 20 + 15)}
    if kind == "chi2":
        return {"bytes": 2 * read + (4 * px if case["dpix"] else 0) + 80 * n, "flops": px * 60}
    if kind == "cutout":
        return {"bytes": read + 40 * n, "flops": px * 8}
    return {"bytes": read + 4 * px + 84 * n, "flops": px * 40}


# ------------------------------------------------------------------ the same results in 64 bits
def _chunks(n, area):
    step = max(1, (1 << 24) // area)
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _grid(s):
    """Pixel coordinates (x, y) of a stamp, float64 [1, h w]."""
    p = torch.arange(s["h"] * s["w"], device="cuda")
    return (p % s["w"]).double().view(1, -1), torch.div(p, s["w"], rounding_mode="floor").double().view(1, -1)


def _decoded(s, i, j):
    a = s["h"] * s["w"]
    v = s["pix"].detach()[i * a:j * a].view(j - i, a).double()
    return v if s["scale"] is None else v * s["scale"][i:j, None].double()


def _ellipse_r2(x, y, g1, g2):
    return ((1 - g1) ** 2 + g2 ** 2) * x * x + ((1 + g1) ** 2 + g2 ** 2) * y * y - 4 * g2 * x * y


def _exact_b(n):
    """b(n) with P(2n, b) = 1/2, by bisection on the regularised incomplete gamma function."""
    lo, hi = torch.zeros_like(n), 2 * n
    for _ in range(70):
        mid = (lo + hi) / 2
        over = torch.special.gammainc(2 * n, mid) > 0.5
        lo, hi = torch.where(over, lo, mid), torch.where(over, mid, hi)
    return (lo + hi) / 2


def _exact_chi2(case, s):
    n = case["count"]
    P = s["params"].detach().double()
    out = [[], [], []]
    d = 1e-3
    nn = P[:, 6]
    b = _exact_b(nn)
    db = (8 * (_exact_b(nn + d) - _exact_b(nn - d)) - (_exact_b(nn + 2 * d) - _exact_b(nn - 2 * d))) / (12 * d)
    x, y = _grid(s)
    for i, j in _chunks(n, s["h"] * s["w"]):
        I = _decoded(s, i, j)
        wt = 1.0 if s["ivar"] is None else s["ivar"][i * I.shape[1]:j * I.shape[1]].view_as(I).double()
        q = torch.cat([P[i:j], b[i:j, None]], 1).requires_grad_(True)
        x0, y0, g1, g2, I0, re, ns, bs = (q[:, k:k + 1] for k in range(8))
        rs = torch.sqrt(_ellipse_r2(x - x0, y - y0, g1, g2)) / (1 - torch.sqrt(g1 * g1 + g2 * g2))
        m = I0 * torch.exp(-bs * (rs / re) ** (1 / ns))
        r = m - I
        c = (wt * r * r).sum(1)
        (g,) = torch.autograd.grad((c * s["gout"][i:j]).sum(), q)
        out[0].append(c.detach())
        out[1].append(torch.cat([g[:, :6], (g[:, 6] + g[:, 7] * db[i:j])[:, None]], 1))
        if case["dpix"]:
            out[2].append((-2 * wt * r.detach() * s["gout"][i:j, None]).reshape(-1))
    d = {"chi2": torch.cat(out[0]), "dparams": torch.cat(out[1])}
    if case["dpix"]:
        d["dpix"] = torch.cat(out[2])
    return d


def _exact_star(case, s):
    n = case["count"]
    f = s["moments"].view(torch.float32).double()
    moffat = case["profile"] == "moffat"
    gx, gy = _grid(s)
    res = []
    for i, j in _chunks(n, s["h"] * s["w"]):
        I = _decoded(s, i, j)
        x0, y0, g1, g2, sig = (f[i:j, k:k + 1] for k in (0, 1, 2, 3, 14))
        gabs = torch.sqrt(g1 * g1 + g2 * g2)
        r2 = _ellipse_r2(gx - x0, gy - y0, g1, g2) / (1 - gabs) ** 2
        gabs, sig = gabs[:, 0], sig[:, 0]
        q = (1 - gabs) / (1 + gabs)
        sw = (2.35 if moffat else 1.0) * sig / (1 - gabs)
        size, beta, S0 = sw.clone(), torch.zeros_like(sw), torch.zeros_like(sw)
        live, done = torch.ones_like(sw, dtype=torch.bool), torch.zeros_like(sw, dtype=torch.bool)
        for _ in range(60):
            c = 1 / (sw * sw)[:, None]
            W = (1 + r2 * c) ** -3 if moffat else torch.exp(-0.5 * r2 * c)
            fw = I * W
            a0, a2, a4 = fw.sum(1), (fw * r2).sum(1), (fw * r2 * r2).sum(1)
            S0 = torch.where(live, a0, S0)
            live = live & (a0 > 0) & (a2 > 0)
            if moffat:
                ratio = a4 * a0 / (2 * a2 * a2)
                live = live & (ratio > 1)
                beta = torch.where(live, 1 / (ratio - 1), beta)
                new = torch.sqrt(a2 / a0 * (beta + 1))
            else:
                new = torch.sqrt(a2 / a0)
            size = torch.where(live, new, size)
            stop = live & ((size / sw - 1).abs() <= 1e-6)
            sw = torch.where(live, size, sw)
            done |= stop
            live = live & ~stop
            if not bool(live.any()):
                break
        if moffat:
            I0 = S0 * (beta + 2) / (math.pi * size ** 2 * q)
            flux = math.pi * size ** 2 * I0 * q / (beta - 1)
            r50 = size * torch.sqrt(torch.expm1(math.log(2) / (beta - 1)))
        else:
            I0 = S0 / (math.pi * size ** 2 * q)
            flux, r50 = 2 * math.pi * size ** 2 * I0 * q, size * K
        zero = torch.zeros_like(size)
        res.append([size, beta] + [torch.where(done, v, zero) for v in (I0, flux, r50)])
    d = {k: torch.cat([v[c] for v in res]) for k, c in STAR}
    # small Moffat stars run away to an infinite index (a ratio r4 r0 / 2 r2^2 of one): whether and
    # where their iteration fails is decided by rounding, and the column has no exact value
    if moffat and not (float(d["beta"].max()) < 1e3):
        return None
    d.update(iters=None, status=None)
    return d


def _rings(gx, gy, peak, w):
    """Ring index ceil(distance) of every pixel about the brightest one (exact integers)."""
    dx, dy = gx - (peak % w).double()[:, None], gy - torch.div(peak, w, rounding_mode="floor").double()[:, None]
    return torch.ceil(torch.sqrt(dx * dx + dy * dy)).long()


def _growth(I, ring):
    """Crossing ring k of the growth curve, the enclosed sums before and after it, the total."""
    rings = int(ring.max()) + 1
    cum = torch.zeros(I.shape[0], rings, dtype=torch.float64, device="cuda").scatter_add_(1, ring, I).cumsum(1)
    tot = I.sum(1)
    hit = 2 * cum >= tot[:, None]
    k = torch.where(hit.any(1), hit.int().argmax(1), torch.full_like(tot, rings - 1, dtype=torch.long))
    cur = cum.gather(1, k[:, None])[:, 0]
    prev = torch.where(k > 0, cum.gather(1, (k - 1).clamp(min=0)[:, None])[:, 0], torch.zeros_like(cur))
    return k, prev, cur, tot


def _exact_cutout(case, s):
    gx, gy = _grid(s)
    r50 = []
    for i, j in _chunks(case["count"], s["h"] * s["w"]):
        I = _decoded(s, i, j)
        k, prev, cur, tot = _growth(I, _rings(gx, gy, I.argmax(1), s["w"]))
        r = torch.where(k == 0, 0.25 * tot / cur, k - 1 + (tot / 2 - prev) / (cur - prev))
        r50.append(torch.where(tot > 0, r, torch.full_like(r, K)))
    return {"pix": None, "index": None, "square": None, "r50": torch.cat(r50), "status": None}


def _exact_jvp(case, s):
    gx, gy = _grid(s)
    f = s["moments"].view(torch.float32).double()
    status = s["moments"].view(torch.int32)[:, 13]
    res = []
    area = s["h"] * s["w"]
    for i, j in _chunks(case["count"], 4 * area):
        I, U = _decoded(s, i, j), s["tangent"][i * area:j * area].view(j - i, area).double()
        q = f[i:j][:, [0, 1, 2, 3, 14]].clone().requires_grad_(True)
        x0, y0, g1, g2, sw = (q[:, k:k + 1] for k in range(5))
        t1, t2 = gx - x0, gy - y0
        R2 = _ellipse_r2(t1, t2, g1, g2)
        W = torch.exp(-R2 / (2 * sw * sw))
        e = 2 / (1 + g1 * g1 + g2 * g2)
        T = t1 * t1 + t2 * t2
        m = [t1, t2, t1 * t1 - t2 * t2 - e * g1 * T, 2 * t1 * t2 - e * g2 * T]
        J = torch.stack([torch.autograd.grad((I * W * mk).sum(), q, retain_graph=True)[0] for mk in m], 1)
        with torch.no_grad():
            k, prev, cur, tot = _growth(I, ring := _rings(gx, gy, I.argmax(1), s["w"]))
            kk = k[:, None]
            up, ud, ut = (U * (ring <= kk - 1)).sum(1), (U * (ring <= kk)).sum(1), U.sum(1)
            D, H = cur - prev, tot / 2 - prev
            # r50 = (k-1) + H/D, or tot/(4 cur) where the brightest pixel holds half the light
            dr = torch.where(k == 0, (ut / 4 - ud * tot / (4 * cur)) / cur, (ut / 2 - up) / D - H * (ud - up) / (D * D))
            held = ((status[i:j] & B.ST["SIGW_CLAMPED"]) != 0) | (tot <= 0)
            ds = torch.where(held, torch.zeros_like(dr), dr / K)
            rhs = torch.stack([(U * W * mk).sum(1) for mk in m], 1) + J[:, :, 4] * ds[:, None]
            ok = (status[i:j] & B.ST["MOM_CONVERGED"]) != 0
            eye = torch.eye(4, dtype=torch.float64, device="cuda")
            x = torch.linalg.solve(torch.where(ok[:, None, None], J[:, :, :4], eye), -rhs)
            res.append(torch.where(ok[:, None], torch.cat([x, ds[:, None]], 1), torch.zeros(5, device="cuda",
                                                                                            dtype=torch.float64)))
    return {"dtheta": torch.cat(res), "status": None}


def exact(case, seed):
    f = {"chi2": _exact_chi2, "star": _exact_star, "cutout": _exact_cutout, "jvp": _exact_jvp}.get(case["kind"])
    return None if f is None else f(case, prepare(case, seed))
