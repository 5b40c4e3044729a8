"""The pixel-integrated Sersic model of the fit (fse_opts.supersample = S:
the mean of S x S point samples per pixel) on the GPU against the FP64
oracle with the same S, needs a GB300.

Same parity gate as the pixel-centre model (centroid 1e-4 px, e 1e-5, r_e, n
and flux 1e-4 relative, chi^2 1e-5 relative).  The stamps include small,
cuspy galaxies rendered close to the pixel integral (8 x 8 samples), where
the pixel-centre model is biased and the pixel-integrated one is not.
"""
import math

import numpy as np
import pytest
import torch

import parity as PR
from paper_1203_0571_gb300 import binding as B
from paper_1203_0571_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return B.Context(0)


@pytest.fixture(scope="module")
def O(oracle):
    return oracle.get()


def small_galaxies(count, seed, side=32, noise=True):
    """Galaxies with r_e 0.6-1.6 px and n 1-6, rendered with 8 x 8 samples per
    pixel (near the pixel integral), noise sigma 1 (or none), SNR about 100.
    truth: n, r_e, I0, xc, yc, g1, g2 per stamp."""
    rng = np.random.default_rng(seed)
    stamps, truth = [], []
    for _ in range(count):
        n, re = rng.uniform(1.0, 6.0), rng.uniform(0.6, 1.6)
        gabs, phi = rng.uniform(0, 0.4), rng.uniform(0, math.pi)
        g1, g2 = gabs * math.cos(2 * phi), gabs * math.sin(2 * phi)
        xc, yc = (side - 1) / 2 + rng.uniform(-1, 1), (side - 1) / 2 + rng.uniform(-1, 1)
        prof = synth.single_stamp(side, side, n=n, re=re, g1=g1, g2=g2, xc=xc, yc=yc, I0=1.0, supersample=8)
        I0 = 100.0 / math.sqrt((prof ** 2).sum())
        stamps.append((I0 * prof + (rng.normal(0, 1, prof.shape) if noise else 0.0)).astype(np.float32).ravel())
        truth.append((n, re, I0, xc, yc, g1, g2))
    pix = torch.as_tensor(np.concatenate(stamps))
    off = torch.arange(count, dtype=torch.int64) * side * side
    hw = torch.full((count,), side, dtype=torch.int32)
    return synth.StampBatch(pix=pix, offset=off, h=hw, w=hw, truth={"t": np.array(truth)})


def run(ctx, O, batch, S, fn="fit_batch", ivar=None, **kw):
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    mp = int((batch.h.long() * batch.w.long()).max())
    iv = None if ivar is None else torch.as_tensor(ivar).cuda()
    out = getattr(ctx, fn)(b.pix, idx, scale=b.scale, inv_var=iv, opts=B.default_opts(max_pix=mp, supersample=S), **kw)
    torch.cuda.synchronize()
    g = B.results(out)
    ids = np.arange(batch.count)
    o = PR.oracle_results(O, batch, ids, ivar=ivar, opts=O.default_opts(supersample=S))
    rep = PR.compare(g, o, O=O, batch=batch, ids=ids, ivar=None if ivar is None else ivar, supersample=S,
                     orc_opts=O.default_opts(supersample=S))
    print(S, fn, PR.summary(rep))
    PR.dump(f"supersample_{S}_{fn}_{batch.count}", rep)
    return rep, g, o


def assert_gate(rep, max_gpu_short_frac=0.01):
    """The parity gate of tests/parity.py, with at most max_gpu_short_frac of the
    stamps (rounded up) converged by the oracle and not by the GPU."""
    PR.assert_gate(rep, max_gpu_short=int(np.ceil(max_gpu_short_frac * rep["n"])),
                   max_subpixel=int(np.ceil(0.01 * rep["n"])))


@pytest.mark.parametrize("S", [2, 3, 4])
def test_supersampled_chain_small_workload(ctx, O, S):
    rep, _, _ = run(ctx, O, synth.make_workload(0, count=128), S)
    assert_gate(rep)


def test_supersampled_small_cuspy_galaxies(ctx, O):
    """Where pixelation matters: both sides fit S = 4 through the whole chain
    and agree.  On the same galaxies without noise, fitted at their true
    centre and ellipticity (fse_sersic_fit), the model with the renderer's
    8 x 8 sub-grid recovers n and r_e to fp32 precision, while the
    pixel-centre model is off by tens of percent."""
    batch = small_galaxies(200, seed=3)
    rep, _, _ = run(ctx, O, batch, 4)
    assert_gate(rep)
    clean = small_galaxies(200, seed=3, noise=False).to("cuda")
    idx = B.make_index(clean.offset, clean.h, clean.w)
    t = clean.truth["t"]
    rec = np.zeros(clean.count, dtype=B.RESULT_DTYPE)
    rec["x0"], rec["y0"], rec["e1"], rec["e2"] = t[:, 3], t[:, 4], t[:, 5], t[:, 6]
    rec["sigma_w"] = 1.5
    rec["status"] = B.ST["MOM_CONVERGED"]
    err = {}
    for S in (1, 8):
        inout = torch.as_tensor(rec.view(np.uint8).reshape(-1, 64)).cuda()
        ctx.sersic_fit(clean.pix, idx, inout, opts=B.default_opts(max_pix=1024, supersample=S))
        f = B.results(inout)
        ok = (f["status"] & 2) == 2
        err[S] = (ok.mean(), np.median(np.abs(f["n"][ok] / t[ok, 0] - 1)), np.median(np.abs(f["re"][ok] / t[ok, 1] - 1)))
    print("converged, median |n/n_true - 1|, |r_e/r_e,true - 1|: pixel-centre", err[1], "8 x 8 sub-grid", err[8])
    assert err[8][0] > 0.95 and err[8][1] < 1e-3 and err[8][2] < 1e-3
    assert err[1][1] > 0.05


def test_supersampled_ivar_and_bf16(ctx, O):
    batch = synth.make_workload(0, count=96, first=100)
    iv = (0.5 + np.random.default_rng(2).random(batch.pix.numel())).astype(np.float32)
    rep, _, _ = run(ctx, O, batch, 3, ivar=iv)
    assert_gate(rep)
    b16 = synth.encode_bf16(synth.make_workload(0, count=96, first=200))
    rep, _, _ = run(ctx, O, b16, 3)
    assert_gate(rep)


def test_supersampled_fit_stage_and_ragged(ctx, O):
    """fse_sersic_fit from the moments of fse_ellipticity, and the ragged
    launch (one warp per stamp in every size class)."""
    batch = synth.make_workload(0, count=96, first=300)
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    opts = B.default_opts(max_pix=1024, supersample=3)
    mom = ctx.centroid(b.pix, idx, opts=opts)
    ctx.ellipticity(b.pix, idx, mom, opts=opts)
    ctx.sersic_fit(b.pix, idx, mom, opts=opts)
    full = ctx.fit_batch(b.pix, idx, opts=opts)
    torch.cuda.synchronize()
    st, fu = B.results(mom), B.results(full)
    ok = ((st["status"] & 3) == 3) & ((fu["status"] & 3) == 3) & ((fu["status"] & 128) == 0)
    assert ok.mean() > 0.8
    assert np.all(np.abs(st["re"][ok] / fu["re"][ok] - 1) <= 1e-4)
    assert np.all(np.abs(st["n"][ok] / fu["n"][ok] - 1) <= 1e-4)
    rag = synth.make_workload(2, count=200)
    rep, _, _ = run(ctx, O, rag, 2, fn="fit_batch_ragged")
    assert_gate(rep)


def test_supersample_options(ctx):
    batch = synth.make_workload(0, count=4).to("cuda")
    idx = B.make_index(batch.offset, batch.h, batch.w)
    for kw in (dict(supersample=9), dict(supersample=-1), dict(supersample=2, warps_per_stamp=2, warps_per_cta=2)):
        with pytest.raises(B.FseError):
            ctx.fit_batch(batch.pix, idx, opts=B.default_opts(max_pix=1024, **kw))
    # S = 0 and S = 1 are the pixel-centre model, bit for bit
    a = B.results(ctx.fit_batch(batch.pix, idx, opts=B.default_opts(max_pix=1024, supersample=0)))
    c = B.results(ctx.fit_batch(batch.pix, idx, opts=B.default_opts(max_pix=1024)))
    assert a.tobytes() == c.tobytes()


def test_shapes_that_do_not_fit_are_refused(ctx):
    """Launch shapes are accepted by the tile that the library states for them
    (two floats a pixel, three with weights), with the pixel-integrated model as
    without it: eight warps of 64x64 tiles do not fit an SM."""
    batch = synth.make_workload(0, count=8).to("cuda")
    idx = B.make_index(batch.offset, batch.h, batch.w)
    mom = ctx.centroid(batch.pix, idx, opts=B.default_opts(max_pix=1024))
    ctx.ellipticity(batch.pix, idx, mom, opts=B.default_opts(max_pix=1024))
    for ss in (1, 2):
        for warps, fits in ((4, True), (8, False)):
            opts = B.default_opts(max_pix=64 * 64, supersample=ss, warps_per_cta=warps)
            if fits:
                ctx.sersic_fit(batch.pix, idx, mom.clone(), opts=opts)
            else:
                with pytest.raises(B.FseError):
                    ctx.sersic_fit(batch.pix, idx, mom.clone(), opts=opts)
    ctx.sync_check()
