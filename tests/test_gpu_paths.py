"""The kernels' size- and alignment-dependent paths at the sizes where they
change over (needs a GB300): tensor-memory columns of the fit, the halves of a
large batch, vector and scalar loads of the adjoint and moment gradients, the
near square and whole-image passes of the cut-out."""
import numpy as np
import pytest
import torch

import parity as PR
from paper_1203_0571_gb300 import binding as B
from paper_1203_0571_gb300 import synth
from test_gpu_adjoint import check_against_oracle as check_adjoint
from test_gpu_cutout import check_against_oracle as check_cutout
from test_gpu_star import compare as compare_stars, gpu_stars, oracle_moments, oracle_stars

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return B.Context(0)


@pytest.fixture(scope="module")
def O(oracle):
    return oracle.get()


def galaxies(shapes, seed, I0=400.0, lead=0):
    """One galaxy per (h, w), back to back from element `lead` on."""
    rng = np.random.default_rng(seed)
    pix, offs, pos = [np.zeros(lead, np.float32)], [], lead
    for h, w in shapes:
        img = synth.single_stamp(h, w, n=float(rng.uniform(0.8, 3.0)), re=0.11 * min(h, w) + 0.8,
                                 g1=float(rng.uniform(-0.2, 0.2)), g2=float(rng.uniform(-0.2, 0.2)),
                                 xc=w / 2 - 0.5 + float(rng.uniform(-0.4, 0.4)),
                                 yc=h / 2 - 0.5 + float(rng.uniform(-0.4, 0.4)), I0=I0, noise_sigma=1.0,
                                 seed=int(rng.integers(1 << 30)))
        pix.append(img.astype(np.float32).ravel())
        offs.append(pos)
        pos += h * w
    return synth.StampBatch(pix=torch.as_tensor(np.concatenate(pix)), offset=torch.as_tensor(offs),
                            h=torch.as_tensor([s[0] for s in shapes], dtype=torch.int32),
                            w=torch.as_tensor([s[1] for s in shapes], dtype=torch.int32), truth={})


# pixel counts around the multiples of 32 nw x 8 (tensor-memory loads of eight
# columns) and 32 nw (a column), and stamps of fewer pixels than threads
EDGES = {1: [(15, 17), (16, 16), (16, 17), (16, 18), (31, 33), (32, 32), (25, 41), (128, 128)],
         2: [(16, 31), (16, 32), (19, 27), (31, 33), (32, 33), (127, 128)],
         4: [(31, 33), (32, 32), (25, 41), (33, 31), (47, 49), (127, 127)],
         8: [(14, 16), (45, 45), (32, 64), (43, 48), (63, 65), (128, 127)]}


@pytest.mark.parametrize("ivar", [False, True])
@pytest.mark.parametrize("nw", [1, 2, 4, 8])
def test_fit_at_column_edges(ctx, O, nw, ivar):
    """The parity gate; with inverse variances the galaxies are bright enough
    for pixels whose model is formed in fp64."""
    batch = galaxies(EDGES[nw], 17 + nw, I0=3.0e4 if ivar else 400.0)
    iv = (0.5 + np.random.default_rng(nw).random(batch.pix.numel())).astype(np.float32) if ivar else None
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    kw = {} if iv is None else dict(inv_var=torch.as_tensor(iv).cuda())
    g = B.results(ctx.fit_batch(b.pix, idx, opts=B.default_opts(max_pix=128 * 128, warps_per_stamp=nw,
                                                                 warps_per_cta=nw), **kw))
    ids = np.arange(batch.count)
    o = PR.oracle_results(O, batch, ids, ivar=iv)
    PR.assert_gate(PR.compare(g, o, O=O, batch=batch, ids=ids, ivar=iv), max_gpu_short=1, max_subpixel=0)


@pytest.mark.parametrize("nw,count", [(1, 2047), (1, 2049), (2, 1025)])
def test_halves_equal_small_parts(ctx, nw, count):
    """A batch of count x warps >= 2048 runs as two halves on two streams, and
    as one chain under capture; calls of 500 stamps run whole.  Same bytes."""
    batch = synth.make_workload(0, count=count)
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    opts = B.default_opts(max_pix=32 * 32, warps_per_stamp=nw, warps_per_cta=nw)
    out = ctx.fit_batch(b.pix, idx, opts=opts)
    parts = torch.cat([ctx.fit_batch(b.pix, idx[i:i + 500].contiguous(), opts=opts) for i in range(0, count, 500)])
    torch.cuda.synchronize()
    assert torch.equal(out, parts)
    cap = torch.zeros_like(out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.fit_batch(b.pix, idx, opts=opts, out=cap)
    for _ in range(2):
        cap.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, cap)


@pytest.mark.parametrize("h,w", [(3, 3), (3, 5), (7, 6), (41, 48), (128, 128)])
def test_start_up_scales_exactly(ctx, O, h, w):
    """r50 of the growth curve against the oracle (1e-6, as the far-crossing
    test), and the same bits when the pixels are scaled by powers of two: the
    fixed point's scale follows the largest pixel."""
    batch = galaxies([(h, w)] * 3, h * w)
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    opts = B.default_opts(max_pix=max(h * w, 64))
    g = B.results(ctx.centroid(b.pix, idx, opts=opts))
    o, _ = O.batch(batch.pix.numpy(), batch.offset.numpy(), batch.h.numpy(), batch.w.numpy(), stage="centroid")
    assert np.all(np.abs(g["r50"] / o["r50"] - 1) <= 1e-6), (g["r50"], o["r50"])
    for e in (-40, 40):
        s = B.results(ctx.centroid(b.pix * 2.0 ** e, idx, opts=opts))
        assert np.array_equal(s["r50"], g["r50"]), e


@pytest.mark.parametrize("w", [44, 45])
@pytest.mark.parametrize("lead", [0, 1, 4])
def test_adjoint_alignment(ctx, O, w, lead):
    """Rows of four pixels per lane where width and offset allow it, strided
    pixels elsewhere: both against the oracle."""
    batch = galaxies([(45, w), (44, w), (17, w)], 3 + w, lead=lead)
    p = np.array([[w / 2, float(h) / 2, 0.1, -0.05, 380.0, 5.0, 1.7] for h in batch.h], np.float32)
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    chi2, dpar, dp = ctx.chi2_grad(b.pix, idx, torch.as_tensor(p).cuda(), want_dpix=True)
    torch.cuda.synchronize()
    check_adjoint(O, batch, p, chi2.cpu().numpy(), dpar.cpu().numpy(), dp.cpu().numpy())


@pytest.mark.parametrize("w", [44, 45])
def test_moment_gradient_alignment(ctx, w):
    """The same stamps at offsets 0 and 1 (vector and scalar pixel writes and
    loads): the same bits."""
    res = []
    for lead in (0, 1):
        batch = galaxies([(45, w), (44, w), (17, w)], 3 + w, lead=lead)
        b = batch.to("cuda")
        idx = B.make_index(b.offset, b.h, b.w)
        opts = B.default_opts(max_pix=45 * w)
        mom = ctx.centroid(b.pix, idx, opts=opts)
        ctx.ellipticity(b.pix, idx, mom, opts=opts)
        rng = np.random.default_rng(2)
        v = torch.as_tensor(rng.normal(size=(3, 5)).astype(np.float32)).cuda()
        tan = torch.zeros(batch.pix.numel(), device="cuda")
        tan[lead:] = torch.as_tensor(rng.normal(size=batch.pix.numel() - lead).astype(np.float32)).cuda()
        dp = ctx.moment_vjp(b.pix, idx, mom, v)
        res.append((mom, dp[lead:], ctx.moment_jvp(b.pix, idx, mom, tan)))
    torch.cuda.synchronize()
    for x, y in zip(*res):
        assert torch.equal(x, y)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("lead", [0, 1, 3])
def test_cutout_passes(ctx, O, lead, dtype):
    """Crossings inside the near square, next to its last ring and far past
    it; images below and above 2^18 pixels (three and two fixed-point pieces);
    starts that are and are not vector aligned."""
    rng = np.random.default_rng(8)
    pix, offs, hs, ws, pos = [np.zeros(lead, np.float32)], [], [], [], lead
    for k, (h, w) in enumerate([(513, 512), (511, 513), (130, 97), (700, 380), (64, 64), (1, 7)]):
        yy, xx = np.mgrid[0:h, 0:w].astype(np.float64)
        for r50 in (3.0, 24.0, 60.0):
            sig = r50 / 1.1774
            I = 100.0 * np.exp(-((xx - w / 2 + 0.2) ** 2 + (yy - h / 2 - 0.3) ** 2) / (2 * sig * sig))
            I += rng.normal(0, 0.02, (h, w))
            pix.append(I.astype(np.float32).ravel())
            offs.append(pos)
            hs.append(h)
            ws.append(w)
            pos += h * w
    batch = synth.StampBatch(pix=torch.as_tensor(np.concatenate(pix)), offset=torch.as_tensor(offs),
                             h=torch.as_tensor(hs, dtype=torch.int32), w=torch.as_tensor(ws, dtype=torch.int32),
                             truth={})
    if dtype == "bf16":
        batch = synth.encode_bf16(batch)
    batch = batch.to("cuda")
    idx = B.make_index(batch.offset, batch.h, batch.w)
    out, cidx, info = ctx.cutout(batch.pix, idx, scale=batch.scale)
    torch.cuda.synchronize()
    inf = check_cutout(O, batch, out, cidx, info)
    assert np.any(inf["r50"] < 20) and np.any(inf["r50"] > 30)


@pytest.mark.parametrize("h,w", [(15, 15), (16, 16), (16, 17), (17, 21), (22, 16), (25, 25), (23, 32), (32, 32)])
def test_star_window_remainders(ctx, O, h, w):
    """Pixel counts whose last step of 256 holds none, a few, up to three and
    more pixels per lane, with and without lanes that have all eight, in the
    Gaussian weight's loop: the star file's own comparison with the oracle."""
    rng = np.random.default_rng(h * w)
    stamps = [synth.single_stamp(h, w, n=0.5, re=float(rng.uniform(1.6, 2.4)), g1=float(rng.uniform(-0.1, 0.1)),
                                 g2=float(rng.uniform(-0.1, 0.1)), xc=w / 2 - 0.5 + float(rng.uniform(-0.4, 0.4)),
                                 yc=h / 2 - 0.5 + float(rng.uniform(-0.4, 0.4)), I0=1500.0, noise_sigma=1.0,
                                 seed=int(rng.integers(1 << 30))) for _ in range(8)]
    batch = synth.StampBatch(pix=torch.as_tensor(np.concatenate([s.astype(np.float32).ravel() for s in stamps])),
                             offset=torch.arange(8) * h * w, h=torch.full((8,), h, dtype=torch.int32),
                             w=torch.full((8,), w, dtype=torch.int32), truth={})
    mom = oracle_moments(O, batch)
    compare_stars(gpu_stars(ctx, batch, mom, "gauss"), oracle_stars(O, batch, mom, "gauss"), mom, "gauss",
                  min_converged=0.5)
