"""The chi^2 adjoint's forms (four pixels of a row per lane, lane-strided
pixels; vector and scalar accesses) in every instance of the kernel (needs a
GB300)."""
import numpy as np
import pytest
import torch

from paper_1203_0571_gb300 import binding as B
from paper_1203_0571_gb300 import synth
from test_gpu_adjoint import check_against_oracle as check_adjoint
from test_gpu_paths import galaxies

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return B.Context(0)


@pytest.fixture(scope="module")
def O(oracle):
    return oracle.get()


@pytest.mark.parametrize("want", ["chi2", "params", "pixels"])
@pytest.mark.parametrize("ivar", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("w", [44, 45])
def test_adjoint_where_a_stamp_starts(ctx, O, w, dtype, ivar, want):
    """The same stamps from elements 0 to 3 and from a buffer that itself starts
    between four-pixel boundaries: the same bits of chi^2 and of the pixel
    gradient, and the oracle's values of all outputs, at each."""
    shapes = [(45, w), (44, w), (17, w), (3, 4), (128, 128)]
    p = np.array([[sw / 2, sh / 2, 0.1, -0.05, 380.0, 5.0, 1.7] for sh, sw in shapes], np.float32)
    weights = (0.5 + np.random.default_rng(w).random(sum(sh * sw for sh, sw in shapes))).astype(np.float32)
    par = torch.as_tensor(p).cuda()
    first = None
    for lead, shift in ((0, 0), (1, 0), (2, 0), (3, 0), (0, 1), (4, 0)):
        batch = galaxies(shapes, 3 + w, lead=lead)
        if dtype == "bf16":
            batch = synth.encode_bf16(batch)
        n = batch.pix.numel()
        pix = torch.zeros(n + 8, dtype=batch.pix.dtype, device="cuda")[shift:shift + n].copy_(batch.pix)
        iv = None
        if ivar:
            iv = torch.ones(n + 8, device="cuda")[shift:shift + n]
            iv[lead:] = torch.as_tensor(weights).cuda()
        b = batch.to("cuda")
        idx = B.make_index(b.offset, b.h, b.w)
        chi2, dpar, dp = ctx.chi2_grad(pix, idx, par, scale=b.scale, inv_var=iv, want_dparams=want != "chi2",
                                       want_dpix=want == "pixels")
        alone = ctx.chi2_grad(pix, idx, par, scale=b.scale, inv_var=iv, want_dparams=False)[0]
        assert torch.equal(chi2, alone), (lead, shift)
        if dpar is not None:
            check_adjoint(O, batch, p, chi2.cpu().numpy(), dpar.cpu().numpy(), None if dp is None else dp.cpu().numpy(),
                          ivar=None if iv is None else iv.cpu().numpy())
        got = [chi2] if dp is None else [chi2, dp[lead:]]
        first = first or got
        for k, (x, y) in enumerate(zip(got, first)):
            assert torch.equal(x, y), (lead, shift, k, float((x - y).abs().max()))
