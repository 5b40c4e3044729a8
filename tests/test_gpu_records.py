"""Moment records whose fields lie outside the range that the estimator writes
(needs a GB300): the gradients of the moment fixed point take them as data."""
import numpy as np
import pytest
import torch

from paper_1203_0571_gb300 import binding as B
from test_gpu_paths import galaxies

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return B.Context(0)


@pytest.mark.parametrize("w", [44, 45])
def test_radius_past_the_stamp(ctx, w):
    """A recorded r50 past the stamp, infinite or not a number is only a wrong
    first guess of the crossing ring: past the stamp the search ends without
    one (sigma_w then does not depend on the pixels), whatever the value; NaN
    starts at the brightest pixel, as 0 does."""
    batch = galaxies([(45, w)] * 2, 11 + w)
    b = batch.to("cuda")
    idx = B.make_index(b.offset, b.h, b.w)
    opts = B.default_opts(max_pix=45 * w)
    mom = ctx.centroid(b.pix, idx, opts=opts)
    ctx.ellipticity(b.pix, idx, mom, opts=opts)
    rng = np.random.default_rng(w)
    v = torch.as_tensor(rng.normal(size=(2, 5)).astype(np.float32)).cuda()
    tan = torch.as_tensor(rng.normal(size=batch.pix.numel()).astype(np.float32)).cuda()

    def grads(r50):
        m = mom.clone()
        m.view(torch.float32)[:, 15] = r50
        st = torch.zeros(2, dtype=torch.int32, device="cuda")
        return ctx.moment_vjp(b.pix, idx, m, v), ctx.moment_jvp(b.pix, idx, m, tan, status=st), st

    for same, values in ((1.0e4, (300.0, 3.0e9, 1.0e30, float("inf"))), (0.0, (float("nan"), float("-inf")))):
        want = grads(same)
        assert torch.equal(want[2], torch.zeros_like(want[2]))
        for r50 in values:
            assert all(torch.equal(x, y) for x, y in zip(grads(r50), want)), r50
    far, near = grads(1.0e4), grads(float(B.results(mom)["r50"][0]))
    assert torch.all(far[1][:, 4] == 0) and near[1][0, 4] != 0
