"""Index and rounding steps that the kernels take from fse_device.cuh, compiled
for the host from that header and run on the CPU."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_1203_0571_gb300 import _build

SOURCE = r"""
#include <math.h>
#include "fse_device.cuh"
extern "C" int ring_guess(float r50, int h, int w) { return fse::ring_guess(r50, h, w); }
extern "C" int div_small(int a, float ib) { return fse::div_small(a, ib); }
extern "C" void weight_box(float xc, float yc, float g1, float g2, float sw, int h, int w, int* out) {
    const fse::Box b = fse::weight_box(xc, yc, g1, g2, sw, h, w);
    out[0] = b.r0; out[1] = b.c0; out[2] = b.bh; out[3] = b.bw;
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("steps")
    src, lib = d / "steps.cu", d / "steps.so"
    src.write_text(SOURCE)
    r = subprocess.run([_build.nvcc()] + _build.ARCH + _build.FLAGS + ["-shared", str(src), "-o", str(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("h,w", [(1, 1), (3, 3), (7, 128), (48, 48), (47, 45), (128, 128), (1, 16384), (16384, 1)])
def test_ring_candidate_stays_in_range(steps, h, w):
    """From any recorded r50: the box of the candidate ring (and of the seven
    that the search can step to) around any pixel is a non-empty part of the
    stamp in 32-bit integers, and k^2 fits; a radius past the stamp stays past
    every pixel for eight steps down."""
    f = steps.ring_guess
    f.argtypes, f.restype = [ctypes.c_float, ctypes.c_int, ctypes.c_int], ctypes.c_int
    top = (1 << 31) - 1
    for r50 in (float("-inf"), -3.0, float("nan"), 0.0, 0.5):
        assert f(r50, h, w) == 0
    for r50 in (0.51, 1.0, 1.5, 12.3, h + w + 7.5):
        assert f(r50, h, w) == (-int(-r50 // 1) if r50 < h + w + 8 else h + w + 8)
    for r50 in (0.51, 5.0, 300.0, 46341.0, 1e6, 2147483520.0, 2.2e9, 3e9, 1e30, float("inf")):
        k = f(r50, h, w)
        if r50 >= h + w + 8:
            assert k - 7 > h + w
        for kk in range(max(k - 8, 0), k + 9):
            assert kk * kk <= top
            for pr, pc in ((0, 0), (h - 1, w - 1), (h // 2, w // 3)):
                assert pr + kk <= top and pc + kk <= top
                r0, c0 = max(0, pr - kk), max(0, pc - kk)
                bh, bw = min(h - 1, pr + kk) - r0 + 1, min(w - 1, pc + kk) - c0 + 1
                assert 1 <= bh <= h - r0 and 1 <= bw <= w - c0
                assert 0 <= (r0 + bh - 1) * w + c0 + bw - 1 < h * w


@pytest.mark.parametrize("case", ["stamps", "records", "strips"])
def test_weight_box_holds_the_weight(steps, case):
    """Every pixel with W >= 2^-40 lies in the box: for the weights that the
    iteration takes on stamps; for records with |g| >= 1, which only the gradients
    see; and on the strips of up to FSE_MAX_PIX pixels that the gradients accept."""
    f = steps.weight_box
    f.argtypes = [ctypes.c_float] * 5 + [ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    rng = np.random.default_rng(5)
    for _ in range(1500 if case != "strips" else 300):
        if case == "strips":
            long, short = int(rng.integers(129, 16385)), 1
            short = int(rng.integers(1, 16384 // long + 1))
            h, w = (long, short) if rng.random() < 0.5 else (short, long)
            sw = float(np.exp(rng.uniform(np.log(0.5), np.log(4000.0))))
        else:
            h, w = (int(v) for v in rng.integers(1, 129, 2))
            sw = float(rng.uniform(0.05, 40.0))
        ga = rng.uniform(1.0, 8.0) if case == "records" else rng.uniform(0, 0.949)
        phi = rng.uniform(0, 2 * np.pi)
        g1, g2, sw = (np.float32(v) for v in (ga * np.cos(phi), ga * np.sin(phi), sw))
        xc, yc = np.float32(rng.uniform(-0.5, w - 0.5)), np.float32(rng.uniform(-0.5, h - 0.5))
        out = (ctypes.c_int * 4)()
        f(xc, yc, g1, g2, sw, h, w, out)
        r0, c0, bh, bw = out
        assert 0 <= r0 and 0 <= c0 and bh >= 1 and bw >= 1 and r0 + bh <= h and c0 + bw <= w
        t1 = np.arange(w)[None, :] - float(xc)
        t2 = np.arange(h)[:, None] - float(yc)
        a, b = float(g1), float(g2)
        R2 = ((1 - a) ** 2 + b * b) * t1 ** 2 + ((1 + a) ** 2 + b * b) * t2 ** 2 - 4 * b * t1 * t2
        outside = R2 <= 80 * np.log(2) * float(sw) ** 2
        outside[r0:r0 + bh, c0:c0 + bw] = False
        assert not outside.any(), (h, w, g1, g2, sw, xc, yc, (r0, c0, bh, bw))


def test_box_row_of_any_width(steps):
    """The box walk's row from an approximate reciprocal, for every width that the
    gradients' boxes can have."""
    f = steps.div_small
    f.argtypes, f.restype = [ctypes.c_int, ctypes.c_float], ctypes.c_int
    for b in list(range(1, 300)) + [511, 512, 4097, 16384]:
        for ulp in (-4, 0, 4):      # of the reciprocal
            ib = float((np.float32(1.0 / b).view(np.int32) + np.int32(ulp)).view(np.float32))
            for a in {0, 31, 32, 255, 256} | {v for k in range(257 // b + 1) for v in (k * b - 1, k * b) if 0 <= v <= 256}:
                assert f(a, ib) == a // b, (a, b, ulp)


def test_warp_wide_instructions_meet_a_whole_warp():
    """Every tensor-memory instruction that a whole warp has to execute together
    (.sync.aligned) stands in a function that begins by bringing the warp
    together: its callers branch per lane."""
    for src in _build.SOURCES:
        with open(os.path.join(_build.CSRC, src)) as f:
            body, found = [], 0
            for line in f:
                if re.match(r"(template|__device__|__global__|\}|struct )", line):
                    body = []
                body.append(line.strip())
                if re.search(r'"tcgen05\.[^"]*\.sync\.aligned', line):
                    found += 1
                    assert body[0].startswith("__device__ __forceinline__ void tm_"), (src, line)
                    assert body[1] == "__syncwarp();", (src, body[0])
            assert src != "fse_kernels.cu" or found >= 5
