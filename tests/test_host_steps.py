"""Index and rounding steps that the kernels take from fse_device.cuh, compiled
for the host from that header and run on the CPU."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_1203_0571_gb300 import _build

SOURCE = r"""
#include <math.h>
#include "fse_device.cuh"
extern "C" int ring_guess(float r50, int h, int w) { return fse::ring_guess(r50, h, w); }
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
