"""Index and rounding steps that the kernels take from fse_device.cuh: the header
itself, compiled for the host (its __device__ functions are plain ones there;
the few intrinsics that the steps use are given below) and run on the CPU."""
import ctypes
import os
import re
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

from paper_1203_0571_gb300 import _build

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>
#ifndef __noinline__
#define __noinline__
#endif
using std::max;
using std::min;
static struct { int x; } threadIdx;
template <class T> T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T> T __shfl_sync(unsigned, T v, int) { return v; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fdividef(float a, float b) { return a / b; }
static int __float_as_int(float f) { int i; memcpy(&i, &f, 4); return i; }
static float __int_as_float(int i) { float f; memcpy(&f, &i, 4); return f; }
static long long __float2ll_rn(float f) {   // saturating, as the instruction
    return f >= 0x1p63f ? 0x7fffffffffffffffll : f < -0x1p63f ? -0x7fffffffffffffffll - 1 : llrintf(f);
}
#include "fse_device.cuh"
extern "C" int ring_guess(float r50, int h, int w) { return fse::ring_guess(r50, h, w); }
extern "C" int div_small(int a, float ib) { return fse::div_small(a, ib); }
extern "C" void weight_box(float xc, float yc, float g1, float g2, float sw, int h, int w, int* out) {
    const fse::Box b = fse::weight_box(xc, yc, g1, g2, sw, h, w);
    out[0] = b.r0; out[1] = b.c0; out[2] = b.bh; out[3] = b.bw;
}
extern "C" int fix_exponent(float amax, int npix, int b, int* wide) {
    const fse::FixScale f = fse::fix_scale(amax, npix, b);
    *wide = f.wide;
    return ilogbf(f.up0);
}
// the pieces of n values (two: q2 = 0) and what they join to
extern "C" void pieces(float amax, int npix, int b, int two, const float* v, int n, int* q, long long* joined) {
    const fse::FixScale f = fse::fix_scale(amax, npix, b);
    for (int i = 0; i < n; ++i) {
        int* o = q + 3 * i;
        o[2] = fse::kFixBias;
        if (two) fse::fix_split2(f, v[i], o[0], o[1]);
        else fse::fix_split(f, v[i], o[0], o[1], o[2]);
        for (int k = 0; k < 3; ++k) o[k] -= fse::kFixBias;
        joined[i] = fse::fix_join(f, o[0], o[1], o[2]);
    }
}
extern "C" int scatter_lane(int n, int j) { return fse::scatter_lane(n, j); }
template <int N> static int index_of(int n, int lane) {
    if (n == N) return fse::scatter_index<N>(lane);
    if constexpr (N < 32) return index_of<N + 1>(n, lane);
    return -1;
}
extern "C" int scatter_index(int n, int lane) { return index_of<2>(n, lane); }
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("steps")
    src, lib = d / "steps.cc", d / "steps.so"
    src.write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    r = subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fwrapv", "-w", "-shared",
                        "-fPIC", "-I" + cuda, "-I" + _build.CSRC, "-I" + _build.INCLUDE, str(src), "-o", str(lib)],
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


def constant(src, name):
    with open(os.path.join(_build.CSRC, src)) as f:
        return int(re.search(r"constexpr int %s = (\d+);" % name, f.read())[1])


def split(steps, amax, npix, b, two, v):
    v = np.ascontiguousarray(v, np.float32)
    q, joined = np.zeros((v.size, 3), np.int32), np.zeros(v.size, np.int64)
    steps.pieces(ctypes.c_float(amax), npix, b, int(two), v.ctypes.data_as(ctypes.c_void_p), v.size,
                 q.ctypes.data_as(ctypes.c_void_p), joined.ctypes.data_as(ctypes.c_void_p))
    return q.astype(np.int64), joined


def exponent(steps, amax, npix, b):
    wide = ctypes.c_int()
    return steps.fix_exponent(ctypes.c_float(amax), npix, b, ctypes.byref(wide)), bool(wide.value)


# the most pixels of one ring ceil(d) = k, over the rings below K
def ring_population(K):
    k = np.arange(-K, K + 1, dtype=np.int64)
    d2 = (k[:, None] ** 2 + k[None, :] ** 2).ravel()
    r = np.sqrt(d2.astype(np.float64)).astype(np.int64)
    r += (r * r < d2)
    return int(np.bincount(r[r < K]).max())


def uses():
    """(name, npix, bits, two pieces, pixels whose pieces one 32-bit sum holds)
    of every use: the start-up's total and rings (a whole stamp), and the
    cut-out's total (a thread's block), near rings and far rings."""
    out = []
    for npix in (1, 2, 63, 255, 256, 257, 2304, 4096, 4097, 16383, 16384):
        out.append(("start-up", npix, min(22, 31 - (npix - 1).bit_length()), False, npix))
    block, bits, far = (constant("fse_cutout.cu", k) for k in ("kBlock", "kFixBits", "kFarBits"))
    near, rings = constant("fse_cutout.cu", "kNear"), constant("fse_cutout.cu", "kRings")
    pop_near, pop_far = ring_population(near + 1), ring_population(rings)
    threads = constant("fse_cutout.cu", "kCutThreads") * constant("fse_cutout.cu", "kCutCluster")
    for npix in (64, 4096, 200 * 200, (1 << 18) - 1, 1 << 18, 600 * 600, 1 << 21, 1 << 24, 1 << 28):
        for n in (4, 8):            # pixels of a 16-byte vector
            held = min(block * n, n * (-(-npix // (threads * n)) + 1))
            out.append(("total", npix, bits, npix >= 1 << 18, held))
        out.append(("near", npix, bits, False, min(pop_near, npix)))
        out.append(("far", npix, far, False, min(pop_far, npix)))
    return out


@pytest.mark.parametrize("name", ["start-up", "total", "near", "far"])
def test_fixed_point_pieces(steps, name):
    """The pieces join to rn(v 2^S), ties to even, for every pixel; S is the
    largest with |v| npix 2^S < 2^62; and no 32-bit sum of as many pieces as a use
    adds up can leave 32 bits."""
    for _, npix, b, two, held in (u for u in uses() if u[0] == name):
        rng = np.random.default_rng(npix)
        for amax in (np.float32(3.7e4), np.float32(2.0 ** 20 * (1 - 2.0 ** -24)), np.float32(1e-3)):
            S, wide = exponent(steps, amax, npix, b)
            assert wide == (npix << (2 * b) < 1 << 40)
            top = F(float(np.float32(amax * np.float32(npix))))
            assert F(2) ** 61 <= top * F(2) ** S < F(2) ** 62
            v = np.concatenate([rng.normal(0, float(amax) / 4, 200), rng.uniform(-1, 1, 100) * float(amax),
                                rng.normal(0, 2.0 ** -S, 40), (np.arange(-8, 9) + 0.5) * 2.0 ** -S,
                                float(amax) * (1 - np.arange(64) * 2.0 ** -24), [0.0, float(amax), -float(amax)]])
            v = v.astype(np.float32)
            v = v[np.abs(v) <= amax]
            q, joined = split(steps, amax, npix, b, two, v)
            assert [int(x) for x in joined] == [round(F(float(x)) * F(2) ** S) for x in v]
            limit = [1 << b if wide else 1 << (b - 1)] * 2 + [(1 << 62) // npix // (1 << 2 * b) + 1]
            if two:
                limit[1:] = [(1 << 62) // npix // (1 << b) + 1, 0]
            assert np.all(np.abs(q).max(0) <= limit)
            assert all(held * x < 1 << 31 for x in limit), (npix, b, held, limit)


def test_saturated_values_join_to_themselves(steps):
    """Where amax npix overflows fp32 the values saturate at 64 bits; their
    pieces are not negative but for the last, so rings of up to 2^(31 - b) pixels
    (the far rings' and the near ones') hold their sums."""
    big = np.float32(2.0 ** 110)
    v = np.array([big, -big, 1.0, -1.0, 0.7, -0.7, 0.0, 3e-19], np.float32)
    for b, npix in ((constant("fse_cutout.cu", "kFixBits"), 1 << 21), (constant("fse_cutout.cu", "kFarBits"), 1 << 21)):
        assert exponent(steps, big, npix, b)[1]
        q, joined = split(steps, big, npix, b, False, v)
        S = exponent(steps, big, npix, b)[0]
        want = [min(max(round(F(float(x)) * F(2) ** S), -(1 << 63)), (1 << 63) - 1) for x in v]
        assert [int(x) for x in joined] == want
        assert np.all((q[:, :2] >= 0) & (q[:, :2] < 1 << b))
    assert ring_population(constant("fse_cutout.cu", "kRings")) << constant("fse_cutout.cu", "kFarBits") < 1 << 31
    assert ring_population(constant("fse_cutout.cu", "kNear") + 1) << constant("fse_cutout.cu", "kFixBits") < 1 << 31


@pytest.mark.parametrize("n", list(range(2, 33)))
def test_exchange_leaves_each_total_in_its_lane(steps, n):
    """The lanes that the header names hold the totals after the halving
    exchange, each total once."""
    rng = np.random.default_rng(n)
    v = rng.integers(-1000, 1000, (32, n))
    want, m, off = v.sum(0), n, 16
    while off:
        half = (m + 1) // 2
        up = ((np.arange(32) & off) != 0)[:, None]
        if m > 1:
            hi = np.zeros((32, half), v.dtype)
            hi[:, :m - half] = v[:, half:m]
            lo = v[:, :half]
            v, m = np.where(up, hi, lo) + np.where(up, lo, hi)[np.arange(32) ^ off], half
        else:
            v = v + v[np.arange(32) ^ off]
        off >>= 1
    assert [int(v[steps.scatter_lane(n, j), 0]) for j in range(n)] == want.tolist()
    held = [steps.scatter_index(n, lane) for lane in range(32)]
    for j in range(n):
        assert held.count(j) == 1 and int(v[held.index(j), 0]) == want[j]
    assert set(held) <= set(range(n + 1))
