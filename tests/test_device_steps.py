"""Integer and rounding steps of the kernels, restated on the CPU.

- div_small: the row of a box pixel, (a + 1/2) times an approximate 1 / b;
- the three (or two) pieces of a fixed-point pixel value, each a rounding add
  of what is left, against the nearest integer of v 2^S;
- the lanes that hold the totals after the halving exchange of a warp sum.
"""
from fractions import Fraction as F

import numpy as np
import pytest


def test_div_small_exhaustive():
    a = np.arange(0, 257, dtype=np.float32) + np.float32(0.5)
    for b in range(1, 129):
        want = np.arange(0, 257) // b
        for ulp in (-4, 0, 4):      # of the approximate reciprocal
            ib = np.float32(1.0 / b)
            ib = (ib.view(np.int32) + np.int32(ulp)).view(np.float32)
            assert np.array_equal((a * ib).astype(np.int32), want), (b, ulp)


@pytest.mark.parametrize("npix,b", [(1, 22), (255, 22), (256, 22), (2304, 19), (16384, 17), (1 << 18, 22),
                                    (1 << 24, 22)])
def test_fixed_point_pieces_are_the_nearest_integer(npix, b):
    """Exact rational arithmetic: every remainder of the chain is an fp32
    value (so the device's fused multiply-adds round only where they add
    1.5 2^23), every piece lies within the range of that rounding, and the
    pieces rebuild rn(v 2^S), ties to even."""
    rng = np.random.default_rng(npix)
    amax = np.float32(3.7e4)
    top = amax * np.float32(npix)
    S = 62 - int(np.frexp(top)[1])
    v = np.concatenate([rng.normal(0, float(amax) / 4, 300), rng.uniform(-1, 1, 100) * float(amax),
                        rng.normal(0, 1e-12, 40), rng.normal(0, 2.0 ** -S, 60),
                        (np.arange(-8, 9) + 0.5) * 2.0 ** -S, [0.0, float(amax), -float(amax)]]).astype(np.float32)
    v = v[np.abs(v) <= amax]
    two = 1 << b
    pieces = 2 if npix >= 1 << 18 else 3
    for x in v:
        r = F(float(x))
        q = []
        for k in range(pieces - 1, -1, -1):
            p = round(r * F(2) ** (S - k * b))             # to nearest, ties to even
            assert abs(p) <= 1 << 22
            r -= p * F(2) ** (k * b - S)
            if k:
                assert F(float(np.float32(float(r)))) == r   # the remainder is exact in fp32
            q.append(p)
        assert sum(p * two ** k for k, p in zip(range(pieces - 1, -1, -1), q)) == round(F(float(x)) * F(2) ** S)
        if pieces == 3:
            assert all(abs(p) * npix < 1 << 31 for p in q) or b > 17 and npix <= 1 << (30 - b + 1)


def scatter_lane(n, j):
    lane, off = 0, 16
    while off > 0 and n > 1:
        m = (n + 1) // 2
        if j >= m:
            lane |= off
            j -= m
        n = m
        off >>= 1
    return lane


def scatter_index(n_all, lane):
    j, n, real, off = 0, n_all, n_all, 16
    while off:
        m = (n + 1) // 2
        up = bool(lane & off)
        if n > 1:
            j += m if up else 0
            real = real - m if up else min(real, m)
        elif up:
            real = 0
        n = m
        off >>= 1
    return j if real > 0 else n_all


@pytest.mark.parametrize("n", list(range(2, 33)))
def test_exchange_leaves_each_total_in_its_lane(n):
    rng = np.random.default_rng(n)
    x = rng.integers(-1000, 1000, (32, n))
    want = x.sum(0)
    v, m, off = x.copy(), n, 16
    while off:
        part = np.arange(32) ^ off
        up = (np.arange(32) & off) != 0
        if m > 1:
            half = (m + 1) // 2
            hi = np.zeros((32, half), dtype=x.dtype)
            hi[:, :m - half] = v[:, half:m]
            lo = v[:, :half]
            keep, send = np.where(up[:, None], hi, lo), np.where(up[:, None], lo, hi)
            v, m = keep + send[part], half
        else:
            v = v + v[part]
        off >>= 1
    assert [int(v[scatter_lane(n, j), 0]) for j in range(n)] == want.tolist()
    held = [scatter_index(n, lane) for lane in range(32)]
    for j in range(n):
        assert held.count(j) == 1 and int(v[held.index(j), 0]) == want[j]
