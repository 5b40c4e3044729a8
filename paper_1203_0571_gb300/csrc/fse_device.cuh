// fse_device.cuh -- device helpers shared by the estimator (fse_kernels.cu)
// and the chi^2 adjoint (fse_adjoint.cu): MUFU exp2, double-float
// accumulation, warp reductions, the strided pixel walk and the fp32 b(n)
// lookup.  Internal; each translation unit gets its own copy.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fse_internal.h"

namespace fse {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr float kLog2e = 1.4426950408889634f;
constexpr double kLn2 = 0.6931471805599453;

// ------------------------------------------------------------------ PTX
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Double-float accumulation: (hi, lo) += b, carrying the exact rounding error
// of hi + b (Knuth's two-sum) in lo.
__device__ __forceinline__ void df_add(float& hi, float& lo, float b) {
    const float s = hi + b;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (b - bb);
    hi = s;
    lo += e;
}

// ------------------------------------------------------------------ reductions
// Sums of N values over the warp in every lane.  A plain butterfly costs N
// shuffles and N adds in each of its five steps.  Here a step hands half of a
// lane's values to its partner and keeps the other half (both lanes form the
// same a + b for the values they keep), so the counts fall to N/2, N/4, ..., 1
// and each total ends in one lane (scatter_lane), from which it is read back:
// 24 shuffles and 13 adds for N = 11 instead of 55 and 55.  The additions pair
// the same lanes in the same order as the butterfly, so every bit of the
// totals is the butterfly's.
__host__ __device__ constexpr int scatter_lane(int n, int j) {
    int lane = 0;
    for (int off = 16; off > 0 && n > 1; off >>= 1) {
        const int m = (n + 1) / 2;
        if (j >= m) {
            lane |= off;
            j -= m;
        }
        n = m;
    }
    return lane;
}

// The index of the total that `lane` holds after the scatter steps, or N where
// it holds none (the padding of an odd split, or a copy of another lane's).
template <int N>
__device__ __forceinline__ int scatter_index(int lane) {
    int j = 0, n = N, real = N;   // first index, slots and totals of this lane's part
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const int m = (n + 1) / 2;
        const bool up = (lane & off) != 0;
        if (n > 1) {
            j += up ? m : 0;
            real = up ? real - m : min(real, m);
        } else if (up) {
            real = 0;
        }
        n = m;
    }
    return real > 0 ? j : N;
}

template <int N, int OFF, int CAP>
__device__ __forceinline__ void scatter_sum(float (&v)[CAP], int lane) {
    if constexpr (OFF > 0) {
        if constexpr (N > 1) {
            constexpr int M = (N + 1) / 2;
            const bool up = (lane & OFF) != 0;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const float lo = v[i], hi = M + i < N ? v[M + i < N ? M + i : 0] : 0.f;
                v[i] = (up ? hi : lo) + __shfl_xor_sync(kFull, up ? lo : hi, OFF);
            }
            scatter_sum<M, OFF / 2>(v, lane);
        } else {
            v[0] += __shfl_xor_sync(kFull, v[0], OFF);
            scatter_sum<1, OFF / 2>(v, lane);
        }
    }
}

template <int N>
__device__ __forceinline__ void warp_allsum(float (&v)[N]) {
    if constexpr (N < 3) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
            for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(kFull, v[i], off);
        }
    } else {
        scatter_sum<N, 16>(v, threadIdx.x & 31);
        const float mine = v[0];
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __shfl_sync(kFull, mine, scatter_lane(N, i));
    }
}

__device__ __forceinline__ long long warp_allsum_ll(long long v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
    return v;
}

// (hi, lo) + (oh, ol) with the exact rounding error of hi + oh.  Both partners
// of an exchange form the same pair.
__device__ __forceinline__ void df_merge(float& hi, float& lo, float oh, float ol) {
    const float s = hi + oh;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (oh - bb);
    lo = (lo + ol) + e;
    hi = s;
}

// Sum of (hi, lo) pairs over the warp, by the same exchange as warp_allsum:
// 44 shuffles and 12 pair additions for N = 10 instead of 100 and 50.  Three
// pairs keep the butterfly: with its longer chain the exchange made the Moffat
// star kernel 1 % slower (20,000 stars of 48x48, 546 to 551 us), where two
// pairs make the Gaussian one 9 % faster (50,000 of 32x32, 441 to 401 us).
template <int N, int OFF, int CAP>
__device__ __forceinline__ void scatter_sum_df(float (&hi)[CAP], float (&lo)[CAP], int lane) {
    if constexpr (OFF > 0) {
        constexpr int M = (N + 1) / 2;
        const bool up = N > 1 && (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            float kh = hi[i], kl = lo[i], sh = hi[i], sl = lo[i];
            if constexpr (N > 1) {
                const bool pair = M + i < N;
                const float bh = pair ? hi[pair ? M + i : 0] : 0.f, bl = pair ? lo[pair ? M + i : 0] : 0.f;
                kh = up ? bh : hi[i];
                kl = up ? bl : lo[i];
                sh = up ? hi[i] : bh;
                sl = up ? lo[i] : bl;
            }
            const float oh = __shfl_xor_sync(kFull, sh, OFF);
            const float ol = __shfl_xor_sync(kFull, sl, OFF);
            df_merge(kh, kl, oh, ol);
            hi[i] = kh;
            lo[i] = kl;
        }
        scatter_sum_df<M, OFF / 2>(hi, lo, lane);
    }
}

template <int N>
__device__ __forceinline__ void warp_allsum_df(float (&hi)[N], float (&lo)[N]) {
    if constexpr (N == 1 || N == 3) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const float oh = __shfl_xor_sync(kFull, hi[i], off);
                const float ol = __shfl_xor_sync(kFull, lo[i], off);
                df_merge(hi[i], lo[i], oh, ol);
            }
        }
    } else {
        scatter_sum_df<N, 16>(hi, lo, threadIdx.x & 31);
        const float mh = hi[0], ml = lo[0];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            hi[i] = __shfl_sync(kFull, mh, scatter_lane(N, i));
            lo[i] = __shfl_sync(kFull, ml, scatter_lane(N, i));
        }
    }
}

// Fixed-point pieces of a pixel.  The growth curve sums q = rn(v 2^S), a
// 64-bit integer, exactly.  q = q2 2^(2B) + q1 2^B + q0 with signed pieces
// |q0|, |q1| <= 2^(B-1): with B small enough for the number of pixels no
// piece's sum can leave 32 bits, so native 32-bit adds (registers,
// shared-memory atomics) hold them exactly.
// Each piece is the nearest integer to what is left of v, by adding
// 1.5 2^23 (exact to nearest even for magnitudes up to 2^22) with the scaling
// in the same FMA; the remainders are exact, and 2^B is even, so the last
// rounding is that of the whole value.  Three FMAs and a subtraction per
// piece replace the 64-bit conversion instruction, which issues once in about
// 17 cycles of an SM on this chip's fp64 pipe.
struct FixScale {
    float up2, up1, up0;   // 2^(S - 2B), 2^(S - B), 2^S
    float dn2, dn1;        // -2^(2B - S), -2^(B - S)
    int B;
    bool wide;             // the scale does not bound q: convert in 64 bits
};

// The scale of a stamp or image of npix pixels with largest magnitude amax,
// amax * npix * 2^S < 2^62, and pieces of b bits (at most 22, for the rounding
// adds); the caller chooses b so that its sums of pieces stay below 2^31.
__device__ __forceinline__ FixScale fix_scale(float amax, int npix, int b) {
    int e;
    const float top = amax * static_cast<float>(npix);
    frexpf(top, &e);
    int S = 62 - e;
    S = S > 100 ? 100 : (S < -100 ? -100 : S);
    FixScale f;
    f.B = b;
    f.up0 = ldexpf(1.f, S);
    f.up1 = ldexpf(1.f, S - f.B);
    f.up2 = ldexpf(1.f, S - 2 * f.B);
    f.dn2 = -ldexpf(1.f, 2 * f.B - S);
    f.dn1 = -ldexpf(1.f, f.B - S);
    // |q2| <= 2^(62 - 2b) / npix has to be at most 2^22 (the rounding add), or the
    // 64-bit conversion is taken; so too where the scale itself overflows
    f.wide = !(top < INFINITY) || (b < 20 && npix < 1 << (40 - 2 * b));
    return f;
}

// The pieces (plus kFixBias) of the saturated 64-bit conversion.  Out of line:
// inlined, its conversion is issued for every pixel and then not selected.
constexpr int kFixBias = 0x4B400000;
struct FixPieces {
    int q0, q1, q2;
};
__device__ __noinline__ FixPieces fix_split_wide(float y, int B) {
    const long long q = __float2ll_rn(y);
    const long long m = (1ll << B) - 1;
    return {static_cast<int>(q & m) + kFixBias, static_cast<int>((q >> B) & m) + kFixBias,
            static_cast<int>(q >> (2 * B)) + kFixBias};
}

// The pieces plus 0x4B400000 each (the bits of 1.5 2^23 + piece); with `wide`
// the pieces of the saturated 64-bit conversion in the same form.
__device__ __forceinline__ void fix_split3(const FixScale& f, float v, int& q0, int& q1, int& q2) {
    constexpr float kRound = 12582912.f;
    const float z2 = fmaf(v, f.up2, kRound);
    const float r1 = fmaf(__fsub_rn(z2, kRound), f.dn2, v);
    const float z1 = fmaf(r1, f.up1, kRound);
    const float r0 = fmaf(__fsub_rn(z1, kRound), f.dn1, r1);
    const float z0 = fmaf(r0, f.up0, kRound);
    q2 = __float_as_int(z2);
    q1 = __float_as_int(z1);
    q0 = __float_as_int(z0);
}
__device__ __forceinline__ void fix_split(const FixScale& f, float v, int& q0, int& q1, int& q2) {
    if (!f.wide) {
        fix_split3(f, v, q0, q1, q2);
    } else {
        const FixPieces w = fix_split_wide(v * f.up0, f.B);
        q0 = w.q0;
        q1 = w.q1;
        q2 = w.q2;
    }
}

// The same in two pieces, q = q1 2^B + q0, where |q| < 2^62 / npix < 2^(B + 22).
__device__ __forceinline__ void fix_split2(const FixScale& f, float v, int& q0, int& q1) {
    constexpr float kRound = 12582912.f;
    const float z1 = fmaf(v, f.up1, kRound);
    const float r0 = fmaf(__fsub_rn(z1, kRound), f.dn1, v);
    q1 = __float_as_int(z1);
    q0 = __float_as_int(fmaf(r0, f.up0, kRound));
}

__device__ __forceinline__ long long fix_join(const FixScale& f, int s0, int s1, int s2) {
    return static_cast<long long>(s0) + static_cast<long long>(s1) * (1ll << f.B) +
           static_cast<long long>(static_cast<unsigned long long>(static_cast<long long>(s2)) << (2 * f.B));
}

// ceil(sqrt(d2)) for an integer 0 <= d2 < 2^23 (any two pixels of an image with
// sides up to 2048), with one MUFU operation and integer arithmetic: d2
// becomes a float through the bits of 2^23 + d2, and the root is rounded to
// the nearest integer k0 by adding 2^23 (whose ulp is 1).  sqrt.approx.f32 is
// within about 2^-22 relative of the square root, under 1e-3 here, so k0 is
// the floor or the ceiling of the true root, and the comparison k0^2 < d2
// turns either into the ceiling.
__device__ __forceinline__ int ring_of(int d2) {
    const float f = __int_as_float(0x4B000000 | d2) - 8388608.f;
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(f));
    const int k0 = __float_as_int(r + 8388608.f) - 0x4B000000;
    return k0 + (k0 * k0 < d2 ? 1 : 0);
}

// Pixel iterator: thread t handles p = t, t + nt, ... of a w-wide stamp.
struct PixelWalk {
    int row, col, dr, dc, w;
    __device__ PixelWalk(int t, int w_, int nt = 32) : w(w_) {
        row = t / w;
        col = t - row * w;
        dr = nt / w;
        dc = nt - dr * w;
    }
    __device__ __forceinline__ void next() {
        col += dc;
        row += dr;
        if (col >= w) {
            col -= w;
            ++row;
        }
    }
};

// Pixel coordinates of p = t, t + nt, ... of a w-wide stamp as floats.  They
// are integers, so every step is exact, and so is t = coordinate - centre.
struct FWalk {
    float c, r, dc, dr, wf;
    __device__ FWalk(int t, int w, int nt = 32) {
        const int row = t / w;
        c = static_cast<float>(t - row * w);
        r = static_cast<float>(row);
        dr = static_cast<float>(nt / w);
        dc = static_cast<float>(nt - (nt / w) * w);
        wf = static_cast<float>(w);
    }
    __device__ __forceinline__ void next() {
        c += dc;
        r += dr;
        if (c >= wf) {
            c -= wf;
            r += 1.f;
        }
    }
};

// The moment sums run over the pixels whose weight W = 2^(-R^2 log2(e) /
// (2 s_w^2)) is at least 2^-40, i.e. R^2 <= 80 ln 2 s_w^2: a pixel outside
// adds less than 2^-40 |I| |theta|^k to a sum, so all of them together move
// the centre by less than 2^-40 sum|I| max|theta| / sum I W (below 1e-9 px on
// the benchmark's faintest stamps) and g and s_w by as little.  The ellipse
// A t1^2 + B t2^2 - 4 g2 t1 t2 <= Rc^2 (Eq. A1; the determinant of the form
// is (1 - |g|^2)^2) lies inside |t1| <= Rc sqrt(B) / (1 - |g|^2), |t2| <=
// Rc sqrt(A) / (1 - |g|^2); the box adds a pixel of margin and is cut to the
// stamp (2^15 px is past any: the gradients take strips of up to FSE_MAX_PIX
// pixels).  (A record with |g| > 1 gets the whole stamp, or a box of the centre's
// neighbours where the ellipse is narrower than that.)  Compact objects (stars, small galaxies) cover a fraction of their
// stamp, which is the work saved.
constexpr float kWeightCut = 7.4446500f;   // sqrt(80 ln 2)

struct Box {
    int r0, c0;   // first row and column
    int bh, bw;   // rows and columns (at least one each)
    // stamp index of the box's last pixel
    __device__ __forceinline__ int last(int w) const { return (r0 + bh - 1) * w + c0 + bw - 1; }
};

__host__ __device__ __forceinline__ Box weight_box(float xc, float yc, float g1, float g2, float sw, int h, int w) {
    const float gg = g1 * g1 + g2 * g2;
    const float rc = kWeightCut * sw / (1.f - gg);
    const float hx = fminf(rc * sqrtf(1.f + gg + 2.f * g1) + 1.f, 32768.f);
    const float hy = fminf(rc * sqrtf(1.f + gg - 2.f * g1) + 1.f, 32768.f);
    Box b;
    b.c0 = max(0, static_cast<int>(floorf(xc - hx)));
    b.r0 = max(0, static_cast<int>(floorf(yc - hy)));
    const int c1 = min(w - 1, static_cast<int>(ceilf(xc + hx)));
    const int r1 = min(h - 1, static_cast<int>(ceilf(yc + hy)));
    // a centre outside the stamp (the iteration then stops) or a non-finite
    // state falls back to the whole stamp
    if (!(c1 >= b.c0 && r1 >= b.r0) || !(hx > 0.f && hy > 0.f)) {
        b.c0 = b.r0 = 0;
        b.bw = w;
        b.bh = h;
    } else {
        b.bw = c1 - b.c0 + 1;
        b.bh = r1 - b.r0 + 1;
    }
    return b;
}

// a / b for 0 <= a <= 256 and 1 <= b, from ib = 1 / b to a few ulps: for b <= 256
// (a + 1/2) / b lies at least 1/512 from every integer, and the product is off by
// less than 1e-4; above, both are below 1.
__host__ __device__ __forceinline__ int div_small(int a, float ib) {
    return static_cast<int>((static_cast<float>(a) + 0.5f) * ib);
}

// The pixels q = t, t + nt, ... of a box, row-major within it (the stamp
// index p grows with q, so a walk ends once p passes the box's last pixel;
// a thread with t beyond the box starts past it): their offsets
// (column - xr, row - yr) from the reference pixel and their index in the
// stamp of width w.  The offsets are integers below 2^24, exact in fp32, so
// stepping them with float adds gives the same values as converting the
// integer offsets, without a conversion per pixel.
struct BoxWalk {
    float u, v;
    int p;
    float du, dv, wrap, fbw;
    int dp, dwrap;
    __device__ __forceinline__ BoxWalk(int t, const Box& b, int w, int nt, int xr, int yr) {
        fbw = static_cast<float>(b.bw);
        const float ib = __fdividef(1.f, fbw);
        const int row = div_small(t, ib), col = t - row * b.bw;
        const int dr = div_small(nt, ib), dc = nt - dr * b.bw;
        u = static_cast<float>(b.c0 + col - xr);
        v = static_cast<float>(b.r0 + row - yr);
        p = (b.r0 + row) * w + b.c0 + col;
        du = static_cast<float>(dc);
        dv = static_cast<float>(dr);
        wrap = static_cast<float>(b.c0 + b.bw - xr);
        dp = dr * w + dc;
        dwrap = w - b.bw;
    }
    __device__ __forceinline__ void next() {
        u += du;
        v += dv;
        p += dp;
        if (u >= wrap) {
            u -= fbw;
            v += 1.f;
            p += dwrap;
        }
    }
};

// The first candidate of the growth curve's crossing ring from a recorded r50 =
// (k - 1) + frac, frac in (0, 1].  The record is the caller's, so a radius past
// the stamp (infinity included) stops at the ring h + w + 8: every pixel lies
// within h + w, so the search's eight steps end without a crossing, as they do
// from any farther ring, and neither the ring's box nor k^2 can leave 32 bits.
// NaN and radii up to 1/2 start at the brightest pixel.
__host__ __device__ inline int ring_guess(float r50, int h, int w) {
    const int far = h + w + 8;
    if (!(r50 > 0.5f)) return 0;
    return r50 < static_cast<float>(far) ? static_cast<int>(ceilf(r50)) : far;
}

// b(n), b'(n) in fp32 from a table of (b, b') at n = kBnLo + k kBnStep:
// cubic Hermite interpolation for b; b' as the linear interpolation of the
// node values of b' (error O(h^2 b''') ~ 1e-9).  Differentiating the
// interpolant of b instead would difference node values of b that carry fp32
// rounding, which the division by the step amplifies to ~1e-4.
__device__ __forceinline__ void bn_lookup_f(const float2* __restrict__ tab, float n, float* b,
                                            float* db) {
    const float x = (n - static_cast<float>(kBnLo)) * static_cast<float>(1.0 / kBnStep);
    int k = static_cast<int>(floorf(x));
    k = k < 0 ? 0 : (k > kBnNodes - 2 ? kBnNodes - 2 : k);
    const float t = x - static_cast<float>(k);
    const float2 p0 = tab[k], p1 = tab[k + 1];
    const float h = static_cast<float>(kBnStep);
    const float t2 = t * t, t3 = t2 * t;
    *b = p0.x + t2 * (3.f - 2.f * t) * (p1.x - p0.x) + (t3 - 2.f * t2 + t) * h * p0.y +
         (t3 - t2) * h * p1.y;
    *db = fmaf(t, p1.y - p0.y, p0.y);
}

}  // namespace
}  // namespace fse
