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

// Pixel coordinates of p = t, t + 32, ... of a w-wide stamp as floats.  They
// are integers, so every step is exact, and so is t = coordinate - centre.
struct FWalk {
    float c, r, dc, dr, wf;
    __device__ FWalk(int t, int w) {
        const int row = t / w;
        c = static_cast<float>(t - row * w);
        r = static_cast<float>(row);
        dr = static_cast<float>(32 / w);
        dc = static_cast<float>(32 - (32 / w) * w);
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
