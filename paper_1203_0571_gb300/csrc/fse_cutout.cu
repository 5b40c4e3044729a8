// fse_cutout.cu -- the cut-out of Sec. 4.1: from each large image, the
// square of side side_factor * r50 (six in the paper) around the brightest
// pixel, r50 from the growth curve around that pixel.  The cut-outs are
// packed back to back into a stamp buffer with its fse_stamp index, ready for
// the estimator.
//
// Three launches:
//   cutout_measure_kernel  one cluster of 8 CTAs per image, each over an
//                          eighth of its pixels: brightest pixel (ties to the
//                          lowest row-major index), exact 64-bit fixed-point
//                          total and ring histograms (the sums do not depend
//                          on their order), merged through distributed shared
//                          memory; r50 and the square, cut to the image;
//   cutout_scan_kernel     one CTA: exclusive prefix sum of h * w into the
//                          offsets of the packed buffer;
//   cutout_copy_kernel     one CTA per cut-out, a warp per row, lane loads.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cooperative_groups.h>

#include "fse_device.cuh"
#include "fse_internal.h"

namespace cg = cooperative_groups;

namespace fse {
namespace {

constexpr int kCutThreads = 256;
constexpr int kCutWarps = kCutThreads / 32;
constexpr int kCutCluster = 8;   // CTAs per image (a portable cluster size)
// Rings of the growth-curve histogram; a crossing beyond the last ring (r50
// above 2047 px) takes the largest side and reports r50 = NaN.
constexpr int kRings = 2048;
constexpr double kSqrt2Ln2D = 1.1774100225154747;

template <int DT>
__device__ __forceinline__ float img_pix(const CutoutArgs& a, int64_t off, float sc) {
    return DT == FSE_BF16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(a.images)[off]) * sc
                          : __ldg(static_cast<const float*>(a.images) + off);
}

// The ring k = ceil(sqrt(d2)) of a squared distance d2 < 2^31, with one MUFU
// operation: sqrt.approx of the float nearest d2 is within about 2^-22
// relative of the root, under 0.012 for roots up to 46341, so it truncates to
// c - 2, c - 1 or c, c the ceiling; two conditional increments give c (k * k
// stays below 2^32).
__device__ __forceinline__ unsigned ring_ceil32(unsigned d2) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(__uint2float_rn(d2)));
    unsigned k = __float2uint_rz(r);
    k += k * k < d2 ? 1u : 0u;
    k += k * k < d2 ? 1u : 0u;
    return k;
}

// 16 bytes of an image: four floats or eight bf16, decoded.
template <int DT>
struct ImgVec;
template <>
struct ImgVec<FSE_F32> {
    static constexpr int N = 4;
    __device__ static __forceinline__ void get(const uint4& r, float, float (&v)[N]) {
        v[0] = __uint_as_float(r.x);
        v[1] = __uint_as_float(r.y);
        v[2] = __uint_as_float(r.z);
        v[3] = __uint_as_float(r.w);
    }
};
template <>
struct ImgVec<FSE_BF16> {
    static constexpr int N = 8;
    __device__ static __forceinline__ void get(const uint4& r, float sc, float (&v)[N]) {
        const unsigned u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {   // a bf16 is the upper half of a float
            v[2 * i] = __uint_as_float(u[i] << 16) * sc;
            v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u) * sc;
        }
    }
};

// The range [lo, hi) of an image's pixels as a 16-byte-aligned body of vectors
// and up to N - 1 single pixels before and after it.
template <int DT>
struct ImgRange {
    static constexpr int N = ImgVec<DT>::N;
    const uint4* body;
    int lo, head, nvec, tail;   // first pixel; pixels before the body, vectors, pixels after
    __device__ __forceinline__ ImgRange(const CutoutArgs& a, int64_t off, int lo_, int hi) : lo(lo_) {
        constexpr int esz = 16 / N;
        const char* p = static_cast<const char*>(a.images) + (off + lo) * esz;
        const int mis = static_cast<int>(reinterpret_cast<uintptr_t>(p) & 15);
        head = ((16 - mis) & 15) / esz;
        if (head > hi - lo) head = hi - lo;
        nvec = (hi - lo - head) / N;
        tail = hi - lo - head - nvec * N;
        body = reinterpret_cast<const uint4*>(p + head * esz);
    }
    // pixel index of this thread's single pixel, or -1
    __device__ __forceinline__ int single(int t) const {
        if (t < head) return lo + t;
        return t - head < tail ? lo + head + nvec * N + (t - head) : -1;
    }
    __device__ __forceinline__ int first(int j) const { return lo + head + j * N; }
};

// max(a, |b|) that keeps a NaN of either.
__device__ __forceinline__ float max_abs_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(fabsf(b)));
    return r;
}

// One cluster of kCutCluster CTAs per image; CTA r takes the r-th of
// kCutCluster equal ranges of the image's pixels (row-major), read twice (the
// second time from L2): for the brightest pixel and the largest magnitude, and,
// with the scale that gives, for the exact total.  Both passes take 16 bytes a
// lane.  The growth curve needs only the rings up to the one that crosses half
// the total: nine images of ten cross within kNear pixels of the brightest one
// (500 synthetic images of 512x512), so the ring histogram takes the square of
// that half-side, spread over the cluster, and only where that does not reach
// half the light the whole image.  What the CTAs find goes through distributed
// shared memory and is combined in the same order in each of them, so they
// hold the same values and take the same branches.
//   500 images of 512x512 fp32 (524 MB, 0.077 ms at the copy rate), whole call:
//   0.85 ms with every pixel binned (152 instructions a pixel), 0.20 ms with the
//   square.  What is left: 0.07 ms for the first pass (DRAM), 0.02 for the second,
//   the images that need every ring (a tenth; 0.03), and the cluster barriers and
//   starts; clusters of four cost 0.03 ms more, five CTAs per SM 0.02.
constexpr int kNear = 24;                 // half-side of the square, and its last ring
constexpr int kFixBits = 22;              // piece width of the total and the near rings (at
                                          // most 200 pixels each)
constexpr int kBlock = 127;               // vectors a thread sums before it empties its pieces:
                                          // fewer than 2^10 pixels of |q0| <= 2^21 (and, of two
                                          // pieces, npix / 2^11 pixels of |q1| <= 2^40 / npix)
constexpr int kFarBits = 17;              // piece width of the whole image's rings (at most
                                          // 2^14 pixels each)
constexpr int kRun = 4;                   // consecutive pixels a thread bins at a time (2: 0.242
                                          // ms, 8: 0.232, 16: 0.253)

// The ring at which the enclosed sum first reaches half the total (k, -1 if
// none) and the sums before and after it.
struct Crossing {
    int k;
    long long prev, cur;
};

// Finds the crossing among the near rings, lane k holding ring k; one warp.
__device__ __forceinline__ void scan_near(const long long* s_ring, long long tot, int lane, Crossing* out) {
    static_assert(kNear < 32, "a ring per lane");
    const long long own = lane <= kNear ? s_ring[lane] : 0;
    long long incl = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const long long o2 = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += o2;
    }
    const unsigned hit = __ballot_sync(kFull, lane <= kNear && 2 * incl >= tot);
    const int src = hit ? __ffs(hit) - 1 : 0;
    if (lane == src) *out = {hit ? src : -1, incl - own, incl};
}

// The first `rings` ring sums of the cluster (pieces `stride` apart in `part`
// of every CTA), in this CTA's s_ring, by its first threads.
__device__ __forceinline__ void merge_rings(cg::cluster_group& cl, int* part, int stride, int rings, int tid,
                                            const FixScale& f, long long* s_ring) {
    if (tid < rings) {
        int s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int r = 0; r < kCutCluster; ++r) {
            const int* o = cl.map_shared_rank(part, r);
            s0 += o[tid];
            s1 += o[stride + tid];
            s2 += o[2 * stride + tid];
        }
        s_ring[tid] = fix_join(f, s0, s1, s2);
    }
}

// r50 and the square of one image, from its total and crossing (status 0), or
// an empty square with the status.
__device__ void write_square(const CutoutArgs& a, int64_t img, const fse_stamp& ix, uint32_t st, int pr, int pc,
                             long long tot, const Crossing& x) {
    fse_cutout_info info = {0, 0, 0, 0, 0.f, 0u};
    if (st == 0) {
        double r50;
        if (tot <= 0) {
            st |= FSE_ST_INIT_FALLBACK;
            r50 = kSqrt2Ln2D;
        } else if (x.k < 0) {
            r50 = NAN;                            // crossing beyond the last ring
        } else if (x.k == 0) {
            r50 = 0.25 * static_cast<double>(tot) / static_cast<double>(x.cur);
        } else {
            r50 = static_cast<double>(x.k - 1) +
                  static_cast<double>(tot - 2 * x.prev) / (2.0 * static_cast<double>(x.cur - x.prev));
        }
        long long side = isfinite(r50) ? static_cast<long long>(floor(a.side_factor * r50 + 0.5))
                                       : static_cast<long long>(a.max_side);
        side = side < a.min_side ? a.min_side : (side > a.max_side ? a.max_side : side);
        int r0 = pr - static_cast<int>(side / 2), c0 = pc - static_cast<int>(side / 2);
        int r1 = r0 + static_cast<int>(side), c1 = c0 + static_cast<int>(side);
        r0 = r0 < 0 ? 0 : r0;
        c0 = c0 < 0 ? 0 : c0;
        r1 = r1 > ix.h ? ix.h : r1;
        c1 = c1 > ix.w ? ix.w : c1;
        info.row0 = r0;
        info.col0 = c0;
        info.h = r1 - r0;
        info.w = c1 - c0;
        info.r50 = static_cast<float>(r50);
    }
    info.status = st;
    a.info[img] = info;
    a.out_idx[img] = {0, info.h, info.w};
}

template <int DT>
__global__ void __cluster_dims__(kCutCluster, 1, 1) __launch_bounds__(kCutThreads, 4)
    cutout_measure_kernel(CutoutArgs a) {
    constexpr int N = ImgVec<DT>::N;
    __shared__ float s_v[kCutWarps], s_amax[kCutWarps];
    __shared__ int s_i[kCutWarps];
    __shared__ long long s_tot[kCutWarps];
    // this CTA's part, read by the other CTAs of the cluster
    __shared__ float c_v, c_amax;
    __shared__ int c_i;
    __shared__ long long c_tot;
    __shared__ int c_near[3 * (kNear + 1)];
    __shared__ long long s_ring[kNear + 1];
    __shared__ int hist[3 * kRings];   // pieces of the whole image's rings
    __shared__ Crossing s_x;
    __shared__ long long s_all;
    __shared__ int s_first;
    __shared__ float s_ba;
    __shared__ int s_bi;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = static_cast<int>(cl.block_rank());
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t ncl = gridDim.x / kCutCluster;
    // every CTA of a cluster runs the same images and the same cluster
    // barriers: the loop bounds depend on the cluster alone
    for (int64_t img = blockIdx.x / kCutCluster; img < a.count; img += ncl) {
        const fse_stamp ix = a.img_idx[img];
        const long long npl = static_cast<long long>(ix.h) * ix.w;
        const bool size_ok = ix.h >= 1 && ix.w >= 1 && npl <= (1LL << 28);
        const int npix = size_ok ? static_cast<int>(npl) : 0;
        const int lo = static_cast<int>(static_cast<long long>(npix) * rank / kCutCluster);
        const int hi = static_cast<int>(static_cast<long long>(npix) * (rank + 1) / kCutCluster);
        const float sc = (DT == FSE_BF16 && a.scale) ? a.scale[img] : 1.f;
        const ImgRange<DT> rg(a, ix.offset, lo, hi);
        // pass 1: brightest pixel, largest |I| (NaN or infinite if a pixel is)
        float vmax = -INFINITY, amax = 0.f;
        int imax = 0x7fffffff, jmax = -1;
#pragma unroll 4
        for (int j = tid; j < rg.nvec; j += kCutThreads) {
            float v[N];
            ImgVec<DT>::get(__ldg(rg.body + j), sc, v);
            float m = v[0];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                m = fmaxf(m, v[i]);
                amax = max_abs_nan(amax, v[i]);
            }
            if (m > vmax) { vmax = m; jmax = j; }
        }
        if (jmax >= 0) {   // the first pixel of that vector with the value
            float v[N];
            ImgVec<DT>::get(__ldg(rg.body + jmax), sc, v);
#pragma unroll
            for (int i = N - 1; i >= 0; --i)
                if (v[i] == vmax) imax = rg.first(jmax) + i;
        }
        const int single = rg.single(tid);
        float vs = 0.f;
        if (single >= 0) {
            vs = img_pix<DT>(a, ix.offset + single, sc);
            amax = max_abs_nan(amax, vs);
            if (vs > vmax || (vs == vmax && single < imax)) { vmax = vs; imax = single; }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float ov = __shfl_xor_sync(kFull, vmax, off);
            const int oi = __shfl_xor_sync(kFull, imax, off);
            if (ov > vmax || (ov == vmax && oi < imax)) { vmax = ov; imax = oi; }
            amax = max_abs_nan(amax, __shfl_xor_sync(kFull, amax, off));
        }
        if (lane == 0) {
            s_v[warp] = vmax;
            s_i[warp] = imax;
            s_amax[warp] = amax;
        }
        __syncthreads();
        if (tid == 0) {
            float bv = s_v[0], ba = s_amax[0];
            int bi = s_i[0];
            for (int k = 1; k < kCutWarps; ++k) {
                if (s_v[k] > bv || (s_v[k] == bv && s_i[k] < bi)) { bv = s_v[k]; bi = s_i[k]; }
                ba = max_abs_nan(ba, s_amax[k]);
            }
            c_v = bv;
            c_i = bi;
            c_amax = ba;
        }
        cl.sync();   // every CTA's part of pass 1 is visible to the cluster
        for (int k = tid; k < 3 * (kNear + 1); k += kCutThreads) c_near[k] = 0;
        if (warp == 0) {
            // lane r reads CTA r's part; the lanes past the cluster repeat it
            const int r = lane & (kCutCluster - 1);
            vmax = *cl.map_shared_rank(&c_v, r);
            imax = *cl.map_shared_rank(&c_i, r);
            amax = *cl.map_shared_rank(&c_amax, r);
#pragma unroll
            for (int off = kCutCluster / 2; off > 0; off >>= 1) {
                const float ov = __shfl_xor_sync(kFull, vmax, off);
                const int oi = __shfl_xor_sync(kFull, imax, off);
                if (ov > vmax || (ov == vmax && oi < imax)) { vmax = ov; imax = oi; }
                amax = max_abs_nan(amax, __shfl_xor_sync(kFull, amax, off));
            }
            if (lane == 0) {
                s_bi = imax;
                s_ba = amax;
            }
        }
        __syncthreads();
        imax = s_bi;
        amax = s_ba;
        const bool fin = amax < INFINITY;
        const int pr = npix ? imax / ix.w : 0, pc = npix ? imax - (imax / ix.w) * ix.w : 0;
        // pass 2: the total in fixed point, and the rings of the near square
        const FixScale fx = fix_scale(amax, npix, kFixBits);
        long long tot = 0;
        if (size_ok && fin) {
            int q0, q1, q2;
            if (single >= 0) {
                fix_split(fx, vs, q0, q1, q2);
                tot = fix_join(fx, q0 - kFixBias, q1 - kFixBias, q2 - kFixBias);
            }
            const bool two = npix >= (1 << 18) && !fx.wide;   // |q| < 2^44: two pieces do
            for (int j0 = tid; j0 < rg.nvec; j0 += kBlock * kCutThreads) {
                const int jend = min(rg.nvec, j0 + kBlock * kCutThreads);
                const unsigned n = (jend - j0 + kCutThreads - 1) / kCutThreads * N;
                unsigned t0 = 0, t1 = 0, t2 = 0;   // modulo 2^32: only the difference is small
                if (two) {
#pragma unroll 4
                    for (int j = j0; j < jend; j += kCutThreads) {
                        float v[N];
                        ImgVec<DT>::get(__ldg(rg.body + j), sc, v);
#pragma unroll
                        for (int i = 0; i < N; ++i) {
                            fix_split2(fx, v[i], q0, q1);
                            t0 += q0;
                            t1 += q1;
                        }
                    }
                    t2 = n * kFixBias;
                } else if (fx.wide) {
                    // 64-bit values one by one, modulo 2^64 (their pieces run to
                    // 2^22, not to half of it either way, and a block of bf16
                    // vectors has too many of those for 32 bits)
                    unsigned long long t = 0;
#pragma unroll 1
                    for (int j = j0; j < jend; j += kCutThreads) {
                        float v[N];
                        ImgVec<DT>::get(__ldg(rg.body + j), sc, v);
#pragma unroll 1
                        for (int i = 0; i < N; ++i)
                            t += static_cast<unsigned long long>(__float2ll_rn(v[i] * fx.up0));
                    }
                    tot = static_cast<long long>(static_cast<unsigned long long>(tot) + t);
                    continue;
                } else {
#pragma unroll 2
                    for (int j = j0; j < jend; j += kCutThreads) {
                        float v[N];
                        ImgVec<DT>::get(__ldg(rg.body + j), sc, v);
#pragma unroll
                        for (int i = 0; i < N; ++i) {
                            fix_split3(fx, v[i], q0, q1, q2);
                            t0 += q0;
                            t1 += q1;
                            t2 += q2;
                        }
                    }
                }
                tot += fix_join(fx, static_cast<int>(t0 - n * kFixBias), static_cast<int>(t1 - n * kFixBias),
                                static_cast<int>(t2 - n * kFixBias));
            }
            const int r0 = max(0, pr - kNear), r1 = min(ix.h - 1, pr + kNear);
            const int c0 = max(0, pc - kNear), c1 = min(ix.w - 1, pc + kNear);
            const int bw = c1 - c0 + 1, area = (r1 - r0 + 1) * bw;
            for (int i = rank * kCutThreads + tid; i < area; i += kCutCluster * kCutThreads) {
                const int row = r0 + i / bw, col = c0 + i % bw;
                const int di = row - pr, dj = col - pc;
                const int key = ring_of(di * di + dj * dj);
                if (key <= kNear) {
                    fix_split(fx, img_pix<DT>(a, ix.offset + static_cast<int64_t>(row) * ix.w + col, sc), q0, q1, q2);
                    atomicAdd(&c_near[key], q0 - kFixBias);
                    atomicAdd(&c_near[kNear + 1 + key], q1 - kFixBias);
                    atomicAdd(&c_near[2 * (kNear + 1) + key], q2 - kFixBias);
                }
            }
        }
        tot = warp_allsum_ll(tot);
        if (lane == 0) s_tot[warp] = tot;
        __syncthreads();
        if (tid == 0) {
            long long t = 0;
            for (int k = 0; k < kCutWarps; ++k) t += s_tot[k];
            c_tot = t;
        }
        cl.sync();   // every CTA's near rings and total are complete
        if (tid == 32 * (kCutWarps - 1)) {
            long long t = 0;
#pragma unroll
            for (int r = 0; r < kCutCluster; ++r) t += *cl.map_shared_rank(&c_tot, r);
            s_all = t;
        }
        merge_rings(cl, c_near, kNear + 1, kNear + 1, tid, fx, s_ring);
        __syncthreads();
        if (warp == 0) scan_near(s_ring, s_all, lane, &s_x);
        __syncthreads();
        tot = s_all;
        if (size_ok && fin && tot > 0 && s_x.k < 0) {   // the same in every CTA
            // pass 3: the ring histogram of the whole image, without the rings
            // past the last one (they cannot cross, and the total is known).
            // Each thread bins runs of kRun consecutive pixels, so that the
            // lanes of a warp stand kRun pixels apart, mostly on different
            // rings: the three atomics of a pixel seldom meet on one address.
            const FixScale ff = fix_scale(amax, npix, kFarBits);
            const bool fast = ix.h <= 2048 && ix.w <= 2048 && !ff.wide;
            const bool narrow = ix.h <= 32768 && ix.w <= 32768;
            for (int k = tid; k < 3 * kRings; k += kCutThreads) hist[k] = 0;
            __syncthreads();
            for (long long p0 = lo + tid * kRun; p0 < hi; p0 += kCutThreads * kRun) {
                const int run = min(kRun, hi - static_cast<int>(p0));
                int row = static_cast<int>(p0) / ix.w, col = static_cast<int>(p0) % ix.w;
                int64_t at = ix.offset + p0;
                auto add = [&](int key, int q0, int q1, int q2) {
                    atomicAdd(&hist[key], q0 - kFixBias);
                    atomicAdd(&hist[kRings + key], q1 - kFixBias);
                    atomicAdd(&hist[2 * kRings + key], q2 - kFixBias);
                };
                int q0, q1, q2;
                if (fast && run == kRun && col + kRun <= ix.w) {
                    // a whole run within one row of an image with sides up to
                    // 2048 (d2 < 2^23): all its loads in flight, d2 stepped
                    float v[kRun];
#pragma unroll
                    for (int i = 0; i < kRun; ++i) v[i] = img_pix<DT>(a, at + i, sc);
                    const int di = row - pr, dj = col - pc;
                    const int d0 = di * di + dj * dj;
#pragma unroll
                    for (int i = 0; i < kRun; ++i) {
                        const int key = ring_of(d0 + i * (2 * dj + i));
                        fix_split3(ff, v[i], q0, q1, q2);
                        if (key < kRings) add(key, q0, q1, q2);
                    }
                    continue;
                }
#pragma unroll 1
                for (int i = 0; i < run; ++i) {
                    int key;
                    if (narrow) {   // both sides <= 32768: d2 < 2^31
                        const int di = row - pr, dj = col - pc;
                        key = static_cast<int>(ring_ceil32(static_cast<unsigned>(di * di + dj * dj)));
                    } else {
                        const long long di = row - pr, dj = col - pc;
                        const long long d2 = di * di + dj * dj;
                        long long k = static_cast<long long>(sqrtf(static_cast<float>(d2)));
                        while (k * k < d2) ++k;                   // k = ceil(sqrt(d2)): k-1 < d <= k,
                        while (k > 0 && (k - 1) * (k - 1) >= d2) --k;   // exact in integers
                        key = k < kRings ? static_cast<int>(k) : kRings;
                    }
                    if (key < kRings) {
                        fix_split(ff, img_pix<DT>(a, at, sc), q0, q1, q2);
                        add(key, q0, q1, q2);
                    }
                    ++at;
                    if (++col == ix.w) {
                        col = 0;
                        ++row;
                    }
                }
            }
            cl.sync();   // every CTA's histogram is complete
            // each CTA sums an eighth of the pieces over the cluster into CTA
            // 0's histogram (in place: a word is read by its owner only)
            int* sum = cl.map_shared_rank(hist, 0);
            for (int k = rank * (3 * kRings / kCutCluster) + tid; k < (rank + 1) * (3 * kRings / kCutCluster);
                 k += kCutThreads) {
                int s = 0;
#pragma unroll
                for (int r = 0; r < kCutCluster; ++r) s += cl.map_shared_rank(hist, r)[k];
                sum[k] = s;
            }
            cl.sync();   // CTA 0 has the cluster's rings
            if (rank == 0) {
                // crossing ring: thread t owns rings [t * ch, t * ch + ch)
                constexpr int ch = kRings / kCutThreads;
                long long ring[ch], own = 0;
#pragma unroll
                for (int i = 0; i < ch; ++i) {
                    const int k = tid * ch + i;
                    ring[i] = fix_join(ff, hist[k], hist[kRings + k], hist[2 * kRings + k]);
                    own += ring[i];
                }
                long long incl = own;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const long long o2 = __shfl_up_sync(kFull, incl, off);
                    if (lane >= off) incl += o2;
                }
                if (lane == 31) s_tot[warp] = incl;
                if (tid == 0) s_first = kRings;
                __syncthreads();
                long long run = incl - own;
                for (int k = 0; k < warp; ++k) run += s_tot[k];
                Crossing x = {-1, 0, 0};
#pragma unroll
                for (int i = 0; i < ch; ++i) {
                    const long long nxt = run + ring[i];
                    if (x.k < 0 && 2 * nxt >= tot) x = {tid * ch + i, run, nxt};
                    run = nxt;
                }
                if (x.k >= 0) atomicMin(&s_first, x.k);
                __syncthreads();
                if (x.k >= 0 && x.k == s_first) s_x = x;
                __syncthreads();
            }
        }
        if (rank == 0 && tid == 0)
            write_square(a, img, ix, !size_ok ? FSE_ST_BAD_SIZE : (!fin ? FSE_ST_NONFINITE : 0u), pr, pc, tot, s_x);
        // No cluster barrier here: what other CTAs read of this one (c_v, c_i and
        // c_amax before the second one, c_near, c_tot and hist after it) is
        // written again only past the next image's first or second.
        __syncthreads();   // s_x and s_all have been read
    }
    cl.sync();   // no CTA leaves while another reads its shared memory
}

// Exclusive prefix sum of h * w over the cut-outs, in one CTA of 1024
// threads, chunk by chunk with a running carry.
__global__ void __launch_bounds__(1024) cutout_scan_kernel(fse_stamp* out_idx, int64_t count, int64_t* total) {
    __shared__ long long warp_sum[32];
    __shared__ long long carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < count; base += 1024) {
        const int64_t i = base + tid;
        const long long n = i < count ? static_cast<long long>(out_idx[i].h) * out_idx[i].w : 0;
        long long incl = n;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const long long o = __shfl_up_sync(kFull, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            long long ws = warp_sum[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const long long o = __shfl_up_sync(kFull, ws, off);
                if (lane >= off) ws += o;
            }
            warp_sum[lane] = ws;                      // inclusive over warps
        }
        __syncthreads();
        const long long before = carry + (warp ? warp_sum[warp - 1] : 0) + incl - n;
        if (i < count) out_idx[i].offset = before;
        __syncthreads();
        if (tid == 1023) carry = before + n;
        __syncthreads();
    }
    if (tid == 0) *total = carry;
}

// One CTA per cut-out: its warps take rows in turn, lanes along the row.  A
// cut-out that does not fit in the output gets FSE_ST_NO_ROOM and is not
// copied.
template <typename T>
__global__ void __launch_bounds__(256) cutout_copy_kernel(CutoutArgs a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const T* src = static_cast<const T*>(a.images);
    T* dst = static_cast<T*>(a.out_pix);
    for (int64_t i = blockIdx.x; i < a.count; i += gridDim.x) {
        const fse_cutout_info info = a.info[i];
        const fse_stamp o = a.out_idx[i];
        const long long n = static_cast<long long>(o.h) * o.w;
        if (n == 0) continue;
        if (o.offset + n > a.out_capacity) {
            if (threadIdx.x == 0) a.info[i].status = info.status | FSE_ST_NO_ROOM;
            continue;
        }
        const fse_stamp im = a.img_idx[i];
        // a row is at most four lane loads wide (sides of 128 at most); two rows'
        // loads are in flight before the stores
        const T* s = src + im.offset + static_cast<int64_t>(info.row0) * im.w + info.col0;
        T* d = dst + o.offset;
        for (int r = warp; r < o.h; r += 2 * nwarp) {
            T v[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (r + q * nwarp < o.h && lane + 32 * u < o.w)
                        v[q][u] = s[static_cast<int64_t>(r + q * nwarp) * im.w + lane + 32 * u];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (r + q * nwarp < o.h && lane + 32 * u < o.w)
                        d[static_cast<int64_t>(r + q * nwarp) * o.w + lane + 32 * u] = v[q][u];
        }
    }
}

}  // namespace

cudaError_t launch_cutout(const CutoutArgs& a, cudaStream_t stream) {
    if (a.count <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // a cluster of kCutCluster CTAs per image, handed out by the hardware as
    // clusters finish; beyond 64 per SM a cluster takes several images
    long long clusters = static_cast<long long>(sms) * 64;
    if (clusters > a.count) clusters = a.count;
    const long long grid = clusters * kCutCluster;
    if (a.dtype == FSE_BF16)
        cutout_measure_kernel<FSE_BF16><<<static_cast<unsigned>(grid), kCutThreads, 0, stream>>>(a);
    else
        cutout_measure_kernel<FSE_F32><<<static_cast<unsigned>(grid), kCutThreads, 0, stream>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cutout_scan_kernel<<<1, 1024, 0, stream>>>(a.out_idx, a.count, a.out_total);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    long long cgrid = a.count;
    const long long cap = static_cast<long long>(sms) * 8;
    if (cgrid > cap) cgrid = cap;
    if (a.out_pix) {
        if (a.dtype == FSE_BF16)
            cutout_copy_kernel<__nv_bfloat16><<<static_cast<unsigned>(cgrid), 256, 0, stream>>>(a);
        else
            cutout_copy_kernel<float><<<static_cast<unsigned>(cgrid), 256, 0, stream>>>(a);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace fse
