// fse_adjoint.cu -- chi^2 of the elliptical Sérsic model (Eqs. 10, 11) at
// given parameters and its adjoint (the vector-Jacobian product with the
// parameters and the pixels), for fse_sersic_chi2_grad.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "fse_device.cuh"
#include "fse_internal.h"

namespace fse {
namespace {

// ------------------------------------------------------------------ adjoint
// chi^2 (Eq. 11) of the elliptical Sérsic model (Eq. 10) at caller-given
// parameters p = (x0, y0, e1, e2, I0, r_e, n), and the vector-Jacobian product
// of the upstream gradient gout[s] with d chi^2 / dp and d chi^2 / dI (pixels).
// With residual r = m - I and weights w:
//   d chi^2/dp = 2 sum w r dm/dp,   d chi^2/dI_i = -2 w_i r_i,
// m = I0 E, E = exp(-b u), u = (r_s / r_e)^(1/n).  The centre and the
// ellipticity act through the Sérsic radius r_s = R(g) / (1 - |g|) (Eq. A1).
// In the principal frame of the ellipse (t_par along the major axis at angle
// phi, 2 phi = arg g; t_perp across it) the radius is
//   r_s^2 = t_par^2 + k^2 t_perp^2,   k = (1 + |g|) / (1 - |g|),
// and with g = |g| (cos 2phi, sin 2phi)
//   d r_s^2/dg1 = cos2phi K1 t_perp^2 + sin2phi K2 t_par t_perp,
//   d r_s^2/dg2 = sin2phi K1 t_perp^2 - cos2phi K2 t_par t_perp,
//   K1 = 4 (1 + |g|) / (1 - |g|)^3,   K2 = 4 / (1 - |g|)^2,
//   d r_s^2/dx0 = -2 (cos phi t_par - sin phi k^2 t_perp),
//   d r_s^2/dy0 = -2 (sin phi t_par + cos phi k^2 t_perp).
// This form has no cancellation: written through R^2 and 1 - |g| separately,
// the two parts of dr_s/dg cancel exactly along the major axis.  At g = 0 the
// derivative of |g| is taken as 0 (the kink), which leaves
// d r_s^2/dg = (2 (t2^2 - t1^2), -4 t1 t2).  dm/d(r_s^2) = -m b u / (2 n r_s^2).
// One warp per stamp; each pixel is used once, so it is read straight from
// global memory (the lanes take consecutive pixels: coalesced).
// A stamp whose rows are multiples of four pixels and which starts on a
// multiple of four elements gives each lane four consecutive pixels of a row,
// which share the row's terms and one load and store, without bounds checks:
// about half the instructions per pixel of the lane-strided form.  The
// arithmetic of a pixel is the same in both; chi^2 is summed in the strided
// form's order in both (a warp's squared residuals pass through shared memory),
// so its bits depend neither on the form nor on the outputs asked for.  The
// parameter gradient's seven sums follow the form: for a stamp whose width is a
// multiple of four they round differently (about 1e-7 of the sums) where it
// starts on a multiple of four elements and where it does not.  One order for
// both was measured and left: with a third loop, or the accesses chosen in the
// four-pixel one, the aligned pixel gradients of 30,000 stamps of 64x64 took 321 to
// 325 us instead of 302, those of 47x45 up to 209 instead of 188.
//   65,536 stamps of 64x64: chi^2 alone (1.07 GB, 0.16 ms at the copy rate)
//   0.33 to 0.25 ms; parameter gradient 0.53 to 0.45; with the pixel gradient
//   (2.15 GB, 0.32 ms) and the caller's zero fill 0.71 to 0.63.

// Four consecutive pixels of a stamp (p a multiple of four, 16- or 8-byte
// aligned), decoded.
template <int DT>
__device__ __forceinline__ void load4(const void* pix, int64_t off, float sc, float (&v)[4]) {
    if (DT == FSE_BF16) {
        const uint2 r = __ldcs(reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(pix) + off));
        v[0] = __uint_as_float(r.x << 16) * sc;
        v[1] = __uint_as_float(r.x & 0xffff0000u) * sc;
        v[2] = __uint_as_float(r.y << 16) * sc;
        v[3] = __uint_as_float(r.y & 0xffff0000u) * sc;
    } else {
        const float4 r = __ldcs(reinterpret_cast<const float4*>(static_cast<const float*>(pix) + off));
        v[0] = r.x;
        v[1] = r.y;
        v[2] = r.z;
        v[3] = r.w;
    }
}

template <int DT, bool IVAR, bool GRAD, bool DPIX>
__global__ void __launch_bounds__(256, GRAD ? 3 : (IVAR ? 5 : 6)) chi2_grad_kernel(GradArgs a) {
    __shared__ __align__(16) float s_sq[8][256];   // a block's weighted squared residuals, per warp
    float* sq = s_sq[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const float n_lo = static_cast<float>(kBnLo + 2 * kBnStep);
    const float n_hi = static_cast<float>(kBnLo + (kBnNodes - 3) * kBnStep);
    for (;;) {
        unsigned sidx = 0;
        if (lane == 0) sidx = atomicAdd(a.queue, 1u);
        sidx = __shfl_sync(kFull, sidx, 0);
        if (sidx >= static_cast<unsigned long long>(a.count)) break;
        const int64_t si = static_cast<int64_t>(sidx);
        const fse_stamp ix = a.idx[si];
        const long long npl = static_cast<long long>(ix.h) * ix.w;
        const bool size_ok = ix.h >= 1 && ix.w >= 1 && npl <= FSE_MAX_PIX;
        float p[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) p[i] = a.params[si * 7 + i];
        const float x0 = p[0], y0 = p[1], g1 = p[2], g2 = p[3], I0 = p[4], re = p[5], n = p[6];
        const float gabs = sqrtf(g1 * g1 + g2 * g2);
        bool ok = size_ok && re > 0.f && n >= n_lo && n <= n_hi && gabs < 1.f && isfinite(I0) &&
                  isfinite(x0) && isfinite(y0) && isfinite(re);
        const int npix = size_ok ? static_cast<int>(npl) : 0;
        const float gof = a.gout ? static_cast<float>(a.gout[si]) : 1.f;
        if (!ok) {
            // parameters outside the model's domain: NaN results, NaN pixel gradient
            if (lane == 0) {
                if (a.chi2) a.chi2[si] = NAN;
                if (GRAD && a.dparams)
#pragma unroll
                    for (int i = 0; i < 7; ++i) a.dparams[si * 7 + i] = NAN;
            }
            if (DPIX)
                for (int q = lane; q < npix; q += 32) a.dpix[ix.offset + q] = NAN;
            continue;
        }
        float b, db;
        bn_lookup_f(a.bnf, n, &b, &db);
        const float inv_n = 1.f / n;
        // principal frame: cos 2phi, sin 2phi, then cos phi, sin phi
        const float c2 = gabs > 0.f ? g1 / gabs : 1.f, s2 = gabs > 0.f ? g2 / gabs : 0.f;
        const float cph = sqrtf(fmaxf(0.5f * (1.f + c2), 0.f));
        const float sph = copysignf(sqrtf(fmaxf(0.5f * (1.f - c2), 0.f)), s2);
        const float kap = (1.f + gabs) / (1.f - gabs), kap2 = kap * kap;
        const float zg = gabs > 0.f ? 0.f : 1.f;            // the g = 0 convention
        const float c0 = log2f(re);                          // log2(r_s / r_e) = 0.5 log2 r_s^2 - c0
        const float nbl = -b * kLog2e;
        const float kn = b * static_cast<float>(kLn2) * inv_n * inv_n;   // dm/dn = m u (kn a - b')
        const float sc = (DT == FSE_BF16 && a.scale) ? a.scale[si] : 1.f;
        const float* pf = static_cast<const float*>(a.pix) + ix.offset;
        const __nv_bfloat16* pb = static_cast<const __nv_bfloat16*>(a.pix) + ix.offset;
        const float* iv = IVAR ? a.inv_var + ix.offset : nullptr;
        float* dp = DPIX ? a.dpix + ix.offset : nullptr;
        float ch[1] = {0.f}, cl[1] = {0.f};
        // S: sum c E, sum c m u, sum c m u (kn a - b'), and with q = c m u / r_s^2:
        // sum q t_par, sum q k^2 t_perp, sum q (t_perp^2 - zg t_par^2),
        // sum q t_par t_perp   (c = 2 w r, a = log2(r_s / r_e)).  The n term is
        // combined per pixel before it is summed, so its parts do not cancel.
        float S[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) S[i] = 0.f;
        // (with weights and pixel gradients both, the two forms in one kernel need
        // more registers than three CTAs per SM leave: strided only)
        bool vec = false;
        if constexpr (!(IVAR && DPIX)) vec = a.aligned && (ix.w & 3) == 0 && (ix.offset & 3) == 0;
        if (vec) {
            FWalk pw(4 * lane, ix.w, 128);
            for (int b0 = 0; b0 < npix; b0 += 256) {
                float fv[2][4], wv[2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = b0 + 128 * h + 4 * lane;
                    if (q < npix) {
                        load4<DT>(a.pix, ix.offset + q, sc, fv[h]);
                        if (IVAR) load4<FSE_F32>(a.inv_var, ix.offset + q, 1.f, wv[h]);
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = b0 + 128 * h + 4 * lane;
                    float g[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
                    if (q < npix) {
                        const float t2 = pw.r - y0;
                        const float pa0 = t2 * sph;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float t1 = (pw.c + static_cast<float>(j)) - x0;
                            const float tpa = fmaf(t1, cph, pa0);
                            const float tpe = fmaf(t2, cph, -t1 * sph);
                            const float kte = kap2 * tpe;
                            const float r2 = fmaf(kte, tpe, tpa * tpa);
                            // at r = 0 the log2 is -inf and u its limit 0
                            const float av = fmaf(0.5f, __log2f(r2), -c0);
                            const float u = ex2(av * inv_n);
                            const float E = ex2(u * nbl);
                            const float res = fmaf(I0, E, -fv[h][j]);
                            const float wr = IVAR ? wv[h][j] * res : res;
                            s2[j] = __fmul_rn(wr, res);
                            if (GRAD) {
                                const float c = 2.f * wr;
                                g[j] = __fmul_rn(-c, gof);
                                const float cmu = c * (I0 * E) * u;
                                S[0] = fmaf(c, E, S[0]);
                                S[1] += cmu;
                                S[2] = fmaf(cmu, r2 > 0.f ? fmaf(kn, av, -db) : 0.f, S[2]);
                                const float qv = r2 > 0.f ? __fdividef(cmu, r2) : 0.f;
                                S[3] = fmaf(qv, tpa, S[3]);
                                S[4] = fmaf(qv, kte, S[4]);
                                S[5] = fmaf(qv, fmaf(-zg * tpa, tpa, tpe * tpe), S[5]);
                                S[6] = fmaf(qv, tpa * tpe, S[6]);
                            }
                        }
                        if (DPIX) __stcs(reinterpret_cast<float4*>(dp + q), make_float4(g[0], g[1], g[2], g[3]));
                    }
                    pw.next();
                    if (!GRAD || a.chi2)
                        *reinterpret_cast<float4*>(sq + 128 * h + 4 * lane) = make_float4(s2[0], s2[1], s2[2], s2[3]);
                }
                if (!GRAD || a.chi2) {
                    // the block's sum in the strided form's order
                    __syncwarp();
                    float cp = 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) cp += sq[lane + 32 * j];
                    df_add(ch[0], cl[0], cp);
                    __syncwarp();
                }
            }
        } else {
            // Each lane loads KB pixels (and weights) ahead of using them: the
            // kernel reads every byte once, so how many loads are in flight
            // matters.  Per lane the pixels are taken in the order lane, lane + 32,
            // ...; blocks of 256 pixels inside the stamp need no bounds checks.
            constexpr int KB = 8;
            FWalk pw(lane, ix.w);
            auto block = [&](int q0, auto whole) {
                constexpr bool kFullBlock = decltype(whole)::value;
                float fv[KB], wv[KB];
#pragma unroll
                for (int j = 0; j < KB; ++j) {
                    const int q = q0 + 32 * j;
                    const bool in = kFullBlock || q < npix;
                    if (DT == FSE_BF16)
                        fv[j] = in ? __bfloat162float(pb[q]) * sc : 0.f;
                    else
                        fv[j] = in ? __ldcs(pf + q) : 0.f;
                    wv[j] = IVAR ? (in ? __ldcs(iv + q) : 0.f) : 1.f;
                }
                float cp = 0.f;   // this lane's chi^2 over the KB pixels, then one double-float add
#pragma unroll
                for (int j = 0; j < KB; ++j) {
                    const int q = q0 + 32 * j;
                    if (!kFullBlock && q >= npix) continue;
                    const float f = fv[j];
                    const float t1 = pw.c - x0;
                    const float t2 = pw.r - y0;
                    pw.next();
                    const float tpa = fmaf(t1, cph, t2 * sph);
                    const float tpe = fmaf(t2, cph, -t1 * sph);
                    const float kte = kap2 * tpe;
                    const float r2 = fmaf(kte, tpe, tpa * tpa);
                    float u = 0.f, av = 0.f;
                    if (r2 > 0.f) {
                        // MUFU log2: absolute error ~2^-22, the size of the rounding of
                        // log2 r_s^2 itself at these magnitudes
                        av = fmaf(0.5f, __log2f(r2), -c0);
                        u = ex2(av * inv_n);
                    }
                    const float E = ex2(u * nbl);
                    const float wgt = wv[j];
                    // one rounding for the residual, and an uncontracted square, in
                    // every instance of the kernel, so that chi^2 does not depend on
                    // which outputs were requested
                    const float res = fmaf(I0, E, -f);
                    const float wr = wgt * res;
                    cp += __fmul_rn(wr, res);
                    if (GRAD) {
                        const float c = 2.f * wr;
                        if (DPIX) __stcs(dp + q, __fmul_rn(-c, gof));
                        const float cmu = c * (I0 * E) * u;
                        S[0] = fmaf(c, E, S[0]);
                        S[1] += cmu;
                        S[2] = fmaf(cmu, fmaf(kn, av, -db), S[2]);
                        const float qv = r2 > 0.f ? __fdividef(cmu, r2) : 0.f;
                        S[3] = fmaf(qv, tpa, S[3]);
                        S[4] = fmaf(qv, kte, S[4]);
                        S[5] = fmaf(qv, fmaf(-zg * tpa, tpa, tpe * tpe), S[5]);
                        S[6] = fmaf(qv, tpa * tpe, S[6]);
                    }
                }
                df_add(ch[0], cl[0], cp);
            };
            int q0 = lane;
            for (; q0 - lane + 32 * KB <= npix; q0 += 32 * KB) block(q0, std::true_type{});
            if (q0 < npix) block(q0, std::false_type{});
        }
        warp_allsum_df(ch, cl);
        if (GRAD) warp_allsum(S);
        if (lane == 0) {
            if (a.chi2) a.chi2[si] = static_cast<double>(ch[0]) + static_cast<double>(cl[0]);
            if (GRAD && a.dparams) {
                const float kr = -0.5f * b * inv_n;       // c dm/d(r_s^2) = kr q
                const float om = 1.f / (1.f - gabs);
                const float K2 = 4.f * om * om, K1 = (1.f + gabs) * om * K2;
                // d chi^2/dp, then times the upstream gradient as the last rounding
                float d[7];
                d[0] = -2.f * kr * fmaf(cph, S[3], -sph * S[4]);
                d[1] = -2.f * kr * fmaf(sph, S[3], cph * S[4]);
                if (gabs > 0.f) {
                    d[2] = kr * fmaf(c2 * K1, S[5], s2 * K2 * S[6]);
                    d[3] = kr * fmaf(s2 * K1, S[5], -c2 * K2 * S[6]);
                } else {
                    d[2] = 2.f * kr * S[5];
                    d[3] = -4.f * kr * S[6];
                }
                d[4] = S[0];
                d[5] = b * inv_n / re * S[1];
                d[6] = S[2];
                float* o = a.dparams + si * 7;
#pragma unroll
                for (int i = 0; i < 7; ++i) o[i] = __fmul_rn(d[i], gof);
            }
        }
    }
}

template <int DT, bool IVAR, bool GRAD, bool DPIX>
cudaError_t launch_grad_t(const GradArgs& a, cudaStream_t stream) {
    auto kern = chi2_grad_kernel<DT, IVAR, GRAD, DPIX>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long grid = static_cast<long long>(per_sm) * sms;
    const long long need = (a.count + 7) / 8;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    kern<<<static_cast<unsigned>(grid), 256, 0, stream>>>(a);
    return cudaGetLastError();
}

template <int DT, bool IVAR>
cudaError_t launch_grad_dt(const GradArgs& a, cudaStream_t stream) {
    if (a.dpix) return launch_grad_t<DT, IVAR, true, true>(a, stream);
    if (a.dparams) return launch_grad_t<DT, IVAR, true, false>(a, stream);
    return launch_grad_t<DT, IVAR, false, false>(a, stream);
}

}  // namespace

cudaError_t launch_chi2_grad(const GradArgs& a_in, cudaStream_t stream) {
    GradArgs a = a_in;
    if (a.count <= 0) return cudaSuccess;
    if (!a.bnf) return cudaErrorInvalidValue;
    // the buffers' own alignment, for the four-pixel accesses
    auto at = [](const void* p, uintptr_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; };
    a.aligned = at(a.pix, a.dtype == FSE_BF16 ? 8 : 16) && at(a.inv_var, 16) && at(a.dpix, 16);
    const bool iv = a.inv_var != nullptr;
    if (a.dtype == FSE_BF16)
        return iv ? launch_grad_dt<FSE_BF16, true>(a, stream) : launch_grad_dt<FSE_BF16, false>(a, stream);
    return iv ? launch_grad_dt<FSE_F32, true>(a, stream) : launch_grad_dt<FSE_F32, false>(a, stream);
}

}  // namespace fse
