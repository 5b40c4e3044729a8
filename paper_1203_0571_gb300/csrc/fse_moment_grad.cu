// fse_moment_grad.cu -- implicit-function derivatives of the moment fixed
// point (Secs. 2-3) with respect to the pixels: VJP (fse_moment_vjp) and JVP
// (fse_moment_jvp).
//
// The moment iteration stops where its steps vanish.  With theta = (xc, yc,
// g1, g2, sigma_w), t = pixel - centre, R^2 of Eq. A1, W = exp(-R^2/2 s^2) and
// e_w = 2g/(1+g^2), that point solves F_k = sum_p I_p W m_k(t) = 0 with
//   m_1 = t1, m_2 = t2                         zero centroid step (Eqs. 3-6)
//   m_3 = (t1^2 - t2^2) - e_w1 (t1^2 + t2^2)   e^obs = e_w, where the step of
//   m_4 = 2 t1 t2 - e_w2 (t1^2 + t2^2)         Eq. 9 vanishes
//   m_5 = R^2 - s^2                            matched weight
// so d theta / d I_p = -J^-1 W(p) m(p) with J_kl = sum_p I_p d(W m_k)/d theta_l.
// Every m_k and every d R^2 / d theta_l is a polynomial of degree <= 2 in t,
// so J is a fixed combination of the 15 weighted moments
// M_ab = sum I W t1^a t2^b (a + b <= 4).  A warp per stamp accumulates them,
// assembles J with a lane per entry and solves the 5 x 5 system across its
// lanes (moment_grad_kernel); for the VJP a streaming kernel then writes dL/dI.
// sigma_w from the start-up growth curve (r50 / sqrt(2 ln 2), Sec. 4.1) is
// an explicit function of the pixels: it is piecewise constant in the three
// regions of the crossing ring (inside the disc k-1, in ring k, outside),
// found from double-float disc sums around the brightest pixel.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "fse_device.cuh"
#include "fse_internal.h"

namespace fse {
namespace {

constexpr float kInvSqrt2Ln2F = 0.849321800f;   // 1 / sqrt(2 ln 2)

// Index of the monomial t1^a t2^b among the 15 of degree <= 4, by degree and
// then by the power of t2.
__host__ __device__ constexpr int mono(int a, int b) { return (a + b) * (a + b + 1) / 2 + b; }
template <int DT>
__device__ __forceinline__ float load_pix(const MomentGradArgs& a, int64_t off, float sc) {
    return DT == FSE_BF16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(a.pix)[off]) * sc
                          : __ldg(static_cast<const float*>(a.pix) + off);
}

// The growth curve of the start-up (Sec. 4.1) around the brightest pixel, for
// d sigma_w / d I: the crossing ring k (the first whose enclosed sum reaches
// half the total) and the constants of d sigma_w / d I_p in the three regions
// d <= k-1, k-1 < d <= k and d > k; for the JVP the tangent's sums over the
// two discs.
struct R50Grad {
    int on;                  // sigma_w depends on the pixels
    int pr, pc, k;
    float c_in, c_ring, c_out;
    float u_in, u_disc;      // JVP: tangent summed over d <= k-1 and d <= k
};

// A warp's sums of one stamp, in shared memory: the 15 weighted moments as
// float pairs and the tangent's six weighted moments of degree <= 2 (JVP); and
// the coefficient tables of the solve: the polynomials m_k and, in du, those of
// d R^2 / d theta_l (l < 4) and R^2.
struct MomSums {
    float Mh[15], Ml[15], U[6];
    float m[5][6], du[5][6];
};

// Stamp geometry at theta.
struct Geom {
    float x0, y0, g1, g2, s;
    float A, B, G4, cw;      // R^2 = A t1^2 + B t2^2 - G4 t1 t2; W = 2^(cw R^2)
};

__device__ __forceinline__ Geom stamp_geom(const MomentGradArgs& a, const fse_result& mom) {
    const bool ellip = (a.mode & FSE_MOM_ELLIP) != 0;
    Geom q;
    q.x0 = mom.x0;
    q.y0 = mom.y0;
    q.g1 = ellip ? mom.e1 : 0.f;
    q.g2 = ellip ? mom.e2 : 0.f;
    q.s = mom.sigma_w;
    const float gg = q.g1 * q.g1 + q.g2 * q.g2;
    q.A = 1.f + gg - 2.f * q.g1;
    q.B = 1.f + gg + 2.f * q.g1;
    q.G4 = 4.f * q.g2;
    q.cw = -kLog2e / (2.f * q.s * q.s);
    return q;
}

// Double-float helpers: the exact product error by FMA, Knuth's two-sum.
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = a * b;
    e = fmaf(a, b, -p);
}

__device__ __forceinline__ void df_acc(float& hi, float& lo, float p, float e) {
    const float s = hi + p;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (p - bb);
    hi = s;
    lo += err + e;
}

// The polynomial factors of J (coefficients of 1, t1, t2, t1^2, t1 t2, t2^2)
// into the warp's tables; the entries set here are the only ones that are ever
// nonzero (the kernel clears the tables once).
__device__ __forceinline__ void jac_tables(const Geom& q, int lane, MomSums* t) {
    if (lane == 0) {
        const float g1 = q.g1, g2 = q.g2, gg = g1 * g1 + g2 * g2;
        const float ew1 = 2.f * g1 / (1.f + gg), ew2 = 2.f * g2 / (1.f + gg);
        t->m[0][1] = 1.f;
        t->m[1][2] = 1.f;
        t->m[2][3] = 1.f - ew1; t->m[2][5] = -(1.f + ew1);
        t->m[3][3] = -ew2; t->m[3][4] = 2.f; t->m[3][5] = -ew2;
        t->m[4][0] = -q.s * q.s; t->m[4][3] = q.A; t->m[4][4] = -q.G4; t->m[4][5] = q.B;
        t->du[0][1] = -2.f * q.A; t->du[0][2] = q.G4;
        t->du[1][1] = q.G4; t->du[1][2] = -2.f * q.B;
        t->du[2][3] = 2.f * (g1 - 1.f); t->du[2][5] = 2.f * (g1 + 1.f);
        t->du[3][3] = 2.f * g2; t->du[3][4] = -4.f; t->du[3][5] = 2.f * g2;
        t->du[4][3] = q.A; t->du[4][4] = -q.G4; t->du[4][5] = q.B;
    }
}

// J_kl = sum I W [a_l m_k + dm_k/dtheta_l] from the 15 moments: with V[i] =
// sum_j m_k[j] M_(i+j), J_kl = sum_i a_l[i] V[i] + sum_i dm_kl[i] M_i, where a_l
// is the derivative of log W (-du_l / 2 s^2, or R^2 / s^3 for sigma_w) and
// dm_k/dtheta_l follows from m_k: the centre moves t, so l = 0, 1 give -dm_k/dt1
// and -dm_k/dt2; g enters m_3, m_4 through e_w and m_5 through R^2; sigma_w
// enters m_5 alone.  The combination cancels by up to an order of magnitude
// (e.g. J_55 = sum I W [R^2 (R^2 - s^2) / s^3 - 2 s]), so each product and
// partial sum is carried in double-float.  One entry per lane.
__device__ __forceinline__ float jac_entry(const Geom& q, const MomSums* t, int k, int l) {
    const bool lin = l < 2;                 // a_l has the monomials t1, t2; else the squares
    float hi = 0.f, lo = 0.f;
    {
        const float* mk = t->m[k];
        float c0 = 0.f, c1 = 0.f, c2 = 0.f; // dm_kl at 1, t1, t2 or at the squares
        if (lin) {
            c0 = -mk[1 + l];
            c1 = l == 0 ? -2.f * mk[3] : -mk[4];
            c2 = l == 0 ? -mk[4] : -2.f * mk[5];
        } else if (k == 4) {
            c0 = l < 4 ? t->du[l][3] : -2.f * q.s;
            c1 = l < 4 ? t->du[l][4] : 0.f;
            c2 = l < 4 ? t->du[l][5] : 0.f;
        } else if (k >= 2 && l < 4) {
            const float gg = q.g1 * q.g1 + q.g2 * q.g2, qq = (1.f + gg) * (1.f + gg);
            const float d = q.g1 * q.g1 - q.g2 * q.g2;
            const float de = k != l ? -4.f * q.g1 * q.g2 : 2.f * (k == 2 ? 1.f - d : 1.f + d);
            c0 = c2 = -(de / qq);
        }
        const int b = l >= 2 && l < 4 ? 3 : 0;
        const float c[3] = {c0, c1, c2};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float p, e;
            two_prod(c[i], t->Mh[b + i], p, e);
            df_acc(hi, lo, p, fmaf(c[i], t->Ml[b + i], e));
        }
    }
    const float fac = l < 4 ? -(1.f / (2.f * q.s * q.s)) : 1.f / (q.s * q.s * q.s);
    const int n0 = lin ? 1 : 2;             // degree of a_l's monomials
    const int tri[3] = {n0 * (n0 + 1) / 2, (n0 + 1) * (n0 + 2) / 2, (n0 + 2) * (n0 + 3) / 2};
#pragma unroll
    for (int i = 0; i < 3; ++i) {           // t1, t2 or t1^2, t1 t2, t2^2: power i of t2
        const float a = lin && i == 2 ? 0.f : fac * t->du[l][(lin ? 1 : 3) + (lin && i == 2 ? 0 : i)];
        float vh = 0.f, vl = 0.f, p, e;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            // degree and power of t2 of the j-th monomial
            const int dj = j == 0 ? 0 : j < 3 ? 1 : 2, bj = j == 2 || j == 4 ? 1 : j == 5 ? 2 : 0;
            const int b = lin && i == 2 ? 0 : tri[dj] + bj + i;
            const float c = t->m[k][j];
            two_prod(c, t->Mh[b], p, e);
            df_acc(vh, vl, p, fmaf(c, t->Ml[b], e));
        }
        two_prod(a, vh, p, e);
        df_acc(hi, lo, p, fmaf(a, vl, e));
    }
    return hi + lo;
}

// Solve a 5 x 5 system held by 30 lanes, entry (r, c) in lane 6 r + c and the
// right-hand side in column 5, by Gaussian elimination with partial pivoting
// (rows are marked, not swapped).  Every lane gets the solution.  Returns
// false if a pivot is below 1e-6 of `big`.
__device__ __forceinline__ bool solve5(float X, float big, int lane, float (&x)[5]) {
    const int r = lane / 6, c = lane - 6 * r;
    unsigned done = 0;       // rows that have been pivots
    int prow[5];             // pivot row of each column
    if (!(big > 0.f)) return false;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        float pv = -1.f, val = 0.f;
        int piv = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const float v = __shfl_sync(kFull, X, 6 * i + s);
            if (!(done >> i & 1) && fabsf(v) > pv) {
                pv = fabsf(v);
                val = v;
                piv = i;
            }
        }
        if (!(pv > 1e-6f * big)) return false;
        const float inv = 1.f / val;
        const float mine = __shfl_sync(kFull, X, 6 * (r < 5 ? r : 0) + s);
        const float row = __shfl_sync(kFull, X, 6 * piv + c);
        done |= 1u << piv;
        prow[s] = piv;
        if (!(done >> r & 1)) X = fmaf(-(mine * inv), row, X);
    }
#pragma unroll
    for (int s = 4; s >= 0; --s) {
        float acc = __shfl_sync(kFull, X, 6 * prow[s] + 5);
#pragma unroll
        for (int j = s + 1; j < 5; ++j) acc = fmaf(-__shfl_sync(kFull, X, 6 * prow[s] + j), x[j], acc);
        x[s] = acc / __shfl_sync(kFull, X, 6 * prow[s] + s);
    }
    return true;
}

// The growth curve of the start-up (Sec. 4.1) around the brightest pixel:
// the crossing ring k (the first whose enclosed sum reaches half the total)
// and the constants of d sigma_w / d I_p in the three regions d <= k-1,
// k-1 < d <= k and d > k.  The disc sums are double-float, so k is the
// start-up's own except where an enclosed sum lies within ~1e-13 of half the
// total.  For the JVP the tangent's sums over the two discs come with them.

// Only the square that holds the disc is read (from L1 or L2: the stamp was
// read just before).
template <int DT, bool JVP>
__device__ R50Grad r50_ring(const MomentGradArgs& a, const fse_stamp& ix, float sc, float r50_hint, int peak,
                            float tot_h, float tot_l, int lane) {
    R50Grad o;
    o.on = 0;
    o.pr = peak / ix.w;
    o.pc = peak - o.pr * ix.w;
    o.k = 0;
    o.c_in = o.c_ring = o.c_out = o.u_in = o.u_disc = 0.f;
    const float tot = tot_h + tot_l;
    if (!(tot > 0.f)) return o;                  // fallback radius: no dependence
    int k = ring_guess(r50_hint, ix.h, ix.w);   // candidate from the start-up radius
#pragma unroll 1
    for (int tries = 0; tries < 8; ++tries) {
        float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
        const float km2 = static_cast<float>((k - 1) * (k - 1)), k2 = static_cast<float>(k * k);
        Box bx;
        bx.r0 = max(0, o.pr - k);
        bx.c0 = max(0, o.pc - k);
        bx.bh = min(ix.h - 1, o.pr + k) - bx.r0 + 1;
        bx.bw = min(ix.w - 1, o.pc + k) - bx.c0 + 1;
        const int plast = bx.last(ix.w);
        BoxWalk bk(lane, bx, ix.w, 32, o.pc, o.pr);
#pragma unroll 1
        while (__any_sync(kFull, bk.p <= plast)) {
            // four loads in flight per lane
            float v[4], uu[4], d2[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = bk.p <= plast;
                v[u] = in ? load_pix<DT>(a, ix.offset + bk.p, sc) : 0.f;
                if (JVP) uu[u] = in ? __ldg(a.tangent + ix.offset + bk.p) : 0.f;
                d2[u] = fmaf(bk.v, bk.v, bk.u * bk.u);       // an exact integer
                bk.next();
            }
            float ph[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in0 = k >= 1 && d2[u] <= km2, in1 = d2[u] <= k2;   // zero-filled past the end
                ph[0] += in0 ? v[u] : 0.f;
                ph[1] += in1 ? v[u] : 0.f;
                if (JVP) {
                    ph[2] += in0 ? uu[u] : 0.f;
                    ph[3] += in1 ? uu[u] : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < (JVP ? 4 : 2); ++i) df_add(h[i], l[i], ph[i]);
        }
        if constexpr (JVP) {
            warp_allsum_df(h, l);
        } else {
            float h2[2] = {h[0], h[1]}, l2[2] = {l[0], l[1]};
            warp_allsum_df(h2, l2);
            h[0] = h2[0]; h[1] = h2[1]; l[0] = l2[0]; l[1] = l2[1];
        }
        // 2 E - tot in double-float: the sign decides the crossing
        const float d1 = (2.f * h[1] - tot_h) + (2.f * l[1] - tot_l);
        const float d0 = (2.f * h[0] - tot_h) + (2.f * l[0] - tot_l);
        if (d1 < 0.f) {
            ++k;
        } else if (k >= 1 && d0 >= 0.f) {
            --k;
        } else {
            o.k = k;
            o.on = 1;
            o.u_in = h[2] + l[2];
            o.u_disc = h[3] + l[3];
            if (k == 0) {
                // r50 = H / (2 S) with S the brightest pixel
                const float Sf = h[1] + l[1], H = 0.5f * tot;
                o.c_ring = 0.5f * (0.5f * Sf - H) / (Sf * Sf) * kInvSqrt2Ln2F;
                o.c_out = 0.25f / Sf * kInvSqrt2Ln2F;
            } else {
                // r50 = (k-1) + (H - P) / (S - P); the differences from the pair sums
                const float D = (h[1] - h[0]) + (l[1] - l[0]);
                const float HP = 0.5f * ((tot_h - 2.f * h[0]) + (tot_l - 2.f * l[0]));
                o.c_out = 0.5f / D * kInvSqrt2Ln2F;
                o.c_ring = (0.5f * D - HP) / (D * D) * kInvSqrt2Ln2F;
                o.c_in = -0.5f / D * kInvSqrt2Ln2F;
            }
            return o;
        }
    }
    return o;
}

// The moment terms of one pixel at t = (t1, t2): f = I W times the 15
// monomials of degree <= 4 into P; for the JVP, the tangent u W times the
// six of degree <= 2 into PU.
template <bool JVP>
__device__ __forceinline__ void moment_terms(const Geom& q, float t1, float t2, float v, float uu, float (&P)[15],
                                             float (&PU)[6]) {
    const float R2 = fmaf(q.A, t1 * t1, fmaf(q.B, t2 * t2, -q.G4 * (t1 * t2)));
    const float W = ex2(R2 * q.cw);
    const float f = v * W;
    const float f1 = f * t1, f2 = f * t2;
    const float f11 = f1 * t1, f12 = f1 * t2, f22 = f2 * t2;
    const float f111 = f11 * t1, f112 = f11 * t2, f122 = f12 * t2, f222 = f22 * t2;
    P[mono(0, 0)] += f;
    P[mono(1, 0)] += f1;
    P[mono(0, 1)] += f2;
    P[mono(2, 0)] += f11;
    P[mono(1, 1)] += f12;
    P[mono(0, 2)] += f22;
    P[mono(3, 0)] += f111;
    P[mono(2, 1)] += f112;
    P[mono(1, 2)] += f122;
    P[mono(0, 3)] += f222;
    P[mono(4, 0)] = fmaf(f111, t1, P[mono(4, 0)]);
    P[mono(3, 1)] = fmaf(f111, t2, P[mono(3, 1)]);
    P[mono(2, 2)] = fmaf(f112, t2, P[mono(2, 2)]);
    P[mono(1, 3)] = fmaf(f122, t2, P[mono(1, 3)]);
    P[mono(0, 4)] = fmaf(f222, t2, P[mono(0, 4)]);
    if (JVP) {
        const float h = uu * W;
        const float h1 = h * t1, h2 = h * t2;
        PU[0] += h;
        PU[1] += h1;
        PU[2] += h2;
        PU[3] = fmaf(h1, t1, PU[3]);
        PU[4] = fmaf(h1, t2, PU[4]);
        PU[5] = fmaf(h2, t2, PU[5]);
    }
}

// The weighted sums of one stamp, by one warp, in one pass over its pixels
// (eight loads in flight per lane): finiteness; with sigma_w from the growth
// curve the brightest pixel and the total; the 15 weighted moments; and for the
// JVP the tangent's total and its six: eight pixels per lane in fp32, then
// double-float.  The VJP leaves out blocks of 256 pixels whose rows do not meet the
// weight's box (W >= 2^-40, weight_box; they add less than 2^-40 |I| |t|^4 to a sum,
// the iteration's own cut).  The JVP takes every block: a tangent may be all where
// the weight is small, as the VJP writes every pixel; and 20,000 stamps of 48x48
// take 217 us, with the tangent alone summed outside the box 247, with both cut to
// it 225 (64x64 316, 337, 295).  Then the growth curve's crossing ring (r50_ring).
// The totals go to rec from the lanes that hold them after the exchange.  (A
// second pass over the box's pixels alone has a third fewer weights to evaluate,
// but its walk and its wait for the loads cost more.)
template <int DT, bool JVP>
__device__ __forceinline__ void stamp_grad(const MomentGradArgs& a, int64_t si, int lane, MomSums* rec) {
    const fse_stamp ix = a.idx[si];
    const fse_result mom = a.moments[si];
    const long long npl = static_cast<long long>(ix.h) * ix.w;
    uint32_t status = 0;
    R50Grad rg;
    rg.on = 0;
    rg.pr = rg.pc = rg.k = 0;
    rg.c_in = rg.c_ring = rg.c_out = rg.u_in = rg.u_disc = 0.f;
    float dsw = 0.f;
    const Geom q = stamp_geom(a, mom);
    const bool ellip = (a.mode & FSE_MOM_ELLIP) != 0;
    const bool sig_held = (a.mode & FSE_MOM_SIGW_FIXED) || (mom.status & FSE_ST_SIGW_CLAMPED);
    const bool sig_r50 = !sig_held && (a.mode & FSE_MOM_SIGW_R50);
    if (ix.h < 1 || ix.w < 1 || npl > FSE_MAX_PIX) {
        status = FSE_ST_BAD_SIZE;
    } else {
        const int npix = static_cast<int>(npl);
        if (!(mom.status & FSE_ST_MOM_CONVERGED)) status |= FSE_ST_MOM_FAILED;
        if (!(q.s > 0.f) || !isfinite(q.cw)) status |= FSE_ST_MOM_FAILED;
        const float sc = (DT == FSE_BF16 && a.scale) ? a.scale[si] : 1.f;
        if (status == 0) {
            float vmax = -INFINITY, zero = 0.f;
            int imax = 0x7fffffff;
            float th[2] = {0.f, 0.f}, tl[2] = {0.f, 0.f};   // totals of the pixels and of the tangent
            float Mh[15], Ml[15], Uh[6], Ul[6];
#pragma unroll
            for (int i = 0; i < 15; ++i) Mh[i] = Ml[i] = 0.f;
#pragma unroll
            for (int i = 0; i < 6; ++i) Uh[i] = Ul[i] = 0.f;
            // the pixels of the box's rows
            const Box bx = weight_box(q.x0, q.y0, q.g1, q.g2, q.s, ix.h, ix.w);
            const int box0 = bx.r0 * ix.w, box1 = (bx.r0 + bx.bh) * ix.w;
            FWalk pw(lane, ix.w);
#pragma unroll 1
            for (int b0 = 0; b0 < npix; b0 += 256) {
                float v[8], uu[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int p = b0 + 32 * u + lane;
                    v[u] = p < npix ? load_pix<DT>(a, ix.offset + p, sc) : 0.f;
                    if (JVP) uu[u] = p < npix ? __ldg(a.tangent + ix.offset + p) : 0.f;
                }
                float pt = 0.f, pu = 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    zero = fmaf(v[u], 0.f, zero);   // NaN from a NaN or infinite pixel
                    pt += v[u];
                    if (JVP) pu += uu[u];
                }
                if (sig_r50) {
                    // the lane's maximum of the eight, and its index where it leads
                    float m8 = v[0];
                    if (b0 + 256 <= npix) {
#pragma unroll
                        for (int u = 1; u < 8; ++u) m8 = fmaxf(m8, v[u]);
                    } else {
                        m8 = -INFINITY;
#pragma unroll
                        for (int u = 0; u < 8; ++u) m8 = b0 + 32 * u + lane < npix ? fmaxf(m8, v[u]) : m8;
                    }
                    if (m8 > vmax) {
                        vmax = m8;
#pragma unroll
                        for (int u = 7; u >= 0; --u)
                            if (v[u] == m8 && b0 + 32 * u + lane < npix) imax = b0 + 32 * u + lane;
                    }
                    df_add(th[0], tl[0], pt);
                }
                if (JVP) df_add(th[1], tl[1], pu);
                if (!JVP && (b0 + 256 <= box0 || b0 >= box1)) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) pw.next();
                    continue;
                }
                float P[15], PU[6];
#pragma unroll
                for (int i = 0; i < 15; ++i) P[i] = 0.f;
#pragma unroll
                for (int i = 0; i < 6; ++i) PU[i] = 0.f;
                // (pixels past the end are zero and add nothing)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    moment_terms<JVP>(q, pw.c - q.x0, pw.r - q.y0, v[u], JVP ? uu[u] : 0.f, P, PU);
                    pw.next();
                }
#pragma unroll
                for (int i = 0; i < 15; ++i) df_add(Mh[i], Ml[i], P[i]);
                if (JVP) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) df_add(Uh[i], Ul[i], PU[i]);
                }
            }
            scatter_sum_df<15, 16>(Mh, Ml, lane);
            const int j = scatter_index<15>(lane);
            if (j < 15) {
                rec->Mh[j] = Mh[0];
                rec->Ml[j] = Ml[0];
            }
            if (JVP) {
                scatter_sum_df<6, 16>(Uh, Ul, lane);
                const int i = scatter_index<6>(lane);
                if (i < 6) rec->U[i] = Uh[0] + Ul[0];
            }
            if (sig_r50) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    const float ov = __shfl_xor_sync(kFull, vmax, off);
                    const int oi = __shfl_xor_sync(kFull, imax, off);
                    if (ov > vmax || (ov == vmax && oi < imax)) { vmax = ov; imax = oi; }
                }
            }
            if (JVP || sig_r50) warp_allsum_df(th, tl);
            float chk = zero;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) chk += __shfl_xor_sync(kFull, chk, off);
            if (JVP) chk += th[1] + (sig_r50 ? th[0] : 0.f);
            if (!isfinite(chk)) status |= FSE_ST_NONFINITE;
            if (status == 0 && sig_r50 && isfinite(th[0])) {
                rg = r50_ring<DT, JVP>(a, ix, sc, mom.r50, imax, th[0], tl[0], lane);
                if (JVP && rg.on)
                    dsw = rg.c_out * (th[1] + tl[1]) + (rg.c_ring - rg.c_out) * rg.u_disc +
                          (rg.c_in - rg.c_ring) * rg.u_in;
            }
        }
    }
    // J, a lane per entry, and the solve
    float xs[5] = {0.f, 0.f, 0.f, 0.f, 0.f}, Jcol4[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    if (status == 0) {
        jac_tables(q, lane, rec);
        __syncwarp();   // the sums and the tables are in place
        if (!isfinite(rec->Mh[0] + rec->Ml[0] + (JVP ? rec->U[0] : 0.f))) status |= FSE_ST_NONFINITE;
    }
    if (status == 0) {
        // lane 6 r + c: entry (r, c) of J (JVP) or of its transpose (VJP), the
        // right-hand side in column 5
        const int r = lane < 30 ? lane / 6 : 0, c = lane < 30 ? lane - 6 * (lane / 6) : 0;
        const int k = JVP || c == 5 ? r : c, l = c == 5 ? 4 : (JVP ? c : r);
        float X = jac_entry(q, rec, k, l);      // column 5: J_r4, for the coupling to sigma_w
        // lane of J_i4: (i, 4), or (4, i) in the transpose
#pragma unroll
        for (int i = 0; i < 5; ++i) Jcol4[i] = __shfl_sync(kFull, X, JVP ? 6 * i + 4 : 24 + i);
        // held parameters: rows and columns of a diagonal entry as large as the
        // active block's largest, with a zero right-hand side
        const unsigned act = 3u | (ellip ? 12u : 0u) | (sig_held || sig_r50 ? 0u : 16u);
        const bool on = (act >> k & 1) && (act >> l & 1) && c < 5 && lane < 30;
        const float big = __uint_as_float(__reduce_max_sync(kFull, on ? __float_as_uint(fabsf(X)) : 0u));
        if (c == 5) {
            float rv;
            if (JVP) {
                // -(sum u psi + J_as dsigma_w); psi_k = W m_k
                float S5 = 0.f;
#pragma unroll
                for (int j = 5; j >= 0; --j) S5 = fmaf(rec->m[r][j], rec->U[j], S5);
                rv = -(S5 + X * dsw);
            } else {
                rv = a.v[si * 5 + r];
            }
            X = (act >> r & 1) ? rv : 0.f;
        } else if (!on) {
            X = r == c ? big : 0.f;
        }
        if (!solve5(X, big, lane, xs)) status |= FSE_ST_FIT_SINGULAR;
    }
    if (JVP) {
        float val = 0.f;
        if (rg.on) xs[4] = dsw;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if (lane == i && status == 0) val = xs[i];
        if (lane < 5) a.dtheta[si * 5 + lane] = val;
    } else if (lane == 0) {
        // dL/dI_p = -W(p) sum_k lambda_k m_k(p) + kappa d sigma_w / d I_p:
        // the per-stamp coefficients, for the write kernel
        VjpCoef cf;
        cf.x0 = q.x0;
        cf.y0 = q.y0;
        cf.A = q.A;
        cf.B = q.B;
        cf.G4 = q.G4;
        cf.cw = q.cw;
#pragma unroll
        for (int i = 0; i < 6; ++i) cf.c[i] = 0.f;
        cf.kc_in = cf.kc_ring = cf.kc_out = 0.f;
        cf.pc = static_cast<float>(rg.pc);
        cf.pr = static_cast<float>(rg.pr);
        cf.km2 = rg.k >= 1 ? static_cast<float>((rg.k - 1) * (rg.k - 1)) : -1.f;
        cf.k2 = static_cast<float>(rg.k * rg.k);
        cf.ring = rg.on && status == 0;
        cf.ok = status == 0;
        if (status == 0) {
            const float gg = q.g1 * q.g1 + q.g2 * q.g2;
            const float ew1 = 2.f * q.g1 / (1.f + gg), ew2 = 2.f * q.g2 / (1.f + gg);
            cf.c[0] = -xs[4] * q.s * q.s;
            cf.c[1] = xs[0];
            cf.c[2] = xs[1];
            cf.c[3] = xs[2] * (1.f - ew1) - xs[3] * ew2 + xs[4] * q.A;
            cf.c[4] = 2.f * xs[3] - xs[4] * q.G4;
            cf.c[5] = -xs[2] * (1.f + ew1) - xs[3] * ew2 + xs[4] * q.B;
            if (rg.on) {
                float kappa = a.v[si * 5 + 4];
#pragma unroll
                for (int i = 0; i < 4; ++i) kappa = fmaf(-xs[i], Jcol4[i], kappa);
                cf.kc_in = kappa * rg.c_in;
                cf.kc_ring = kappa * rg.c_ring;
                cf.kc_out = kappa * rg.c_out;
            }
        }
        a.coef[si] = cf;
    }
    if (lane == 0 && a.status) a.status[si] = status;
    __syncwarp();   // the sums have been read
}

// One warp per stamp, from the work counter.
//   50,000 stamps of 48x48 (JVP, sigma_w from the growth curve; 922 MB read,
//   0.136 ms at the copy rate): 0.85 ms with the ring's disc sums over the whole
//   stamp, a generic 42-term entry of J per lane and the 5 x 5 solve repeated in
//   every lane; 0.73 ms with the warp sums by exchange; 0.53 ms as it is, bound by
//   issue and instruction fetch (2,000 instructions outside the pixel loop).  A
//   lane per stamp for the solve, 32 stamps at a time, took 0.42 ms here but 75
//   instead of 53 us at 2,090 stamps of 62x62, where it fetches its code for one
//   stamp per warp.
template <int DT, bool JVP>
__global__ void __launch_bounds__(256, 2) moment_grad_kernel(MomentGradArgs a) {
    __shared__ MomSums s_rec[8];
    const int lane = threadIdx.x & 31;
    MomSums* rec = &s_rec[threadIdx.x >> 5];
    if (lane < 30) {
        rec->m[lane / 6][lane % 6] = 0.f;
        rec->du[lane / 6][lane % 6] = 0.f;
    }
    __syncwarp();
    for (;;) {
        unsigned sidx = 0;
        if (lane == 0) sidx = atomicAdd(a.queue, 1u);
        sidx = __shfl_sync(kFull, sidx, 0);
        if (sidx >= static_cast<unsigned long long>(a.count)) break;
        stamp_grad<DT, JVP>(a, static_cast<int64_t>(sidx), lane, rec);
    }
}

// The VJP's pixel gradient from the per-stamp coefficients: it depends on
// the pixels only through the coefficients, so this pass reads none and
// streams the writes.  One warp per stamp, stamps in grid-stride order;
// stamps of invalid size are left unwritten; a stamp without a solution gets
// zeros.  Where rows are multiples of four pixels and the stamp starts on 16
// bytes, a lane writes four pixels of a row at once and shares the row's terms
// between them: 20 instructions a pixel instead of 41.
//   20,000 stamps of 48x48 (184 MB written, 0.027 ms at the copy rate): 67 to 38
//   us.
__global__ void __launch_bounds__(256) moment_vjp_write_kernel(MomentGradArgs a) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t si = gw; si < a.count; si += nw) {
        const fse_stamp ix = a.idx[si];
        const long long npl = static_cast<long long>(ix.h) * ix.w;
        if (ix.h < 1 || ix.w < 1 || npl > FSE_MAX_PIX) continue;
        const int npix = static_cast<int>(npl);
        const VjpCoef cf = a.coef[si];
        float* out = a.dpix + ix.offset;
        const bool vec = (ix.w & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
        if (!cf.ok) {
            for (int p = lane; p < npix; p += 32) __stcs(out + p, 0.f);
            continue;
        }
        // one value from a row's terms and a column: the same operations on both
        // paths, so that a gradient does not depend on where its stamp starts
        float t2, di2, e0, e1, k0, k1;
        auto row = [&](float r) {
            t2 = r - cf.y0;
            const float di = r - cf.pr;
            di2 = di * di;
            e0 = cf.B * t2 * t2;
            e1 = -cf.G4 * t2;
            k0 = fmaf(t2, fmaf(cf.c[5], t2, cf.c[2]), cf.c[0]);
            k1 = fmaf(cf.c[4], t2, cf.c[1]);
        };
        auto value = [&](float x) {
            const float t1 = x - cf.x0;
            const float W = ex2(fmaf(t1, fmaf(cf.A, t1, e1), e0) * cf.cw);
            float g = -W * fmaf(t1, fmaf(cf.c[3], t1, k1), k0);
            if (cf.ring) {
                const float dj = x - cf.pc;
                const float d2 = fmaf(dj, dj, di2);
                g += d2 <= cf.km2 ? cf.kc_in : (d2 <= cf.k2 ? cf.kc_ring : cf.kc_out);
            }
            return g;
        };
        if (vec) {
            FWalk pw(4 * lane, ix.w, 128);
            float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll 2
            for (int p = lane; p < npix / 4; p += 32) {
                row(pw.r);
                const float4 g = make_float4(value(pw.c), value(pw.c + 1.f), value(pw.c + 2.f), value(pw.c + 3.f));
                pw.next();
                __stcs(o4 + p, g);
            }
            continue;
        }
        FWalk pw(lane, ix.w);
        for (int p = lane; p < npix; p += 32) {
            row(pw.r);
            const float g = value(pw.c);
            pw.next();
            __stcs(out + p, g);
        }
    }
}

template <int DT, bool JVP>
cudaError_t launch_t(const MomentGradArgs& a, cudaStream_t stream) {
    auto kern = moment_grad_kernel<DT, JVP>;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long grid = static_cast<long long>(per_sm) * sms;
    const long long need = (a.count + 7) / 8;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    kern<<<static_cast<unsigned>(grid), 256, 0, stream>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess || JVP) return e;
    long long wgrid = (a.count + 7) / 8;          // eight stamps (warps) per CTA
    const long long wcap = static_cast<long long>(sms) * 8;
    if (wgrid > wcap) wgrid = wcap;
    moment_vjp_write_kernel<<<static_cast<unsigned>(wgrid), 256, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_moment_grad(const MomentGradArgs& a, cudaStream_t stream) {
    if (a.count <= 0) return cudaSuccess;
    const bool jvp = a.tangent != nullptr;
    if (a.dtype == FSE_BF16) return jvp ? launch_t<FSE_BF16, true>(a, stream) : launch_t<FSE_BF16, false>(a, stream);
    return jvp ? launch_t<FSE_F32, true>(a, stream) : launch_t<FSE_F32, false>(a, stream);
}

}  // namespace fse
