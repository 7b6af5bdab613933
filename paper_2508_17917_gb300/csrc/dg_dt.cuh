// dg_dt.cuh -- the FP64 time-step bound of one mesh (Eq. rayleigh_bound) in
// two passes: an FP32 screen of every element, then FP64 for the few
// elements that can hold the maximum.
//
// dt = cfl / max_K Lambda_K needs only the largest Lambda_K, and evaluating
// every element in FP64 costs about 30 penalty norms per element on a pipe
// at 1/60 of the FP32 rate.  The screen evaluates Lambda_K in FP32 from the
// FP64 state.  With its values within e of the exact ones, relative, the
// element with the largest Lambda_K is within (1 - e) / (1 + e) of the
// screen's maximum; the FP64 pass takes all elements within kDtMargin =
// 1 - 2^-11 of it, which holds for e <= 2^-12 = 2.4e-4.
//
// Lambda_K is formed of sums, products and maxima of positive terms, some
// tens of roundings of u = 6e-8, except for
//  - the penalty norm N = |B| of the trace: a41 = -(|v|^2 + vn^2/3) -
//    gamma/Pr (e - |v|^2) cancels where gamma/Pr > 2.  Its inputs and terms
//    carry at most 8 u Q, Q = gamma/Pr (e + |v|^2) + 4/3 |v|^2, and an error
//    of one entry of B is at most that in |B|, so Q <= kDtSpread N bounds the
//    relative error by 8 u kDtSpread = 4.8e-5; and at the double root of the
//    eigenvalue's cubic the error of r enters with its square root, 1.5e-4 in
//    N at most.  Measured over states that pass the guard: 1.3e-5 and
//    7.0e-5; without the guard 9e-4 (gamma/Pr = 3, speeds of 9e3);
//  - the sound speed: the pressure's rounding is some u of rho |v|^2 / 2, and
//    p > 1e-3 rho |v|^2 bounds it by 7e-5 of p, 4e-5 of the speed; for the
//    wall ghost, whose energy is formed from p, p > 1e-2 rho |v|^2 and
//    Q <= 4 N give 3e-5 in its norm.
// An element where a guard fails, or with a value that is not finite or
// extreme, is marked (infinity) and goes to the FP64 pass, so the FP64
// maximum over what the pass takes is the maximum over all elements.
// A uniform state on a uniform mesh marks every element; the FP64 pass then
// does what a pass over all elements would.
// 40,800 elements at p = 4: 816 us (one thread per element in FP64, one
// block for the maximum) before, 22 us of screen and 32 us of FP64 now.
#pragma once
#include "dg_stage.cuh"
#include "pair2.cuh"

namespace dg {

constexpr float kDtMargin = 1.0f - 1.0f / 2048.0f;
constexpr float kDtSpread = 100.0f;

// the size of the terms of one trace's norm, Q / rho
__device__ __forceinline__ float norm_terms(float ir, float vsq, float e, float gPr)
{
    return ir * fmaf(gPr, fabsf(e) + vsq, (4.0f / 3.0f) * vsq);
}

// words: [0] largest screened Lambda (FP32 bits), [1] finished blocks,
// [2, 3] largest FP64 Lambda (bits), [4] a candidate was not finite; all zero
// between calls
template <int P>
__global__ void __launch_bounds__(Shape<P>::NT)
dt_screen_kernel(const double *U, const double *geo, const int4 *conn, const int *fmask, long long K, Phys<float> ph,
                 double gm1d, float sig_fac, float *lam, unsigned *words)
{
    using Sh = Shape<P>;
    constexpr int Np = Sh::Np, Nfp = Sh::Nfp, NF = Sh::NF, E = Sh::E;
    __shared__ float sNorm[E * NF], sRmin[E * NF], sBeta[E * Np];
    __shared__ int sMark[E];
    const int tid = threadIdx.x;
    const long long k0 = static_cast<long long>(blockIdx.x) * E;
    const int ne = static_cast<int>((K - k0) < E ? (K - k0) : E);
    if (tid < E) sMark[tid] = 0;
    __syncthreads();
    const int fe = tid / NF, fm = tid - (tid / NF) * NF;
    if (fe < ne) {
        const long long k = k0 + fe;
        const int ff = fm / Nfp, fi = fm - ff * Nfp;
        const int4 cn = conn[k];
        const int f2 = (cn.w >> (2 * ff)) & 3, bt = (cn.w >> (8 + 2 * ff)) & 3;
        const int vm = fmask[fm];
        const double *g = geo + k * 16;
        const float n1 = cvt_d2f(g[G_NX + ff]), n2 = cvt_d2f(g[G_NY + ff]);
        float u[4], w[4];
        double Ed = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Ed = U[(k * 4 + c) * Np + vm];
            u[c] = cvt_d2f(Ed);
        }
        float rmin = u[0];
        if (bt == BCT_INTERIOR) {
            const long long nb = (ff == 0) ? cn.x : (ff == 1 ? cn.y : cn.z);
            const int vp = fmask[f2 * Nfp + (Nfp - 1 - fi)];
#pragma unroll
            for (int c = 0; c < 4; ++c) w[c] = cvt_d2f(U[(nb * 4 + c) * Np + vp]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) w[c] = ph.Uinf[c];
        }
        if (bt != BCT_WALL) rmin = fminf(rmin, w[0]);
        const float pw = (bt == BCT_WALL) ? pressure<float>(u, Ed, gm1d) : 0.f;
        const float ir = 1.0f / u[0];
        const float nrm = trace_norms_max(u, ir, pw, bt, w, n1, n2, ph);
        // the guards; what is not finite reaches `own` or `other`, and the
        // comparisons are written so that a NaN fails them
        const float msq = u[1] * u[1] + u[2] * u[2];
        const float own = norm_terms(ir, msq * ir * ir, u[3] * ir, ph.gPr);
        float other;
        bool ok = rmin > 1e-12f && fmaxf(u[0], w[0]) < 1e12f && nrm < 1e15f && (nrm > 1e-15f || ph.mu == 0.f);
        if (bt == BCT_WALL) {
            const float wsq = ph.vw1 * ph.vw1 + ph.vw2 * ph.vw2;
            other = norm_terms(ir, wsq, fmaf(0.5f, wsq, pw / ph.gm1 * ir), ph.gPr);
            ok = ok && pw > 1e-2f * (msq * ir) && ph.mu * other <= 4.0f * nrm;
        } else {
            const float iw = 1.0f / w[0];
            other = norm_terms(iw, (w[1] * w[1] + w[2] * w[2]) * iw * iw, w[3] * iw, ph.gPr);
        }
        ok = ok && ph.mu * (own + other) <= kDtSpread * nrm;
        sNorm[fm + fe * NF] = nrm;
        sRmin[fm + fe * NF] = rmin;
        if (!ok) sMark[fe] = 1;
    }
    const int ve = tid / Np, vi = tid - (tid / Np) * Np;
    if (ve < ne) {
        const long long k = k0 + ve;
        float u[4];
        double Ed = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Ed = U[(k * 4 + c) * Np + vi];
            u[c] = cvt_d2f(Ed);
        }
        const float ir = 1.0f / u[0], p = pressure<float>(u, Ed, gm1d);
        const float v1 = u[1] * ir, v2 = u[2] * ir;
        const float c = sqrtf(ph.gamma * p * ir);
        const float b1 = fabsf(v1 - ph.vw1) + c, b2 = fabsf(v2 - ph.vw2) + c;
        const float beta = sqrtf(b1 * b1 + b2 * b2);
        sBeta[ve * Np + vi] = beta;
        const bool ok = beta > 1e-12f && beta < 1e12f && p > 1e-3f * (u[1] * v1 + u[2] * v2);
        if (!ok) sMark[ve] = 1;
    }
    __syncthreads();
    if (tid >= ((E + 31) & ~31)) return;
    float L = 0.f;
    if (tid < ne) {
        const long long k = k0 + tid;
        const double *g = geo + k * 16;
        const int4 cn = conn[k];
        const float pp = 0.5f * float((P + 1) * (P + 2));
        float GK = 0.f, sigK = 0.f, ciK = 0.f, perim = 0.f, beta = 0.f;
        const float gdiff = fmaxf(4.0f / 3.0f, ph.gPr) * ph.mu, J = cvt_d2f(g[G_J]);
        bool ok = sMark[tid] == 0 && J > 1e-18f && J < 1e18f;
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            float gbar = 0.f, rmin = INFINITY;
            for (int i = 0; i < Nfp; ++i) {
                gbar = fmaxf(gbar, sNorm[tid * NF + f * Nfp + i]);
                rmin = fminf(rmin, sRmin[tid * NF + f * Nfp + i]);
            }
            const float fs = cvt_d2f(g[G_FS + f]);
            const float ci = pp * fs;
            float cmax = ci;
            if (((cn.w >> (8 + 2 * f)) & 3) == BCT_INTERIOR) {
                const long long nb = (f == 0) ? cn.x : (f == 1 ? cn.y : cn.z);
                cmax = fmaxf(ci, pp * cvt_d2f(geo[nb * 16 + G_FS + ((cn.w >> (2 * f)) & 3)]));
            }
            ok = ok && fs > 1e-9f && cmax < 1e12f;
            GK = fmaxf(GK, gdiff / rmin);
            sigK = fmaxf(sigK, sig_fac * gbar * cmax);
            ciK = fmaxf(ciK, ci);
            perim += 2.0f * fs * J;
        }
        for (int i = 0; i < Np; ++i) beta = fmaxf(beta, sBeta[tid * Np + i]);
        const float rhoK = 4.0f * J / perim;
        L = 1.5f * (float(P * P * P * P) / (rhoK * rhoK)) * GK + 3.0f * ciK * (3.0f * sigK + beta);
        ok = ok && L > 1e-18f && L < 1e30f;
        lam[k] = ok ? L : INFINITY;
        if (!ok) L = 0.f;
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(L));
    if ((tid & 31) == 0 && m > *reinterpret_cast<volatile unsigned *>(words)) atomicMax(words, m);
}

}  // namespace dg
