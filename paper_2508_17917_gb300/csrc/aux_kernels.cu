// aux_kernels.cu -- time step, wall forces and finiteness kernels (FP64).
#include <math.h>

#include "dg_dt.cuh"
#include "f64math.cuh"
#include "launch.h"
#include "rigid.h"

namespace dg {
namespace {

__device__ __forceinline__ void load_node(const double *U, int Np, long long k, int i, double u[4])
{
#pragma unroll
    for (int c = 0; c < 4; ++c) u[c] = U[(k * 4 + c) * Np + i];
}

// The FP64 pass of the time-step bound (dg_dt.cuh): Lambda_K of Eq.
// rayleigh_bound,
//   Lambda_K = 3/2 C_inv,2(K) G_K + (d+1) C_inv,K (3 sigma_K + beta_K) + beta'_K,
// with C_inv,2 = p^4 / rho_K^2 (rho_K the inradius 2|K| / perimeter); G_K the
// largest diffusivity of the system, max(4/3, gamma/Pr) mu / rho, over the
// face-node traces of both sides of the faces of K (the largest eigenvalue of
// N G N^T, which does not depend on the normal); sigma_K the largest penalty
// sigma_e of Eq. penalty_final over the faces of K and C_inv,K the largest
// C_inv; beta_K = max over nodes of |b_ns|_2, (b_ns)_j = |v_j - v_w,j| + c
// (Eq. cfl_general), beta'_K = 0 -- on the elements whose screened value is
// within the margin of the largest.  A block looks through every gridDim-th
// element, so that neighbours in the numbering (a ring of equal elements)
// are spread over the blocks, and works on its candidates eight at a time, a
// thread per face node and then per node.  The last block to finish writes
// the maximum and clears the words for the next call.
//
// The maxima below drop a NaN, and the penalty norm turns one into zero, so
// whatever is not finite on the way -- a node's state, its 1 / rho, a norm, a
// wave speed (a negative pressure has none) -- marks the result instead.
constexpr int kDtTile = 8;

// by the exponent bits: no FP64 instruction
__device__ __forceinline__ bool finite64(double x)
{
    return (static_cast<unsigned>(__double2hiint(x)) & 0x7ff00000u) != 0x7ff00000u;
}
__device__ __forceinline__ bool finite_state(const double u[4], double ir)
{
    return finite64(u[0]) && finite64(u[1]) && finite64(u[2]) && finite64(u[3]) && finite64(ir);
}

__global__ void __launch_bounds__(128)
dt_confirm_kernel(AuxMesh m, Phys<double> ph, double sig_fac, const float *lamS, unsigned *words, double *out)
{
    __shared__ int list[128];
    __shared__ int n, isbad;
    __shared__ unsigned long long best;
    __shared__ double sG[kDtTile * 21], sR[kDtTile * 21], sB[kDtTile * 28];
    const int p = m.p, Np = (p + 1) * (p + 2) / 2, Nfp = p + 1, NF = 3 * Nfp, tid = threadIdx.x;
    const float thr = __uint_as_float(words[0]) * kDtMargin;
    const double pp = 0.5 * (p + 1.0) * (p + 2.0);
    if (tid == 0) {
        best = 0ull;
        isbad = 0;
    }
    const long long G = gridDim.x;
    for (long long c0 = 0; c0 * G < m.K; c0 += 128) {
        __syncthreads();
        if (tid == 0) n = 0;
        __syncthreads();
        const long long kc = (c0 + tid) * G + blockIdx.x;
        if (kc < m.K && lamS[kc] >= thr) list[atomicAdd(&n, 1)] = static_cast<int>(kc);
        __syncthreads();
        for (int t0 = 0; t0 < n; t0 += kDtTile) {
            const int nc = min(kDtTile, n - t0);
            for (int it = tid; it < nc * NF; it += 128) {
                const int q = it / NF, s = it - q * NF, f = s / Nfp, i = s - f * Nfp;
                const long long k = list[t0 + q];
                const int4 cn = m.conn[k];
                const int f2 = (cn.w >> (2 * f)) & 3, bt = (cn.w >> (8 + 2 * f)) & 3;
                const double n1 = m.geo[k * 16 + G_NX + f], n2 = m.geo[k * 16 + G_NY + f];
                double u[4], w[4];
                load_node(m.U, Np, k, m.fmask[s], u);
                const double ir = rcp64(u[0]);
                bool ok = finite_state(u, ir);
                const double a = penalty_norm64(ir, u[1] * ir, u[2] * ir, u[3] * ir, n1, n2, ph);
                double b, rmin = u[0];
                if (bt == BCT_WALL) {             // wall ghost: the interior density and pressure
                    const double pw = pressure<double>(u, u[3], ph.gm1);
                    const double eb = (pw / ph.gm1 + 0.5 * u[0] * (ph.vw1 * ph.vw1 + ph.vw2 * ph.vw2)) * ir;
                    b = penalty_norm64(ir, ph.vw1, ph.vw2, eb, n1, n2, ph);
                } else {
                    if (bt == BCT_INTERIOR) {
                        const long long nb = (f == 0) ? cn.x : (f == 1 ? cn.y : cn.z);
                        load_node(m.U, Np, nb, m.fmask[f2 * Nfp + (Nfp - 1 - i)], w);
                    } else {
                        for (int c = 0; c < 4; ++c) w[c] = ph.Uinf[c];
                    }
                    const double iw = rcp64(w[0]);
                    ok = ok && finite_state(w, iw);
                    b = penalty_norm64(iw, w[1] * iw, w[2] * iw, w[3] * iw, n1, n2, ph);
                    rmin = fmin(rmin, w[0]);
                }
                if (!(ok && finite64(a) && finite64(b))) isbad = 1;
                sG[it] = fmax(a, b);
                sR[it] = rmin;
            }
            for (int it = tid; it < nc * Np; it += 128) {
                const long long k = list[t0 + it / Np];
                double u[4];
                load_node(m.U, Np, k, it - (it / Np) * Np, u);
                const double ir = rcp64(u[0]), v1 = u[1] * ir, v2 = u[2] * ir;
                const double pr = ph.gm1 * (u[3] - 0.5 * (u[1] * v1 + u[2] * v2));
                const double c = sqrt64(ph.gamma * pr * ir);
                const double b1 = fabs(v1 - ph.vw1) + c, b2 = fabs(v2 - ph.vw2) + c;
                const double b = sqrt64(b1 * b1 + b2 * b2);
                sB[it] = b;
                if (!(finite_state(u, ir) && finite64(b))) isbad = 1;
            }
            __syncthreads();
            if (tid < nc) {
                const long long k = list[t0 + tid];
                const double *g = m.geo + k * 16;
                const int4 cn = m.conn[k];
                const double gdiff = fmax(4.0 / 3.0, ph.gPr);
                double GK = 0, sigK = 0, ciK = 0, perim = 0, beta = 0;
                for (int f = 0; f < 3; ++f) {
                    double gbar = 0, rmin = INFINITY;
                    for (int i = 0; i < Nfp; ++i) {
                        gbar = fmax(gbar, sG[tid * NF + f * Nfp + i]);
                        rmin = fmin(rmin, sR[tid * NF + f * Nfp + i]);
                    }
                    const double fs = g[G_FS + f], ci = pp * fs;
                    double cmax = ci;
                    if (((cn.w >> (8 + 2 * f)) & 3) == BCT_INTERIOR) {
                        const long long nb = (f == 0) ? cn.x : (f == 1 ? cn.y : cn.z);
                        cmax = fmax(ci, pp * m.geo[nb * 16 + G_FS + ((cn.w >> (2 * f)) & 3)]);
                    }
                    GK = fmax(GK, gdiff * ph.mu / rmin);
                    sigK = fmax(sigK, sig_fac * gbar * cmax);
                    ciK = fmax(ciK, ci);
                    perim += 2.0 * fs * g[G_J];       // |e| = 2 sJ = 2 Fscale J
                }
                for (int i = 0; i < Np; ++i) beta = fmax(beta, sB[tid * Np + i]);
                const double rhoK = 4.0 * g[G_J] / perim;
                const double cinv2 = double(p) * p * p * p / (rhoK * rhoK);
                const double lam = 1.5 * cinv2 * GK + 3.0 * ciK * (3.0 * sigK + beta);
                if (!isfinite(lam)) isbad = 1;
                else if (lam > 0.0) atomicMax(&best, static_cast<unsigned long long>(__double_as_longlong(lam)));
            }
            __syncthreads();
        }
    }
    __syncthreads();
    unsigned long long *gbest = reinterpret_cast<unsigned long long *>(words + 2);
    if (tid == 0) {
        if (best) atomicMax(gbest, best);
        if (isbad) atomicExch(words + 4, 1u);
        __threadfence();
        if (atomicAdd(words + 1, 1u) == gridDim.x - 1) {
            __threadfence();
            const unsigned long long b = atomicExch(gbest, 0ull);
            *out = atomicExch(words + 4, 0u) ? NAN : __longlong_as_double(static_cast<long long>(b));
            words[0] = 0u;
            words[1] = 0u;
        }
    }
}

// Force and moment of one wall face: traction p n - tau n at its face nodes
// (interior trace, n the element's outward normal), integrated with the LGL
// weights scaled by sJ; moment about (xc, yc).  xy: the face nodes'
// coordinates (x, y interleaved).  4 Nfp lanes per face, from lane `base` of
// the warp: lane base + 4 i + c forms the broken gradient of field c at face
// node i, the four lanes of a node exchange fields by shuffles, and the sums
// over the nodes, in node order, end up in all of them.  Few faces and long FP64 chains: latency bounds this,
// so the Np-term sums of a face run side by side instead of one after the
// other in one thread (120 faces at p = 4: 39 us and a separate 4 us sum
// before, 13 us in all now).  Thousands of faces fill the FP64 pipe, to which
// an idle lane costs as much as a busy one: a warp takes as many faces as fit
// (4,000 faces, us a call: p = 1, 54 and 44; p = 2, 56 and 53 -- one face per
// warp, now).
__host__ __device__ __forceinline__ int faces_per_warp(int Nfp) { return Nfp < 8 ? 8 / Nfp : 1; }

__device__ void wall_face_force(const AuxMesh &m, Phys<double> ph, long long k, int f, const double *xy,
                                const double *wface, double xc, double yc, int base, double out[3])
{
    const int p = m.p, Np = (p + 1) * (p + 2) / 2, Nfp = p + 1;
    if (m.elem_case) ph.mu = m.cases[m.elem_case[k]].mu;
    const int lane = threadIdx.x & 31, i = (lane - base) >> 2, c = lane & 3;
    const int ii = i < Nfp ? i : 0;              // idle lanes repeat node 0 and are not summed
    const double *g = m.geo + k * 16;
    const double rx = g[G_RX], ry = g[G_RY], sx = g[G_SX], sy = g[G_SY];
    const double n1 = g[G_NX + f], n2 = g[G_NY + f], sJ = g[G_FS + f] * g[G_J];
    const int vm = m.fmask[f * Nfp + ii];
    const double *Dr = m.Dr + vm * Np, *Ds = m.Ds + vm * Np, *U = m.U + (k * 4 + c) * Np;
    double ur = 0.0, us = 0.0;
#pragma unroll 7
    for (int j = 0; j < Np; ++j) {
        const double uj = U[j];
        ur += Dr[j] * uj;
        us += Ds[j] * uj;
    }
    const double gxc = rx * ur + sx * us, gyc = ry * ur + sy * us, uc = U[vm];
    double gx[4], gy[4], u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int src = (lane & ~3) + q;
        gx[q] = __shfl_sync(0xffffffffu, gxc, src);
        gy[q] = __shfl_sync(0xffffffffu, gyc, src);
        u[q] = __shfl_sync(0xffffffffu, uc, src);
    }
    double vx[4], vy[4];
    visc_flux(u, gx, gy, ph, vx, vy);
    const double pr = pressure<double>(u, u[3], ph.gm1);
    const double wq = sJ * wface[ii];
    const double tx = wq * (pr * n1 - (vx[1] * n1 + vy[1] * n2));
    const double ty = wq * (pr * n2 - (vx[2] * n1 + vy[2] * n2));
    const double tm = (xy[2 * ii] - xc) * ty - (xy[2 * ii + 1] - yc) * tx;
    out[0] = out[1] = out[2] = 0.0;
    for (int l = 0; l < Nfp; ++l) {
        out[0] += __shfl_sync(0xffffffffu, tx, base + 4 * l);
        out[1] += __shfl_sync(0xffffffffu, ty, base + 4 * l);
        out[2] += __shfl_sync(0xffffffffu, tm, base + 4 * l);
    }
}

constexpr int kWallWarps = 4;      // warps (faces) per block of the wall-force kernels

// Sum of n triples by the calling block (256 values at a time in a fixed
// order, whatever the block size), result in s[c][0].
__device__ void block_sum3(const double *partial, int n, double (*s)[256])
{
    for (int t = threadIdx.x; t < 256; t += blockDim.x) {
        double a[3] = {0, 0, 0};
#pragma unroll 4      // the reads of four faces in flight, the sums in order
        for (int i = t; i < n; i += 256)
            for (int c = 0; c < 3; ++c) a[c] += __ldcg(partial + static_cast<long long>(i) * 3 + c);
        for (int c = 0; c < 3; ++c) s[c][t] = a[c];
    }
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        for (int t = threadIdx.x; t < w; t += blockDim.x)
            for (int c = 0; c < 3; ++c) s[c][t] += s[c][t + w];
        __syncthreads();
    }
}

// Wall faces of one mesh, faces_per_warp to a warp: partial[w] = (Fx, Fy, Mz) of face
// w; the last block to finish (ticket, zero between launches) sums them into
// out, so that no second launch waits for the first.
__global__ void wall_force_kernel(AuxMesh m, Phys<double> ph, const int2 *faces, const double *face_xy,
                                  const double *wface, int nwall, double xc, double yc, double *partial,
                                  unsigned *ticket, double *out)
{
    __shared__ double s[3][256];
    __shared__ bool last;
    const int Nfp = m.p + 1, per = faces_per_warp(Nfp), lane = threadIdx.x & 31;
    const int sub = min(lane / (4 * Nfp), per - 1), base = 4 * Nfp * sub;      // lanes past the last face go with it
    const int w0 = (blockIdx.x * kWallWarps + (threadIdx.x >> 5)) * per, w = w0 + sub;
    if (w0 < nwall) {
        const int v = min(w, nwall - 1);
        double o[3];
        wall_face_force(m, ph, faces[v].x, faces[v].y, face_xy + static_cast<long long>(v) * Nfp * 2, wface, xc, yc,
                        base, o);
        if (lane == base && w < nwall) {
            for (int c = 0; c < 3; ++c) partial[static_cast<long long>(w) * 3 + c] = o[c];
            __threadfence();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    block_sum3(partial, nwall, s);
    if (threadIdx.x == 0) {
        for (int c = 0; c < 3; ++c) out[c] = s[c][0];
        *ticket = 0u;
    }
}

// A warp per wall face of every degree group of a batch: the groups' faces
// are numbered consecutively (group g from wg.g[g].base), and face w writes
// partial[w].
__global__ void batch_wall_force_kernel(WallGroups wg, Phys<double> ph, double *partial)
{
    const int w = blockIdx.x * kWallWarps + (threadIdx.x >> 5);
    if (w >= wg.total) return;
    int gi = 0;
    while (gi + 1 < wg.n && w >= wg.g[gi + 1].base) ++gi;
    const WallGroup &G = wg.g[gi];
    const int i = w - G.base, Nfp = G.m.p + 1;
    double o[3];
    wall_face_force(G.m, ph, G.faces[i].x, G.faces[i].y, G.face_xy + static_cast<long long>(i) * Nfp * 2, G.wface, 0.0,
                    0.0, 0, o);
    if ((threadIdx.x & 31) == 0)
        for (int c = 0; c < 3; ++c) partial[static_cast<long long>(w) * 3 + c] = o[c];
}

__global__ void nonfinite_kernel(const double *x, long long n, int *flag)
{
    long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    bool bad = false;
    for (; i < n; i += stride) bad |= !isfinite(x[i]);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) *flag = 1;
}

// ---- batch of independent cases (Algorithm 3 per case, on the device)

// One block per case: max_K Lambda_K over the case's elements, then
// dt = cfl / max (Eq. rayleigh_bound), or the case's entry of `fixed` when
// the caller fixed the steps (the bound is still evaluated and recorded); a
// bound that is not finite freezes the case (dt = 0, bad = 1) instead of
// spreading NaN.  Thread 0 then takes the case's Newmark step with the lift
// of the previous force evaluation (Algorithm 3: F_r = lift / m), giving v_b
// for the coming RK step.  The scan over a case's elements is a chain of
// dependent L2 reads per thread: 1024 threads with four reads in flight (18k
// elements: 26 us with 256 threads and FP64 comparisons, 6 us now).
constexpr int kDtThreads = 1024;
__global__ void __launch_bounds__(kDtThreads)
batch_dt_newmark_kernel(const double *lam, const long long *seg, BatchCase *cases, double cfl, const double *fixed)
{
    __shared__ long long s[32];
    const int i = blockIdx.x;
    const long long b = seg[2 * i], e = seg[2 * i + 1];
    // a non-negative double orders like its bits, so the maximum runs on the
    // integer units (GB300 compares doubles on its FP64 pipe); anything not
    // finite counts as infinity, a negative bound as zero
    constexpr long long kInf = 0x7ff0000000000000ll;
    long long m = 0;
#pragma unroll 4
    for (long long k = b + threadIdx.x; k < e; k += kDtThreads) {
        const long long v = __double_as_longlong(lam[k]);
        m = max(m, (v & kInf) == kInf ? kInf : v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int w = 1; w < kDtThreads / 32; ++w) m = max(m, s[w]);
    BatchCase &cs = cases[i];
    const double l = m == kInf ? NAN : __longlong_as_double(m);
    cs.lam = l;
    if (cs.bad || !isfinite(l) || !(l > 0.0)) {
        cs.bad = 1;
        cs.dt = 0.0;
        cs.vb = 0.0;
        return;
    }
    cs.dt = fixed ? fixed[i] : cfl / l;
    double y = cs.y, yd = cs.yd, ydd = cs.ydd, vb = 0.0;
    if (newmark_step(cs.Mr, cs.Cr, cs.Kr, cs.Fy / cs.mass, cs.dt, y, yd, ydd, vb)) {
        cs.y = y;
        cs.yd = yd;
        cs.ydd = ydd;
        cs.vb = vb;
        cs.t += cs.dt;
    } else {
        cs.bad = 1;
        cs.vb = 0.0;
    }
}

// One block per case: deterministic tree sum of its wall-face partials into
// the case's (Fx, Fy, Mz); with a history, row *counter of hist gets
// (t, dt, y, y', v_b, Fx, Fy, lam) of the case (rows beyond cap are dropped).
// The last block to finish (ticket) advances the row counter once every
// block has read it.
__global__ void batch_forces_record_kernel(const double *partial, const int *wseg, BatchCase *cases,
                                           double *hist, int cap, int *counter, unsigned *ticket)
{
    __shared__ double s[3][256];
    const int i = blockIdx.x, n = gridDim.x;
    const int b = wseg[2 * i], e = wseg[2 * i + 1];
    double a[3] = {0, 0, 0};
    for (int w = b + threadIdx.x; w < e; w += blockDim.x)
        for (int c = 0; c < 3; ++c) a[c] += partial[static_cast<long long>(w) * 3 + c];
    for (int c = 0; c < 3; ++c) s[c][threadIdx.x] = a[c];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 3; ++c) s[c][threadIdx.x] += s[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    BatchCase &cs = cases[i];
    cs.Fx = s[0][0];
    cs.Fy = s[1][0];
    cs.Mz = s[2][0];
    if (!hist) return;
    const int row = *counter;
    if (row < cap) {
        double *h = hist + (static_cast<long long>(row) * n + i) * 8;
        h[0] = cs.t; h[1] = cs.dt; h[2] = cs.y; h[3] = cs.yd;
        h[4] = cs.vb; h[5] = cs.Fx; h[6] = cs.Fy; h[7] = cs.lam;
    }
    __threadfence();
    if (atomicAdd(ticket, 1u) == static_cast<unsigned>(n - 1)) {
        *ticket = 0u;
        *counter = row + 1;
    }
}

// Viscous source of the advected isentropic vortex, S = -div F_v(U_v), in
// closed form.  With (dx, dy) the offset of the node from the nearest
// periodic image of the centre (x0 + u0 t, y0 + v0 t), r^2 = dx^2 + dy^2,
// f = beta / (2 pi) exp((1 - r^2) / 2) and (du, dv) = f (-dy, dx) the
// velocity perturbation: the perturbation is divergence free and its
// Laplacian is -(4 - r^2)(du, dv), the stress work tau : grad v is
// mu f^2 r^4 and the Laplacian of T = 1 - a exp(1 - r^2) is
// 4 a exp(1 - r^2)(1 - r^2), so
//   S_rho = 0,   S_m = mu (4 - r^2) (du, dv),
//   S_E = mu (4 - r^2)(u0 du + v0 dv)
//         + mu beta^2 / (2 pi^2) exp(1 - r^2) (r^2 (2 - r^2) - (1 - r^2) / Pr).
// One thread per node; (xc, yc) is the centre at the stage's time (host,
// FP64); `real` is the arithmetic after the FP64 offsets (FP64 path: double;
// mixed: float).  The constants come precomputed (VortexSource).
template <typename real>
__device__ __forceinline__ void vortex_source_node(const double *xy, long long nn, long long n, int Np,
                                                   const VortexSource &v, double xc, double yc, double *S)
{
    real dx = real(xy[n] - xc), dy = real(xy[nn + n] - yc);
    dx -= real(v.L) * rint(dx * real(v.invL));
    dy -= real(v.L) * rint(dy * real(v.invL));
    const real r2 = dx * dx + dy * dy;
    const real e1 = exp(real(1) - r2);
    const real f = real(v.f0) * sqrt(e1);
    const real du = -f * dy, dv = f * dx;
    const real mu = real(v.mu), w = mu * (real(4) - r2);
    const real sE = w * (real(v.u0) * du + real(v.v0) * dv) +
                    mu * real(v.c2) * e1 * (r2 * (real(2) - r2) - (real(1) - r2) * real(v.invPr));
    const long long k = n / Np;
    const int i = static_cast<int>(n - k * Np);
    double *o = S + k * 4 * Np + i;
    o[0] = 0.0;
    o[Np] = static_cast<double>(w * du);
    o[2 * Np] = static_cast<double>(w * dv);
    o[3 * Np] = static_cast<double>(sE);
}

// ns source arrays (one per stage time, centres (xc[s], yc[s]) given) in one
// launch: S + s * 4 nn holds the source at stage time s.
template <typename real>
__global__ void vortex_source_kernel(const double *xy, long long nn, int Np, VortexSource v, VortexCentres cen,
                                     double *S)
{
    const long long n = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (n >= nn) return;
    for (int s = 0; s < cen.ns; ++s)
        vortex_source_node<real>(xy, nn, n, Np, v, cen.xc[s], cen.yc[s], S + s * 4 * nn);
}

}  // namespace

cudaError_t launch_vortex_source(bool fp64, const double *xy, long long nn, int Np, const VortexSource &v,
                                 const double *t, int ns, double *S, cudaStream_t st)
{
    if (ns < 1 || ns > 5) return cudaErrorInvalidValue;
    const unsigned blocks = static_cast<unsigned>((nn + 255) / 256);
    VortexCentres cen{};
    cen.ns = ns;
    for (int s = 0; s < ns; ++s) {
        cen.xc[s] = v.x0 + v.u0 * t[s];
        cen.yc[s] = v.y0 + v.v0 * t[s];
    }
    if (fp64)
        vortex_source_kernel<double><<<blocks, 256, 0, st>>>(xy, nn, Np, v, cen, S);
    else
        vortex_source_kernel<float><<<blocks, 256, 0, st>>>(xy, nn, Np, v, cen, S);
    return cudaGetLastError();
}

cudaError_t launch_batch_dt_newmark(const double *lam, const long long *seg, BatchCase *cases, int ncases,
                                    double cfl, const double *fixed, cudaStream_t st)
{
    batch_dt_newmark_kernel<<<ncases, kDtThreads, 0, st>>>(lam, seg, cases, cfl, fixed);
    return cudaGetLastError();
}

cudaError_t launch_batch_wall_forces(const WallGroups &wg, const Phys<double> &ph, double *partial,
                                     cudaStream_t st)
{
    if (wg.total < 1) return cudaSuccess;
    batch_wall_force_kernel<<<(wg.total + kWallWarps - 1) / kWallWarps, 32 * kWallWarps, 0, st>>>(wg, ph, partial);
    return cudaGetLastError();
}

cudaError_t launch_batch_forces_record(const double *partial, const int *wseg, BatchCase *cases, int ncases,
                                       double *hist, int cap, int *counter, unsigned *ticket, cudaStream_t st)
{
    batch_forces_record_kernel<<<ncases, 256, 0, st>>>(partial, wseg, cases, hist, cap, counter, ticket);
    return cudaGetLastError();
}

cudaError_t launch_dt_confirm(const AuxMesh &m, const Phys<double> &ph, double sig_fac, const float *lam,
                              unsigned *words, double *out, cudaStream_t st)
{
    // A block takes its tiles one after the other, and on a uniform state every
    // element is a candidate: few elements go one tile to a block, up to two
    // blocks an SM, many 128 to a block, up to eight.  (More blocks cost the
    // usual call, with a handful of candidates, a microsecond per hundred.)  us
    // a call, uniform state, p = 1, with a block per 128 elements and now: 512
    // elements 252 and 61, 8,192 258 and 100.
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = sms > 0 ? sms : 1;
    const long long tiles = (m.K + kDtTile - 1) / kDtTile, scans = (m.K + 127) / 128;
    const long long most = scans < 2 * sms ? 2 * sms : (scans < 8 * sms ? scans : 8 * sms);
    const int blocks = static_cast<int>(tiles < most ? tiles : most);
    dt_confirm_kernel<<<blocks, 128, 0, st>>>(m, ph, sig_fac, lam, words, out);
    return cudaGetLastError();
}

cudaError_t launch_wall_forces(const AuxMesh &m, const Phys<double> &ph, const int2 *faces, const double *face_xy,
                               const double *wface, int nwall, double xc, double yc, double *partial,
                               unsigned *ticket, double *out, cudaStream_t st)
{
    const int at_once = kWallWarps * faces_per_warp(m.p + 1);
    const int blocks = (nwall + at_once - 1) / at_once;
    wall_force_kernel<<<blocks, 32 * kWallWarps, 0, st>>>(m, ph, faces, face_xy, wface, nwall, xc, yc, partial, ticket,
                                                          out);
    return cudaGetLastError();
}

cudaError_t launch_nonfinite(const double *x, long long n, int *flag, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long want = (n + 255) / 256;
    long long blocks = want < 4LL * sms ? want : 4LL * sms;
    if (blocks < 1) blocks = 1;
    nonfinite_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(x, n, flag);
    return cudaGetLastError();
}

}  // namespace dg
