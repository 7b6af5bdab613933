// dg_stage_handoff.cuh -- the mixed-precision stage kernel with two nodes per
// thread: viscous normal fluxes handed from stage to stage.
//
// Same method as dg_stage_mixed.cuh (strong-form residual of Eq. dg_on_K,
// theta = 0, one stage of Algorithm 1; FP32 arithmetic with FP64 state,
// pressure recovery and registers).  The other shapes are bound by
// instruction issue: they gather all nodes of three neighbours per element
// and form the neighbours' gradients and fluxes at the shared nodes anew
// (731 warp instructions per element at p = 4 in the tensor-core shape).
// Here every element's stage ends with the volume part of the next one,
//   V: gradient and total flux of the new state, which the threads still
//      hold; the divergence, and at the face nodes the pressure and the
//      viscous normal flux, go to memory (16 bytes per node and per face node),
// so that a stage has only
//   F: at every face node, the numerical flux from both traces and both
//      records (5 of a neighbour's 15 nodes at p = 4, no gradient), and
//   U: lift, stage update, FP32 copy and pressure,
// left, with V 585 warp instructions per element at p = 4.  A step's first stage
// (and a residual) starts with a V of its own and a grid barrier; the others
// are ordinary launches.  The price is memory traffic, 52 bytes per DOF and stage
// from DRAM instead of 45.  Measured, us a stage, the shape that was the fastest
// before and this one: p = 5, 128^2 quads 71.1 and 62.6; p = 6, 128^2 88.3 and
// 71.5, 200^2 203 and 164; p = 3, 256^2 112 (one node) and 96; p = 2, 400^2 164
// and 139.  At p = 4 the tensor-core shape stays ahead (478 and 512 on 512^2).
// The contractions use the mirror symmetry r <-> s of the operators as in
// dg_stage64.cuh: a thread owns a pair of mirrored nodes or two nodes of the
// axis, and half the multiply-adds remain; all lanes are busy at every
// degree, where the 32-lane tiles of the tensor-core shape use 18 of 32 for
// the faces at p = 5.
// Rounding: sums and differences of a pair cost a bit that the direct rows do
// not, so fluxes and energy are taken relative to a state of the element, and
// the inviscid fluxes of the two sides of a face node are formed alike.  RMS
// error of a residual against 64 bits, rho, rho v1, rho v2, E, in 1e-5: vortex,
// p = 4: 0.6, 1.9, 1.0, 2.1 (one-node shape 3.0, 7.1, 4.1, 4.6); perturbed free
// stream around a cylinder, in 1e-7: 4.0, 2.4, 10.4, 7.0 (4.1, 3.0, 16.9, 6.2).
#pragma once
#include "bulk.cuh"
#include "dg_stage64.cuh"

namespace dg {

// What the kernel needs beyond StageParams.
struct Stage2 {
    const float4 *ops;         // Sym64 rows, each value twice: (R0, R0, R2, R2), (R1, R1, R3, R3), -LIFT (even, odd)
    const int *nodes;          // [TPE][6]: two nodes (second -1: none), two face slots of each (-1: none)
    const float4 *fin;         // [K][NF]: pressure and Fscale V.n of every face node, this stage's
    float4 *fout;              // ... and the next one's
    float4 *rv;                // [K][Np]: divergence of the flux
    const int *elem_case;      // batch: case of every element (mu, v_b, dt)
    int first, next;           // start with V; end with V of the new state
};

// Groups of GW warps own tiles of EG elements and run independently of each
// other. One warp up to p = 4 (32, 30, 30 and 32 lanes busy, barriers of a
// warp only), the four of the block at p = 5 and 6 (121 and 126 of 128 lanes
// busy; two groups of two warps 55 and 56 of 64). Measured, us a stage with
// one-warp groups and with the block as one group: p = 2, 128^2 quads 23.0 and
// 24.9; p = 3 27.8 and 28.5; p = 4, 512^2 489 and 497; with two-warp groups and
// with the block: p = 5, 128^2 68.6 and 61.1; p = 6, 200^2 175 and 167.
template <int P>
struct Layout2 {
    using S = Sym64<P>;
    static constexpr int GW = P <= 4 ? 1 : 4;
    static constexpr int GT = 32 * GW, NG = S::NT / GT, EG = GT / S::TPE;
    static constexpr int tab = S::oQA;                                   // float4 of operators
    // per element: state components [NE + NO][4], flux components [NE + NO][8]
    static constexpr int gh = S::Np * 4, elem = S::Np * 12;
    static constexpr int FPW = 32 / S::Nfp, NPASS = (3 * EG + FPW - 1) / FPW;     // faces per warp, face passes of a tile
    static constexpr int NpP = (S::Np + 3) & ~3;
    static constexpr size_t al(size_t b) { return (b + 15) & ~size_t(15); }
    static constexpr size_t oFm = sizeof(float4) * tab;
    static constexpr size_t header = al(oFm + sizeof(int) * S::NF);
    // a group's region: components, then its tile's own records, contiguous in memory
    static constexpr size_t oK0 = sizeof(float) * EG * elem;
    static constexpr size_t oK1 = oK0 + sizeof(double) * EG * 4 * S::Np;
    static constexpr size_t oFD = oK1 + sizeof(double) * EG * 4 * S::Np;
    static constexpr size_t oRV = oFD + sizeof(float4) * EG * S::NF;
    static constexpr size_t oU = oRV + sizeof(float4) * EG * S::Np;
    static constexpr size_t oGeo = oU + sizeof(float4) * EG * S::Np;
    static constexpr size_t oConn = oGeo + 64 * EG;
    static constexpr size_t oBar = oConn + sizeof(int4) * EG;
    static constexpr size_t group = oBar + 16;
    static constexpr size_t bytes = header + NG * group;
};

// barrier of a group, and with the conjunction of a predicate.  Both order the
// group's shared-memory accesses; a warp vote alone does not.
template <int GW>
__device__ __forceinline__ void group_sync(int g)
{
    if constexpr (GW == 1) __syncwarp();
    else asm volatile("barrier.cta.sync %0, %1;" ::"r"(g + 1), "n"(32 * GW) : "memory");
}
template <int GW>
__device__ __forceinline__ bool group_and(int g, bool v)
{
    if constexpr (GW == 1) {
        const bool all = __all_sync(0xffffffffu, v);
        __syncwarp();
        return all;
    } else {
        int r;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.s32 p, %1, 0;\n\t"
            "barrier.cta.red.and.pred q, %2, %3, p;\n\t"
            "selp.s32 %0, 1, 0, q;\n\t}"
            : "=r"(r)
            : "r"(int(v)), "r"(g + 1), "n"(32 * GW)
            : "memory");
        return r != 0;
    }
}

__device__ __forceinline__ float4 f4_add(const float4 &a, const float4 &b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 f4_sub(const float4 &a, const float4 &b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }

// acc += o x for the four fields, o given twice
struct acc4 {
    float2 lo = make_float2(0.f, 0.f), hi = make_float2(0.f, 0.f);
    __device__ __forceinline__ void add(const float2 o, const float4 &x)
    {
        lo = __ffma2_rn(o, make_float2(x.x, x.y), lo);
        hi = __ffma2_rn(o, make_float2(x.z, x.w), hi);
    }
    __device__ __forceinline__ float4 f4() const { return make_float4(lo.x, lo.y, hi.x, hi.y); }
};

// sums and differences of a pair's values to the even and odd slots
// ([slot][stride] records), an axis thread's two values to two even slots
template <int P>
__device__ __forceinline__ void put_even_odd2(float4 *ev, float4 *od, int stride, int t, const float4 &a, const float4 &b)
{
    using S = Sym64<P>;
    if (t < S::NO) {
        ev[t * stride] = f4_add(a, b);
        od[t * stride] = f4_sub(a, b);
    } else {
        const int l = S::NO + 2 * (t - S::NO);
        ev[l * stride] = a;
        if (l + 1 < S::NE) ev[(l + 1) * stride] = b;
    }
}

// The products and sums below are written out with their roundings: the fused
// instantiation has the same bits as the five launches.
// contravariant sums G = Fr + Fs and H = Fr - Fs of the total flux
// F_c - v_w U - G grad U at one node, from (Dr +- Ds) u / 2, and its viscous
// part V (x and y; rows 1 to 3).  The flux is taken relative to that of a state
// u0 of the element, except for u0's momentum fluxes other than the pressure
// p0 (about; any constants do): its divergence is the same, its rounding
// smaller.  p0, v0 and H0 = E0 + p0 are the same numbers for all nodes.
struct Ref2 {
    float4 u;
    float p, v1, v2, H;
};
__device__ __forceinline__ Ref2 ref_state2(const float4 &u, float E, float gm1)
{
    const float i = 1.0f / u.x, p = __fmul_rn(gm1, E);
    return {make_float4(u.x, u.y, u.z, E), p, __fmul_rn(u.y, i), __fmul_rn(u.z, i), E + p};
}
__device__ __forceinline__ void node_flux2(const float4 &uu, float p, const Ref2 &r, const float4 &Pu, const float4 &Mu, float ax,
                                           float ay, float bx, float by, const Phys<float> &ph, float4 &Go, float4 &Ho,
                                           float Vx[3], float Vy[3])
{
    float u[4], a[4], b[4], gx[4], gy[4];
    f4_to(uu, u);
    f4_to(Pu, a);
    f4_to(Mu, b);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        gx[c] = fmaf(ax, a[c], bx * b[c]);
        gy[c] = fmaf(ay, a[c], by * b[c]);
    }
    const float ir = 1.0f / u[0], v1 = __fmul_rn(u[1], ir), v2 = __fmul_rn(u[2], ir), e = __fmul_rn(u[3], ir);
    const float v1x = __fmul_rn(fmaf(-v1, gx[0], gx[1]), ir), v1y = __fmul_rn(fmaf(-v1, gy[0], gy[1]), ir);
    const float v2x = __fmul_rn(fmaf(-v2, gx[0], gx[2]), ir), v2y = __fmul_rn(fmaf(-v2, gy[0], gy[2]), ir);
    const float ex = __fmul_rn(fmaf(-e, gx[0], gx[3]), ir), ey = __fmul_rn(fmaf(-e, gy[0], gy[3]), ir);
    const float mu = ph.mu, k = __fmul_rn(mu, ph.gPr);
    Vx[0] = __fmul_rn(mu, fmaf(2.0f / 3.0f, v2y, -4.0f / 3.0f * v1x));
    Vy[1] = __fmul_rn(mu, fmaf(2.0f / 3.0f, v1x, -4.0f / 3.0f * v2y));
    Vx[1] = Vy[0] = __fmul_rn(-mu, v1y + v2x);
    Vx[2] = fmaf(v1, Vx[0], fmaf(v2, Vx[1], -k * fmaf(-v1, v1x, fmaf(-v2, v2x, ex))));
    Vy[2] = fmaf(v1, Vy[0], fmaf(v2, Vy[1], -k * fmaf(-v1, v1y, fmaf(-v2, v2y, ey))));
    const float w1 = v1 - ph.vw1, w2 = v2 - ph.vw2, dr = u[0] - r.u.x, dE = u[3] - r.u.w, dp = p - r.p;
    const float Fx[4] = {fmaf(-ph.vw1, dr, u[1] - r.u.y), fmaf(u[1], w1, dp + Vx[0]), fmaf(u[2], w1, Vx[1]),
                         fmaf(r.H, v1 - r.v1, fmaf(dE, w1, fmaf(dp, v1, Vx[2])))};
    const float Fy[4] = {fmaf(-ph.vw2, dr, u[2] - r.u.z), fmaf(u[1], w2, Vy[0]), fmaf(u[2], w2, dp + Vy[1]),
                         fmaf(r.H, v2 - r.v2, fmaf(dE, w2, fmaf(dp, v2, Vy[2])))};
    float G[4], H[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        G[c] = fmaf(ax, Fx[c], __fmul_rn(ay, Fy[c]));
        H[c] = fmaf(bx, Fx[c], __fmul_rn(by, Fy[c]));
    }
    Go = to_f4(G);
    Ho = to_f4(H);
}

// record of face slot m: the pressure and Fscale V.n.  Fscale n is -grad s,
// grad (r + s), -grad r on faces 0, 1, 2, and a, b = grad (r +- s)
template <int P>
__device__ __forceinline__ void put_trace2(float4 *fd, int m, float p, const float Vx[3], const float Vy[3], float ax, float ay,
                                           float bx, float by)
{
    if (m < 0) return;
    const int f = m / Sym64<P>::Nfp;
    const float a = f == 1 ? 1.0f : -0.5f, b = f == 0 ? 0.5f : (f == 1 ? 0.0f : -0.5f);
    const float nx = fmaf(a, ax, b * bx), ny = fmaf(a, ay, b * by);
    fd[m] = make_float4(p, fmaf(nx, Vx[0], ny * Vy[0]), fmaf(nx, Vx[1], ny * Vy[1]), fmaf(nx, Vx[2], ny * Vy[2]));
}

// inviscid normal flux of one side of a face node
__device__ __forceinline__ void flux_n2(const float u[4], float p, float n1, float n2, const Phys<float> &ph, float F[4])
{
    const float v = __fmul_rn(fmaf(u[1], n1, u[2] * n2), 1.0f / u[0]), w = v - fmaf(ph.vw1, n1, ph.vw2 * n2);
    F[0] = __fmul_rn(u[0], w);
    F[1] = fmaf(u[1], w, p * n1);
    F[2] = fmaf(u[2], w, p * n2);
    F[3] = fmaf(u[3], w, p * v);
}

template <int P, bool BATCH, bool FUSE, int MINB>
__global__ void __launch_bounds__(Sym64<P>::NT, MINB)
stage_handoff_kernel(StageParams sp, Stage2 x, Phys<float> ph)
{
    using S = Sym64<P>;
    using L = Layout2<P>;
    constexpr int Np = S::Np, Nfp = S::Nfp, NF = S::NF, NE = S::NE, NO = S::NO, TPE = S::TPE, NEF = S::NEF;
    constexpr int NpP = L::NpP, FPW = L::FPW, EB = L::EG, GW = L::GW;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *tab = reinterpret_cast<float4 *>(smem_raw);
    int *sFm = reinterpret_cast<int *>(smem_raw + L::oFm);
    const int grp = threadIdx.x / L::GT, gt = threadIdx.x - grp * L::GT;      // group of the block, thread of the group
    unsigned char *gb = smem_raw + L::header + grp * L::group;
    const double *sK0 = reinterpret_cast<const double *>(gb + L::oK0);
    const double *sK1 = reinterpret_cast<const double *>(gb + L::oK1);
    float4 *sFD = reinterpret_cast<float4 *>(gb + L::oFD);     // trace records, then Fscale (F.n - H)
    const float4 *sRV = reinterpret_cast<const float4 *>(gb + L::oRV);
    const float4 *sU = reinterpret_cast<const float4 *>(gb + L::oU);
    const float *sGeo = reinterpret_cast<const float *>(gb + L::oGeo);
    const int4 *sConn = reinterpret_cast<const int4 *>(gb + L::oConn);
    const unsigned sbase = static_cast<unsigned>(__cvta_generic_to_shared(gb)), bar = sbase + unsigned(L::oBar);
    const int tid = threadIdx.x;
    for (int i = tid; i < L::tab; i += S::NT) tab[i] = x.ops[i];
    for (int i = tid; i < NF; i += S::NT) sFm[i] = sp.fmask[i];
    if (gt == 0) {
        mbar_init1(bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int e = gt / TPE, t = gt - (gt / TPE) * TPE;
    const int nA = x.nodes[6 * t], nB = x.nodes[6 * t + 1], nb0 = nB < 0 ? nA : nB;
    const int mA0 = x.nodes[6 * t + 2], mA1 = x.nodes[6 * t + 3], mB0 = x.nodes[6 * t + 4], mB1 = x.nodes[6 * t + 5];
    const float *geo = static_cast<const float *>(sp.geo);
    const long long K = sp.K, ntiles = (K + EB - 1) / EB;
    const long long first_tile = static_cast<long long>(blockIdx.x) * L::NG + grp;
    const long long step = static_cast<long long>(gridDim.x) * L::NG;
    float4 *ev = reinterpret_cast<float4 *>(gb) + e * (L::elem / 4), *od = ev + NE;
    float4 *gev = ev + L::gh / 4, *god = gev + 2 * NE;      // (G, H) records: even, odd
    const bool pair = t < NO, update = sp.mode == STAGE_UPDATE;
    const int h2 = pair ? 1 : 0, o1 = pair ? 0 : 1;         // the second sum's halves of the (G, H) records
    const double gm1d = sp.gm1;
    float dtr = static_cast<float>(sp.dt);
    unsigned parity = 0;
    bool failed = false;       // a copy wait of the group gave up: no more tiles, every grid barrier is still met
    __syncthreads();
    pdl_wait_then_release();

    // V of one tile, from the state and pressure of the thread's two nodes and
    // the element's (rx, ry, sx, sy).  Barriers: ev, od were last read before
    // the one ahead of the divergence of the tile before, gev, god are written
    // after the next one.  `between` runs behind the first one.
    // E0: an energy of the element; the energy is differentiated relative to it.
    auto volume = [&](bool act, long long k, const float4 &uA, const float4 &uB, float pA, float pB, float E0,
                      const float4 &g, auto between) {
        if (act)
            put_even_odd2<P>(ev, od, 1, t, make_float4(uA.x, uA.y, uA.z, uA.w - E0), make_float4(uB.x, uB.y, uB.z, uB.w - E0));
        group_sync<GW>(grp);
        between();
        if (act) {
            acc4 r0, r1, r2, r3;
#pragma unroll
            for (int l = 0; l < NE; ++l) {
                const float4 o = tab[l * TPE + t], v = ev[l];
                r0.add(make_float2(o.x, o.y), v);
                r2.add(make_float2(o.z, o.w), v);
            }
#pragma unroll
            for (int l = 0; l < NO; ++l) {
                const float4 o = tab[S::oB + l * TPE + t], v = od[l];
                r1.add(make_float2(o.x, o.y), v);
                r3.add(make_float2(o.z, o.w), v);
            }
            float4 PA = r0.f4(), MA = r3.f4(), PB = r2.f4(), MB = r1.f4();      // axis: two nodes
            if (pair) {
                const float4 q0 = PA, q1 = MB, q2 = PB, q3 = MA;
                PA = f4_add(q0, q1);
                PB = f4_sub(q0, q1);
                MA = f4_add(q3, q2);
                MB = f4_sub(q3, q2);
            }
            if constexpr (BATCH) {
                const BatchCase &cs = sp.cases[x.elem_case[k]];
                ph.mu = cvt_d2f(cs.mu);
                ph.vw2 = cvt_d2f(cs.vb);
            }
            const float ax = g.x + g.z, ay = g.y + g.w, bx = g.x - g.z, by = g.y - g.w;
            float4 GA, HA, GB, HB;
            float4 *fd = x.fout + k * NF;
            float Vx[3], Vy[3];
            const Ref2 ref = ref_state2(ev[NO], E0, ph.gm1);      // a node on the axis
            node_flux2(uA, pA, ref, PA, MA, ax, ay, bx, by, ph, GA, HA, Vx, Vy);
            put_trace2<P>(fd, mA0, pA, Vx, Vy, ax, ay, bx, by);
            put_trace2<P>(fd, mA1, pA, Vx, Vy, ax, ay, bx, by);
            node_flux2(uB, pB, ref, PB, MB, ax, ay, bx, by, ph, GB, HB, Vx, Vy);
            put_trace2<P>(fd, mB0, pB, Vx, Vy, ax, ay, bx, by);
            put_trace2<P>(fd, mB1, pB, Vx, Vy, ax, ay, bx, by);
            put_even_odd2<P>(gev, god, 2, t, GA, GB);
            put_even_odd2<P>(gev + 1, god + 1, 2, t, HA, HB);
        }
        group_sync<GW>(grp);
        if (act) {
            acc4 s1, s2;
#pragma unroll
            for (int l = 0; l < NE; ++l) {
                const float4 o = tab[l * TPE + t];
                s1.add(make_float2(o.x, o.y), gev[2 * l]);
                s2.add(make_float2(o.z, o.w), gev[2 * l + h2]);
            }
#pragma unroll
            for (int l = 0; l < NO; ++l) {
                const float4 o = tab[S::oB + l * TPE + t];
                s1.add(make_float2(o.z, o.w), god[2 * l + 1]);
                s2.add(make_float2(o.x, o.y), god[2 * l + o1]);
            }
            const float4 a = s1.f4(), b = s2.f4();
            x.rv[k * Np + nA] = pair ? f4_add(a, b) : a;
            if (nB >= 0) x.rv[k * Np + nB] = pair ? f4_sub(a, b) : b;
        }
    };

    for (int stg = 0; stg < (FUSE ? 5 : 1); ++stg) {
    if constexpr (FUSE) {
        fused_stage(sp, stg);
        x.first = stg == 0;
        x.next = stg < 4;
    }
    if (x.first) {
        // into the buffer that this stage reads
        for (long long tile = first_tile; tile < ntiles; tile += step) {
            const long long k = tile * EB + e;
            const bool act = e < EB && k < K;
            float4 uA, uB, g;
            float pA = 0.f, pB = 0.f, E0 = 0.f;
            if (act) {
                uA = __ldcg(sp.Sin + k * Np + nA);
                uB = __ldcg(sp.Sin + k * Np + nb0);
                pA = __ldcg(sp.Pin + k * NpP + nA);
                pB = __ldcg(sp.Pin + k * NpP + nb0);
                E0 = __ldcg(&sp.Sin[k * Np].w);
                g = __ldg(reinterpret_cast<const float4 *>(geo + k * 16));
            }
            volume(act, k, uA, uB, pA, pB, E0, g, [] {});
        }
        fence_async();       // read by bulk copies below
    }
    if (FUSE || x.first) {
        if (!grid_sync(sp.bar, sp.bar_err, gridDim.x, sp.bar_limit)) return;
        float4 *o = const_cast<float4 *>(x.fin);
        x.fin = x.fout;
        x.fout = o;
    }

    // ---- F and U, tile by tile.  A tile's own records arrive by bulk copies,
    // a lane each, issued when the tile before has been read and landing while
    // its V runs; the neighbours' traces are read where they are used.
    const bool need_k1 = update && !sp.first_stage;
    auto issue = [&](long long tile) {
        if (gt >= 32 || tile >= ntiles || failed) return;
        const long long k0 = tile * EB;
        const unsigned ne = static_cast<unsigned>(K - k0 < EB ? K - k0 : EB);
        const unsigned reg = ne * unsigned(sizeof(double) * 4 * Np), nod = ne * unsigned(sizeof(float4) * Np);
        const unsigned fac = ne * unsigned(sizeof(float4) * NF);
        fence_async();
        if (gt == 0)
            mbar_expect(bar, 2u * nod + fac + ne * 80u + (update ? (need_k1 ? 2u : 1u) * reg : 0u));
        __syncwarp();
        if (gt == 0) bulk_g2s(sbase + unsigned(L::oFD), x.fin + k0 * NF, fac, bar);
        if (gt == 1) bulk_g2s(sbase + unsigned(L::oU), sp.Sin + k0 * Np, nod, bar);
        if (gt == 2) bulk_g2s(sbase + unsigned(L::oGeo), geo + k0 * 16, ne * 64u, bar);
        if (gt == 3) bulk_g2s(sbase + unsigned(L::oConn), sp.conn + k0, ne * 16u, bar);
        if (gt == 4) bulk_g2s(sbase + unsigned(L::oRV), x.rv + k0 * Np, nod, bar);
        if (gt == 5 && update) bulk_g2s(sbase + unsigned(L::oK0), sp.K0in + k0 * 4 * Np, reg, bar);
        if (gt == 6 && need_k1) bulk_g2s(sbase + unsigned(L::oK1), sp.K1 + k0 * 4 * Np, reg, bar);
    };
    issue(first_tile);
    for (long long tile = first_tile; tile < ntiles && !failed; tile += step, parity ^= 1u) {
        const long long k0 = tile * EB, k = k0 + e;
        const int ne = static_cast<int>(K - k0 < EB ? K - k0 : EB);
        const bool act = e < ne;
        const bool ok = mbar_wait_bounded(bar, parity, sp.bar_limit);
        if (__all_sync(0xffffffffu, ok)) {
            // ---- F: the Nfp nodes of a face on consecutive lanes
            const int lane = gt & 31, fw = lane / Nfp, i = fw < FPW ? lane - fw * Nfp : 0;
            const float sig = static_cast<float>(sp.sig_fac) * (0.5f * float(P + 1) * float(P + 2));
#pragma unroll 1
            for (int ps = gt >> 5; ps < L::NPASS; ps += GW) {
                if (ps * FPW >= 3 * ne) break;
                const int q = ps * FPW + fw;
                const bool on = fw < FPW && q < 3 * ne;
                const int fe = on ? q / 3 : 0, f = on ? q - 3 * (q / 3) : 0;
                const int4 cn = sConn[fe];
                const long long nb = (f == 0) ? cn.x : (f == 1 ? cn.y : cn.z);
                const int f2 = (cn.w >> (2 * f)) & 3, bt = (cn.w >> (8 + 2 * f)) & 3;
                const int vm = sFm[f * Nfp + i], vp = sFm[f2 * Nfp + (Nfp - 1 - i)];
                // a boundary face names its own element: read, not used
                const float4 w4 = __ldcg(sp.Sin + nb * Np + vp), sb4 = __ldcg(x.fin + nb * NF + f2 * Nfp + (Nfp - 1 - i));
                const float fsb = __ldg(geo + nb * 16 + G_FS + f2);
                const float *g = sGeo + fe * 16;
                const float n1 = g[G_NX + f], n2 = g[G_NY + f], fs = g[G_FS + f];
                float4 *slot = sFD + fe * NF + f * Nfp + i;
                float up[4], um[4], Sa[4], Sb[4], Fa[4], Fb[4], dH[4], D[4];
                f4_to(sU[fe * Np + vm], up);
                f4_to(*slot, Sa);
                f4_to(w4, um);
                f4_to(sb4, Sb);
                const float pp = Sa[0], pm = Sb[0];
                if constexpr (BATCH) {
                    const BatchCase &cs = sp.cases[x.elem_case[k0 + fe]];
                    ph.mu = cvt_d2f(cs.mu);
                    ph.vw2 = cvt_d2f(cs.vb);
                }
                const float nrm = trace_norms_max(up, 1.0f / up[0], pp, bt, um, n1, n2, ph);
                float gbar = 0.f;
#pragma unroll
                for (int l = 0; l < Nfp; ++l) gbar = fmaxf(gbar, __shfl_sync(0xffffffffu, nrm, (lane - i + l) & 31));
                flux_n2(up, pp, n1, n2, ph, Fa);
                Sa[0] = Sb[0] = 0.f;
                if (bt == BCT_INTERIOR) {
                    // Fscale (F+.n - F-.n) / 2: both inviscid fluxes formed alike, so that their rounding cancels
                    // where the traces agree; the viscous ones as stored (the other side's normal is -n)
                    const float sigma = __fmul_rn(__fmul_rn(sig, gbar), fmaxf(fs, fsb)), r = fs / fsb;
                    flux_n2(um, pm, n1, n2, ph, Fb);
                    roe_dissipation(up, pp, um, pm, n1, n2, ph, D);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        dH[c] = fmaf(fs, fmaf(-sigma, up[c] - um[c], 0.5f * ((Fa[c] - Fb[c]) - D[c])), 0.5f * fmaf(r, Sb[c], Sa[c]));
                } else {
                    const float sigma = __fmul_rn(__fmul_rn(sig, gbar), fs);
                    if (bt == BCT_FARFIELD) {
                        const float ub[4] = {ph.Uinf[0], ph.Uinf[1], ph.Uinf[2], ph.Uinf[3]};
                        flux_n2(ub, ph.pinf, n1, n2, ph, Fb);
                        roe_dissipation(up, pp, ub, ph.pinf, n1, n2, ph, D);
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            dH[c] = __fmul_rn(fs, fmaf(-sigma, up[c] - ub[c], 0.5f * ((Fa[c] - Fb[c]) - D[c])));
                    } else {
                        // own broken gradient at the wall node
                        const float *Dr = static_cast<const float *>(sp.ops) + vm * Np, *Ds = Dr + Np * Np;
                        float ur[4] = {0, 0, 0, 0}, us[4] = {0, 0, 0, 0}, gx[4], gy[4], vx[4], vy[4], qx, qy;
                        for (int j = 0; j < Np; ++j) acc_rs(ur, us, make_float2(Dr[j], Ds[j]), sU[fe * Np + j]);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            gx[c] = fmaf(g[G_RX], ur[c], g[G_SX] * us[c]);
                            gy[c] = fmaf(g[G_RY], ur[c], g[G_SY] * us[c]);
                        }
                        const float rb = up[0], kw = 0.5f * rb * (ph.vw1 * ph.vw1 + ph.vw2 * ph.vw2);
                        const float ub[4] = {rb, rb * ph.vw1, rb * ph.vw2, pp / ph.gm1 + kw};
                        flux_n2(ub, pp, n1, n2, ph, Fb);
                        visc_flux_prim(rb, ph.vw1, ph.vw2, ub[3] / rb, gx, gy, ph, vx, vy, &qx, &qy);
                        float vn[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c) vn[c] = fmaf(vx[c], n1, vy[c] * n2);
                        if (ph.adiabatic) vn[3] -= fmaf(qx, n1, qy * n2);
#pragma unroll
                        for (int c = 0; c < 4; ++c) dH[c] = fmaf(fs, fmaf(-sigma, up[c] - ub[c], (Fa[c] - Fb[c]) + vn[c]), Sa[c]);
                    }
                }
                if (on) *slot = to_f4(dH);
            }
        }
        if (!group_and<GW>(grp, ok)) {
            // a copy wait gave up: the flag, then the copies in flight.  They
            // land in this block's memory, and a fused step goes on to its
            // grid barriers: the phase of the mbarrier is not used again.
            failed = true;
            if (gt == 0) {
                if (sp.bar_err) atomicExch(sp.bar_err, 1);
                mbar_wait_bounded(bar, parity, kDrainWaits);
            }
            break;
        }
        // ---- U: s1 is the lift both nodes of a pair share, s2 what changes
        // sign (axis threads: first and second node)
        float4 un2[2], g4;
        float pn[2] = {0.f, 0.f}, E0 = 0.f;
        if (act) {
            acc4 s1, s2;
            const float4 *fd = sFD + e * NF;
#pragma unroll
            for (int m = 0; m < NEF; ++m) {
                const float4 o = tab[S::oL + m * TPE + t], a = fd[m], b = fd[NF - 1 - m];
                const float4 h = m == NF - 1 - m ? a : f4_add(a, b);
                s1.add(make_float2(o.x, o.y), h);
                s2.add(make_float2(o.z, o.w), pair ? f4_sub(a, b) : h);
            }
            if constexpr (BATCH) dtr = cvt_d2f(sp.cases[x.elem_case[k]].dt);
            const float4 a = s1.f4(), b = s2.f4();
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int vi = q ? nB : nA;
                if (q == 1 && nB < 0) break;
                // the tables hold -LIFT: R = -(divergence - lift)
                const float4 l = q ? (pair ? f4_sub(a, b) : b) : (pair ? f4_add(a, b) : a), dv = sRV[e * Np + vi];
                float R[4] = {-(l.x + dv.x), -(l.y + dv.y), -(l.z + dv.z), -(l.w + dv.w)};
                const long long base = k * 4 * Np + vi;
                if (sp.src) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) R[c] += cvt_d2f(sp.src[base + c * Np]);
                }
                if (!update) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) sp.Rout[base + c * Np] = cvt_f2d(R[c]);
                } else {
                    double knew[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const double inc = cvt_f2d(dtr * R[c]);
                        const double k1 = need_k1 ? fma(sp.A, sK1[(e * 4 + c) * Np + vi], inc) : inc;
                        sp.K1[base + c * Np] = k1;
                        knew[c] = fma(sp.B, k1, sK0[(e * 4 + c) * Np + vi]);
                        sp.K0out[base + c * Np] = knew[c];
                    }
                    const float un[4] = {cvt_d2f_trunc(knew[0]), cvt_d2f_trunc(knew[1]), cvt_d2f_trunc(knew[2]),
                                         cvt_d2f_trunc(knew[3])};
                    un2[q] = to_f4(un);
                    pn[q] = pressure<float>(un, knew[3], gm1d);
                    sp.Sout[k * Np + vi] = un2[q];
                    sp.Pout[k * NpP + vi] = pn[q];
                }
            }
            if (nB < 0) {
                un2[1] = un2[0];
                pn[1] = pn[0];
            }
            E0 = sU[e * Np].w;
            g4 = *reinterpret_cast<const float4 *>(sGeo + e * 16);
        }
        if (x.next) {
            volume(act, k, un2[0], un2[1], pn[0], pn[1], E0, g4, [&] { issue(tile + step); });
        } else {
            group_sync<GW>(grp);
            issue(tile + step);
        }
    }
    if (FUSE) fence_async();
    }  // stages
}

}  // namespace dg
