// dg_stage64.cuh -- the FP64 right-hand side and Runge-Kutta stage, in few
// FP64 instructions.
//
// Same method as dg_stage.cuh (strong-form residual of Eq. dg_on_K, IIP or
// with the theta terms, and one stage of Algorithm 1).  GB300 runs FP64 at
// 1/60 of its FP32 rate and the path is bound by the number of FP64
// instructions (one kernel that staged a tile, formed the neighbours'
// gradients and evaluated every face from both sides took about 20,700 per
// element at p = 4 and kept the FP64 pipe full: 1121 us per stage on 32,768
// elements; it is dg_stage.cuh, kept for contexts that this one does not
// suit).  This one takes about 7,000, in three phases of one cooperative
// launch with a grid barrier between them:
//   V  per element: broken gradient, total flux, contravariant components,
//      kept in memory for every node;
//   F  per face, once for both sides: Roe flux, penalty and viscous flux from
//      the two traces and the stored fluxes; Fscale (F.n - H) for each side;
//   U  per element: divergence, lift, stage update.
// The phases' arrays (64 bytes per node and 32 per face node) cost memory
// traffic, of which this path has none to spare: 0.1 of the time.
//
// Contractions by symmetry: the nodes are symmetric under r <-> s, which
// exchanges Dr and Ds.  With x_e = x_j + x_sj and x_o = x_j - x_sj over the
// pairs (j, sj) of mirrored nodes (x_e = x_j on the axis), (Dr + Ds) / 2 maps
// even to even and odd to odd, (Dr - Ds) / 2 even to odd and odd to even, so
// both together cost Np^2 multiply-adds instead of 2 Np^2; LIFT halves the
// same way over the face nodes (slot m mirrors NF - 1 - m).  The metric is
// constant on an element, so it is applied to the sums and differences.  A
// thread owns a pair of mirrored nodes, or two nodes of the axis: four rows
//   R0 (P even), R1 (P odd), R2 (M even), R3 (M odd), P, M = (Dr +- Ds) / 2,
// of node j; out_j = R0 + R1 + R2 + R3, out_sj = R0 - R1 - R2 + R3.  On the
// axis P odd and M even vanish, and a thread takes R0 = P even, R3 = M odd of
// its first node and R2 = P even, R1 = M odd of its second.
#pragma once
#include "dg_stage_mixed.cuh"
#include "f64math.cuh"

namespace dg {

template <int P>
struct Sym64 {
    static constexpr int Np = (P + 1) * (P + 2) / 2, Nfp = P + 1, NF = 3 * Nfp;
    static constexpr int NX = P / 2 + 1;              // nodes on the axis r = s
    static constexpr int NO = (Np - NX) / 2;          // mirrored pairs: odd components
    static constexpr int NE = NO + NX;                // even components
    static constexpr int TPE = NO + (NX + 1) / 2;     // threads per element
    static constexpr int NEF = (NF + 1) / 2;          // even components over the face nodes
    static constexpr int NT = 128, EB = NT / TPE;
    // operator table (double2): D rows (R0, R2) [NE][TPE], (R1, R3) [NO][TPE],
    // -LIFT (even, odd) [NEF][TPE], then (theta) -(P', M') LIFT rows
    // (R0, R2), (R1, R3) [NEF][TPE]
    static constexpr int oB = NE * TPE, oL = oB + NO * TPE, oQA = oL + NEF * TPE, oQB = oQA + NEF * TPE;
    static constexpr int NTAB = oQB + NEF * TPE;
};

template <int P, bool TH>
struct Layout64 {
    using S = Sym64<P>;
    static constexpr int tab = TH ? S::NTAB : S::oQA;                    // double2 of operators
    static constexpr int gh = (S::NE + S::NO) * 8;                       // flux sums and differences
    static constexpr int elem = gh + 2 * S::NEF * 4 + (TH ? 2 * S::NEF * 8 : 0);
    static constexpr size_t oX = sizeof(double2) * tab;
    static constexpr size_t bytes = oX + sizeof(double) * S::EB * elem;
};

// What the FP64 stage needs beyond StageParams.
struct Stage64 {
    const double2 *ops;        // Sym64 operator table
    const int *nodes;          // [TPE][2]: the thread's nodes (second -1: none)
    const int4 *faces;         // (k, neighbour, f | f2 << 2 | type << 4, 0), interior faces first
    int nfaces;
    double *flux;              // [K][Np][8]: G = Fr + Fs, H = Fr - Fs
    double *dh;                // [K][NF][4]: Fscale (F.n - H) of every face node
    double *th;                // theta: [K][NF][8]
};

struct d4 {
    double v[4];
};
__device__ __forceinline__ d4 ld4(const double *p)
{
    const double2 a = __ldcg(reinterpret_cast<const double2 *>(p)), b = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
    return d4{{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ d4 lds4(const double *p)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    return d4{{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(double *p, const double v[4])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}

// sums and differences of a pair's values to the even and odd slots of their
// vectors ([slot][stride], four values each); an axis thread's two values are
// two even slots
template <int P>
__device__ __forceinline__ void put_even_odd(double *ev, double *od, int stride, int t, const double a[4],
                                             const double b[4])
{
    using S = Sym64<P>;
    if (t < S::NO) {
        double s[4], d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            s[c] = a[c] + b[c];
            d[c] = a[c] - b[c];
        }
        st4(ev + t * stride, s);
        st4(od + t * stride, d);
    } else {
        const int l = S::NO + 2 * (t - S::NO);
        st4(ev + l * stride, a);
        if (l + 1 < S::NE) st4(ev + (l + 1) * stride, b);
    }
}

// (Dr + Ds) u / 2 and (Dr - Ds) u / 2 of the thread's two nodes from the
// element's even and odd vectors
template <int P>
__device__ __forceinline__ void sym_gradient(const double2 *tab, const double *ev, const double *od, int t,
                                             double Pu[2][4], double Mu[2][4])
{
    using S = Sym64<P>;
    double r0[4] = {0, 0, 0, 0}, r1[4] = {0, 0, 0, 0}, r2[4] = {0, 0, 0, 0}, r3[4] = {0, 0, 0, 0};
#pragma unroll
    for (int l = 0; l < S::NE; ++l) {
        const double2 o = tab[l * S::TPE + t];
        const d4 x = lds4(ev + 4 * l);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            r0[c] = fma(o.x, x.v[c], r0[c]);
            r2[c] = fma(o.y, x.v[c], r2[c]);
        }
    }
#pragma unroll
    for (int l = 0; l < S::NO; ++l) {
        const double2 o = tab[S::oB + l * S::TPE + t];
        const d4 x = lds4(od + 4 * l);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            r1[c] = fma(o.x, x.v[c], r1[c]);
            r3[c] = fma(o.y, x.v[c], r3[c]);
        }
    }
    if (t < S::NO) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Pu[0][c] = r0[c] + r1[c];
            Pu[1][c] = r0[c] - r1[c];
            Mu[0][c] = r3[c] + r2[c];
            Mu[1][c] = r3[c] - r2[c];
        }
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            Pu[0][c] = r0[c];
            Mu[0][c] = r3[c];
            Pu[1][c] = r2[c];
            Mu[1][c] = r1[c];
        }
    }
}

// total flux F_c - v_w U - G grad U of one node
__device__ __forceinline__ void node_flux64(const double u[4], const double gx[4], const double gy[4],
                                            const Phys<double> &ph, double Fx[4], double Fy[4])
{
    const double ir = rcp64(u[0]), v1 = u[1] * ir, v2 = u[2] * ir, e = u[3] * ir;
    const double p = ph.gm1 * fma(-0.5, fma(u[1], v1, u[2] * v2), u[3]);
    const double ax = fma(-v1, gx[0], gx[1]) * ir, ay = fma(-v1, gy[0], gy[1]) * ir;
    const double bx = fma(-v2, gx[0], gx[2]) * ir, by = fma(-v2, gy[0], gy[2]) * ir;
    const double ex = fma(-e, gx[0], gx[3]) * ir, ey = fma(-e, gy[0], gy[3]) * ir;
    const double m43 = ph.mu * (4.0 / 3.0), m23 = ph.mu * (2.0 / 3.0), k = ph.mu * ph.gPr;
    const double txy = ph.mu * (ay + bx);
    const double p1 = p - fma(m43, ax, -m23 * by), p2 = p - fma(m43, by, -m23 * ax);
    const double qx = k * fma(-v2, bx, fma(-v1, ax, ex)), qy = k * fma(-v2, by, fma(-v1, ay, ey));
    const double w1 = v1 - ph.vw1, w2 = v2 - ph.vw2;
    Fx[0] = u[0] * w1;
    Fx[1] = fma(u[1], w1, p1);
    Fx[2] = fma(u[2], w1, -txy);
    Fx[3] = fma(u[3], w1, fma(v1, p1, fma(-v2, txy, -qx)));
    Fy[0] = u[0] * w2;
    Fy[1] = fma(u[1], w2, -txy);
    Fy[2] = fma(u[2], w2, p2);
    Fy[3] = fma(u[3], w2, fma(v2, p2, fma(-v1, txy, -qy)));
}

// a trace and what the face fluxes need of it
struct Trace64 {
    double u[4], sr, ir, v1, v2, p;     // sqrt(rho), 1 / rho, velocity, pressure
};
__device__ __forceinline__ void trace64(Trace64 &a, const Phys<double> &ph)
{
    const double y = rsqrt64(a.u[0]);
    a.sr = a.u[0] * y;
    a.ir = y * y;
    a.v1 = a.u[1] * a.ir;
    a.v2 = a.u[2] * a.ir;
    a.p = ph.gm1 * fma(-0.5, fma(a.u[1], a.v1, a.u[2] * a.v2), a.u[3]);
}

// roe_dissipation (dg_device.cuh) from two prepared traces
__device__ __forceinline__ void roe64(const Trace64 &a, const Trace64 &b, double n1, double n2, double vwn,
                                      const Phys<double> &ph, double D[4])
{
    const double iw = rcp64(a.sr + b.sr), wa = a.sr * iw, wb = b.sr * iw;
    const double v1 = fma(wa, a.v1, wb * b.v1), v2 = fma(wa, a.v2, wb * b.v2);
    const double H = fma(wa, (a.u[3] + a.p) * a.ir, wb * ((b.u[3] + b.p) * b.ir));
    const double hq = 0.5 * fma(v1, v1, v2 * v2), c2 = ph.gm1 * (H - hq);
    const double y = rsqrt64(c2), c = c2 * y, hic2 = 0.5 * (y * y);
    const double un = fma(v1, n1, v2 * n2), ut = fma(v2, n1, -v1 * n2), rt = a.sr * b.sr;
    const double d1 = a.v1 - b.v1, d2 = a.v2 - b.v2;
    const double dun = fma(d1, n1, d2 * n2), dut = fma(d2, n1, -d1 * n2);
    const double dr = a.u[0] - b.u[0], dp = a.p - b.p, rc = rt * c * dun, wn = un - vwn;
    const double w1 = fabs(wn - c) * ((dp - rc) * hic2), w4 = fabs(wn + c) * ((dp + rc) * hic2);
    const double l2 = fabs(wn), w2 = l2 * fma(-2.0 * dp, hic2, dr), w3 = l2 * rt * dut;
    const double s = w1 + w4 + w2, m = c * (w4 - w1);
    D[0] = s;
    D[1] = fma(v1, s, fma(n1, m, -w3 * n2));
    D[2] = fma(v2, s, fma(n2, m, w3 * n1));
    D[3] = fma(H, w1 + w4, fma(un, m, fma(hq, w2, w3 * ut)));
}

__device__ __forceinline__ void load_trace(Trace64 &a, const double *U, int Np, long long k, int i)
{
#pragma unroll
    for (int c = 0; c < 4; ++c) a.u[c] = U[(k * 4 + c) * Np + i];
}

// Fscale F.n of face f (total flux) from G and H: -Fs, Fr + Fs, -Fr on faces
// 0, 1, 2, whose outward normals are -grad s, grad (r + s), -grad r
__device__ __forceinline__ void normal_flux64(const double *flux, int f, double S[4])
{
    const double a = f == 1 ? 1.0 : -0.5, b = f == 0 ? 0.5 : (f == 1 ? 0.0 : -0.5);
    const d4 g = ld4(flux), h = ld4(flux + 4);
#pragma unroll
    for (int c = 0; c < 4; ++c) S[c] = fma(a, g.v[c], b * h.v[c]);
}

// theta vectors of one side, scaled and mapped to (r + s, r - s)
__device__ __forceinline__ void put_theta64(double *th, const double *g, double rho, double v1, double v2, double e,
                                            const double jmp[4], double n1, double n2, double sc,
                                            const Phys<double> &ph)
{
    double tx[4], ty[4], a[4], b[4];
    theta_vec(rho, v1, v2, e, jmp, n1, n2, ph, tx, ty);
    const double px = sc * (g[G_RX] + g[G_SX]), py = sc * (g[G_RY] + g[G_SY]);
    const double mx = sc * (g[G_RX] - g[G_SX]), my = sc * (g[G_RY] - g[G_SY]);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        a[c] = fma(px, tx[c], py * ty[c]);
        b[c] = fma(mx, tx[c], my * ty[c]);
    }
    st4(th, a);
    st4(th + 4, b);
}

// Four 128-thread blocks per SM (128 registers): enough warps to keep the
// FP64 pipe busy, and a grid of 608 blocks whose barrier costs about 2 us.
template <int P, bool TH>
__global__ void __launch_bounds__(Sym64<P>::NT, 4)
stage64_kernel(StageParams sp, Stage64 x, Phys<double> ph)
{
    using S = Sym64<P>;
    using L = Layout64<P, TH>;
    constexpr int Np = S::Np, Nfp = S::Nfp, NF = S::NF, NE = S::NE, NO = S::NO, TPE = S::TPE, EB = S::EB, NEF = S::NEF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *tab = reinterpret_cast<double2 *>(smem_raw);
    double *sX = reinterpret_cast<double *>(smem_raw + L::oX);
    const int tid = threadIdx.x;
    for (int i = tid; i < L::tab; i += S::NT) tab[i] = x.ops[i];
    const int e = tid / TPE, t = tid - (tid / TPE) * TPE;
    const int nA = x.nodes[2 * t], nB = x.nodes[2 * t + 1], nb0 = nB < 0 ? nA : nB;
    const double *geo = static_cast<const double *>(sp.geo);
    const long long K = sp.K, ntiles = (K + EB - 1) / EB;
    double *mine = sX + e * L::elem;

    // ---- V
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long k = tile * EB + e;
        const bool act = e < EB && k < K;
        double u[2][4];
        __syncthreads();
        if (act) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                u[0][c] = sp.K0in[(k * 4 + c) * Np + nA];
                u[1][c] = sp.K0in[(k * 4 + c) * Np + nb0];
            }
            put_even_odd<P>(mine, mine + 4 * NE, 4, t, u[0], u[1]);
        }
        __syncthreads();
        if (act) {
            double Pu[2][4], Mu[2][4];
            sym_gradient<P>(tab, mine, mine + 4 * NE, t, Pu, Mu);
            const double *g = geo + k * 16;
            const double ax = g[G_RX] + g[G_SX], ay = g[G_RY] + g[G_SY], bx = g[G_RX] - g[G_SX], by = g[G_RY] - g[G_SY];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                double gx[4], gy[4], Fx[4], Fy[4], G[4], H[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    gx[c] = fma(ax, Pu[q][c], bx * Mu[q][c]);
                    gy[c] = fma(ay, Pu[q][c], by * Mu[q][c]);
                }
                node_flux64(u[q], gx, gy, ph, Fx, Fy);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    G[c] = fma(ax, Fx[c], ay * Fy[c]);
                    H[c] = fma(bx, Fx[c], by * Fy[c]);
                }
                double *o = x.flux + (k * Np + (q ? nb0 : nA)) * 8;
                if (q == 0 || nB >= 0) {
                    st4(o, G);
                    st4(o + 4, H);
                }
            }
        }
    }
    if (!grid_sync(sp.bar, sp.bar_err, gridDim.x, sp.bar_limit)) return;

    // ---- F: the Nfp nodes of a face on consecutive lanes
    {
        constexpr int FPW = 32 / Nfp;
        const int lane = tid & 31, fw = lane / Nfp, i = lane - fw * Nfp;
        const long long nw = static_cast<long long>(gridDim.x) * (S::NT / 32);
        const long long groups = (x.nfaces + FPW - 1) / FPW;
        const double vhalf = 0.5 * (P + 1) * (P + 2);
        for (long long gr = static_cast<long long>(blockIdx.x) * (S::NT / 32) + (tid >> 5); gr < groups; gr += nw) {
            const long long fi = gr * FPW + fw;
            const bool act = fw < FPW && fi < x.nfaces;
            const int4 fc = x.faces[act ? fi : x.nfaces - 1];
            const long long k = fc.x, kb = fc.y;
            const int f = fc.z & 3, f2 = (fc.z >> 2) & 3, bt = fc.z >> 4;
            const int ii = act ? i : 0;
            const int vm = sp.fmask[f * Nfp + ii], vp = sp.fmask[f2 * Nfp + (Nfp - 1 - ii)];
            const double *g = geo + k * 16, *gb = geo + kb * 16;
            const double n1 = g[G_NX + f], n2 = g[G_NY + f], fs = g[G_FS + f], fsb = gb[G_FS + f2];
            Trace64 a, b;
            load_trace(a, sp.K0in, Np, k, vm);
            trace64(a, ph);
            if (bt == BCT_INTERIOR) {
                load_trace(b, sp.K0in, Np, kb, vp);
            } else if (bt == BCT_FARFIELD) {
#pragma unroll
                for (int c = 0; c < 4; ++c) b.u[c] = ph.Uinf[c];
            } else {
                // wall ghost: density and pressure of the interior, velocity of the wall
                b.u[0] = a.u[0];
                b.u[1] = a.u[0] * ph.vw1;
                b.u[2] = a.u[0] * ph.vw2;
                b.u[3] = a.p / ph.gm1 + 0.5 * a.u[0] * (ph.vw1 * ph.vw1 + ph.vw2 * ph.vw2);
            }
            trace64(b, ph);
            const double na = penalty_norm64(a.ir, a.v1, a.v2, a.u[3] * a.ir, n1, n2, ph);
            const double nb = penalty_norm64(b.ir, b.v1, b.v2, b.u[3] * b.ir, n1, n2, ph);
            // norms are not negative: their bits order like their values; the
            // larger one of a side that is not a number is the other's
            const double nmax = fmax(na, nb);
            double gbar = 0.0;
#pragma unroll
            for (int l = 0; l < Nfp; ++l) gbar = fmax(gbar, __shfl_sync(0xffffffffu, nmax, (lane - i + l) & 31));
            const double vwn = ph.vw1 * n1 + ph.vw2 * n2;
            double jmp[4], D[4], Sa[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) jmp[c] = a.u[c] - b.u[c];
            if (bt == BCT_INTERIOR) {
                const double sigma = sp.sig_fac * vhalf * gbar * (fs > fsb ? fs : fsb);
                double Sb[4];
                normal_flux64(x.flux + (k * Np + vm) * 8, f, Sa);
                normal_flux64(x.flux + (kb * Np + vp) * 8, f2, Sb);
                roe64(a, b, n1, n2, vwn, ph, D);
                const double ia = 0.5 * rcp64(fs), ib = 0.5 * rcp64(fsb);
                double ha[4], hb[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const double m = fma(Sa[c], ia, Sb[c] * ib), d = fma(0.5, D[c], sigma * jmp[c]);
                    ha[c] = fs * (m - d);
                    hb[c] = fsb * (m + d);
                }
                if (act) {
                    st4(x.dh + (k * NF + f * Nfp + ii) * 4, ha);
                    st4(x.dh + (kb * NF + f2 * Nfp + (Nfp - 1 - ii)) * 4, hb);
                    if constexpr (TH) {
                        // the other side's jump and normal both change sign
                        put_theta64(x.th + (k * NF + f * Nfp + ii) * 8, g, a.u[0], a.v1, a.v2, a.u[3] * a.ir, jmp, n1,
                                    n2, 0.5 * sp.theta * fs, ph);
                        put_theta64(x.th + (kb * NF + f2 * Nfp + (Nfp - 1 - ii)) * 8, gb, b.u[0], b.v1, b.v2,
                                    b.u[3] * b.ir, jmp, n1, n2, 0.5 * sp.theta * fsb, ph);
                    }
                }
            } else {
                const double sigma = sp.sig_fac * vhalf * gbar * fs;
                const Trace64 &s = bt == BCT_WALL ? b : a;               // the state G is taken at
                double Fb[4], dH[4];
                flux_n(b.u, b.p, n1, n2, ph, Fb);
                if (bt == BCT_FARFIELD) {
                    double Fa[4];
                    flux_n(a.u, a.p, n1, n2, ph, Fa);
                    roe64(a, b, n1, n2, vwn, ph, D);
#pragma unroll
                    for (int c = 0; c < 4; ++c) dH[c] = 0.5 * (Fa[c] - Fb[c] - D[c]) - sigma * jmp[c];
                } else {
                    // own broken gradient at the wall node
                    const double *Dr = static_cast<const double *>(sp.ops) + vm * Np, *Ds = Dr + Np * Np;
                    double ur[4] = {0, 0, 0, 0}, us[4] = {0, 0, 0, 0}, gx[4], gy[4], vx[4], vy[4], qx, qy;
                    for (int j = 0; j < Np; ++j) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const double uj = sp.K0in[(k * 4 + c) * Np + j];
                            ur[c] = fma(Dr[j], uj, ur[c]);
                            us[c] = fma(Ds[j], uj, us[c]);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        gx[c] = g[G_RX] * ur[c] + g[G_SX] * us[c];
                        gy[c] = g[G_RY] * ur[c] + g[G_SY] * us[c];
                    }
                    visc_flux_prim(b.u[0], ph.vw1, ph.vw2, b.u[3] * b.ir, gx, gy, ph, vx, vy, &qx, &qy);
                    double vn[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) vn[c] = vx[c] * n1 + vy[c] * n2;
                    if (ph.adiabatic) vn[3] -= qx * n1 + qy * n2;
                    normal_flux64(x.flux + (k * Np + vm) * 8, f, Sa);
                    const double ia = 1.0 / fs;
#pragma unroll
                    for (int c = 0; c < 4; ++c) dH[c] = Sa[c] * ia - (Fb[c] - vn[c] + sigma * jmp[c]);
                }
                if (act) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) dH[c] *= fs;
                    st4(x.dh + (k * NF + f * Nfp + ii) * 4, dH);
                    if constexpr (TH)
                        put_theta64(x.th + (k * NF + f * Nfp + ii) * 8, g, s.u[0], s.v1, s.v2, s.u[3] * s.ir, jmp, n1,
                                    n2, sp.theta * fs, ph);
                }
            }
        }
    }
    if (!grid_sync(sp.bar, sp.bar_err, gridDim.x, sp.bar_limit)) return;

    // ---- U: s1 collects what both nodes of a pair share, s2 what changes
    // sign (axis threads: first and second node); R = -(s1 + s2), -(s1 - s2)
    const bool pair = t < NO;
    const int h2 = pair ? 4 : 0, o1 = pair ? 0 : 4;      // s2's halves of the (G, H) records
    double *od = mine + NE * 8, *he = mine + L::gh, *ho = he + NEF * 4, *te = he + NEF * 8, *to = te + NEF * 8;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long k = tile * EB + e;
        const bool act = e < EB && k < K;
        __syncthreads();
        if (act) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const d4 a = ld4(x.flux + (k * Np + nA) * 8 + 4 * q), b = ld4(x.flux + (k * Np + nb0) * 8 + 4 * q);
                put_even_odd<P>(mine + 4 * q, od + 4 * q, 8, t, a.v, b.v);
            }
            for (int m = t; m < NEF; m += TPE) {
                const int mm = NF - 1 - m;
                auto split = [&](const double *p, int stride, double *ev, double *odd) {
                    d4 a = ld4(p + m * stride), b = ld4(p + mm * stride);
                    double s[4], d[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        s[c] = m == mm ? a.v[c] : a.v[c] + b.v[c];
                        d[c] = a.v[c] - b.v[c];
                    }
                    st4(ev, s);
                    st4(odd, d);
                };
                split(x.dh + k * NF * 4, 4, he + 4 * m, ho + 4 * m);
                if constexpr (TH) {
                    split(x.th + k * NF * 8, 8, te + 8 * m, to + 8 * m);
                    split(x.th + k * NF * 8 + 4, 8, te + 8 * m + 4, to + 8 * m + 4);
                }
            }
        }
        __syncthreads();
        if (!act) continue;
        double s1[4] = {0, 0, 0, 0}, s2[4] = {0, 0, 0, 0};
#pragma unroll
        for (int l = 0; l < NE; ++l) {
            const double2 o = tab[l * TPE + t];
            const d4 a = lds4(mine + 8 * l), b = lds4(mine + 8 * l + h2);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                s1[c] = fma(o.x, a.v[c], s1[c]);
                s2[c] = fma(o.y, b.v[c], s2[c]);
            }
        }
#pragma unroll
        for (int l = 0; l < NO; ++l) {
            const double2 o = tab[S::oB + l * TPE + t];
            const d4 a = lds4(od + 8 * l + 4), b = lds4(od + 8 * l + o1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                s1[c] = fma(o.y, a.v[c], s1[c]);
                s2[c] = fma(o.x, b.v[c], s2[c]);
            }
        }
        const double *h2p = pair ? ho : he;
#pragma unroll
        for (int m = 0; m < NEF; ++m) {
            const double2 o = tab[S::oL + m * TPE + t];
            const d4 a = lds4(he + 4 * m), b = lds4(h2p + 4 * m);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                s1[c] = fma(o.x, a.v[c], s1[c]);
                s2[c] = fma(o.y, b.v[c], s2[c]);
            }
        }
        if constexpr (TH) {
#pragma unroll 2
            for (int m = 0; m < NEF; ++m) {
                const double2 oa = tab[S::oQA + m * TPE + t], ob = tab[S::oQB + m * TPE + t];
                const d4 pe = lds4(te + 8 * m), e2 = lds4(te + 8 * m + h2), mo = lds4(to + 8 * m + 4), q2 = lds4(to + 8 * m + o1);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    s1[c] = fma(oa.x, pe.v[c], fma(ob.y, mo.v[c], s1[c]));
                    s2[c] = fma(oa.y, e2.v[c], fma(ob.x, q2.v[c], s2[c]));
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (q == 1 && nB < 0) break;
            const long long base = k * 4 * Np + (q ? nB : nA);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const long long idx = base + c * Np;
                double R = pair ? (q ? s2[c] - s1[c] : -s1[c] - s2[c]) : (q ? -s2[c] : -s1[c]);
                if (sp.src) R += sp.src[idx];
                if (sp.mode == STAGE_RHS_ONLY) {
                    sp.Rout[idx] = R;
                } else {
                    const double inc = sp.dt * R;
                    const double k1 = sp.first_stage ? inc : fma(sp.A, sp.K1[idx], inc);
                    sp.K1[idx] = k1;
                    sp.K0out[idx] = fma(sp.B, k1, sp.K0in[idx]);
                }
            }
        }
    }
}

// Broken gradient of every element (dg_broken_gradient, FP64), by the same
// symmetric contraction: about 1,250 FP64 instructions per element at p = 4
// against 2,040 with the plain rows, on a kernel bound by their number.
template <int P>
__global__ void __launch_bounds__(Sym64<P>::NT)
grad64_kernel(const double *U, const double *geo, const double2 *ops, const int *nodes, long long K, double *gx, double *gy)
{
    using S = Sym64<P>;
    constexpr int Np = S::Np, NE = S::NE, EB = S::EB, TPE = S::TPE;
    __shared__ double2 tab[S::oL];
    __shared__ __align__(16) double sX[EB * Np * 4];
    const int tid = threadIdx.x;
    for (int i = tid; i < S::oL; i += S::NT) tab[i] = ops[i];
    const int e = tid / TPE, t = tid - (tid / TPE) * TPE;
    const int nA = nodes[2 * t], nB = nodes[2 * t + 1], nb0 = nB < 0 ? nA : nB;
    double *mine = sX + e * Np * 4;
    const long long ntiles = (K + EB - 1) / EB;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long k = tile * EB + e;
        const bool act = e < EB && k < K;
        __syncthreads();
        if (act) {
            double a[4], b[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                a[c] = U[(k * 4 + c) * Np + nA];
                b[c] = U[(k * 4 + c) * Np + nb0];
            }
            put_even_odd<P>(mine, mine + 4 * NE, 4, t, a, b);
        }
        __syncthreads();
        if (!act) continue;
        double Pu[2][4], Mu[2][4];
        sym_gradient<P>(tab, mine, mine + 4 * NE, t, Pu, Mu);
        const double *g = geo + k * 16;
        const double ax = g[G_RX] + g[G_SX], ay = g[G_RY] + g[G_SY], bx = g[G_RX] - g[G_SX], by = g[G_RY] - g[G_SY];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (q == 1 && nB < 0) break;
            const long long o = k * 4 * Np + (q ? nB : nA);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                gx[o + c * Np] = fma(ax, Pu[q][c], bx * Mu[q][c]);
                gy[o + c * Np] = fma(ay, Pu[q][c], by * Mu[q][c]);
            }
        }
    }
}

// The same with a thread per (element, node) and the plain rows.
template <int P>
__global__ void __launch_bounds__(128)
grad64_rows_kernel(const double *U, const double *Dr, const double *Ds, const double *geo, long long K, double *gx, double *gy)
{
    constexpr int Np = Sym64<P>::Np;
    const long long n = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (n >= K * Np) return;
    const long long k = n / Np;
    const int i = static_cast<int>(n - k * Np);
    const double *g = geo + k * 16;
    const double rx = g[G_RX], ry = g[G_RY], sx = g[G_SX], sy = g[G_SY];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double *u = U + (k * 4 + c) * Np;
        double ur = 0.0, us = 0.0;
        for (int j = 0; j < Np; ++j) {
            ur += Dr[i * Np + j] * u[j];
            us += Ds[i * Np + j] * u[j];
        }
        gx[(k * 4 + c) * Np + i] = rx * ur + sx * us;
        gy[(k * 4 + c) * Np + i] = ry * ur + sy * us;
    }
}

}  // namespace dg
