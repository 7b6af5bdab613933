// stage_fp64.cu -- the FP64 stage kernels (p = 1..6): the three-phase kernel
// of dg_stage64.cuh with its operator tables, the kernels of dg_stage.cuh, and
// the FP64 broken gradient.
#include <cmath>
#include <vector>

#include "dg_stage64.cuh"
#include "launch.h"
#include "refops.h"

namespace dg {
namespace {

// the kernel that needs no memory of its own
template <int P, bool TH, bool OI>
cudaError_t shape_alone_p(long long K, LaunchShape &ls)
{
    using L = Smem<P, double, TH, OI>;
    auto kern = stage_kernel<P, double, TH, OI>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Shape<P>::NT, L::bytes);
    if (e != cudaSuccess) return e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (per_sm < 1) per_sm = 1;
    long long ntiles = (K + Shape<P>::E - 1) / Shape<P>::E;
    long long grid = static_cast<long long>(sms) * per_sm;
    ls.grid = static_cast<int>(ntiles < grid ? ntiles : grid);
    ls.threads = Shape<P>::NT;
    ls.smem = L::bytes;
    ls.elems_per_tile = Shape<P>::E;
    ls.theta = TH;
    ls.overint = OI;
    ls.phases = false;
    return cudaSuccess;
}

// three phases in a cooperative launch: as many blocks as are resident at
// once, capped by what the widest phase has for them
template <int P, bool TH>
cudaError_t shape64_p(long long K, LaunchShape &ls)
{
    using S = Sym64<P>;
    using L = Layout64<P, TH>;
    auto kern = stage64_kernel<P, TH>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, S::NT, L::bytes);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (K + S::EB - 1) / S::EB, groups = (3 * K + 4 * (32 / S::Nfp) - 1) / (4 * (32 / S::Nfp));
    const long long most = tiles > groups ? tiles : groups, grid = static_cast<long long>(sms) * per_sm;
    ls.grid = static_cast<int>(most < grid ? most : grid);
    ls.threads = S::NT;
    ls.smem = L::bytes;
    ls.elems_per_tile = S::EB;
    ls.theta = TH;
    ls.overint = false;
    ls.phases = true;
    return cudaSuccess;
}

template <int P>
cudaError_t launch64_p(const LaunchShape &ls, const StageParams &sp, const Stage64 &x, const Phys<double> &ph,
                       cudaStream_t st)
{
    if (!ls.phases) {
        if (ls.overint)
            stage_kernel<P, double, false, true><<<ls.grid, ls.threads, ls.smem, st>>>(sp, ph);
        else if (ls.theta)
            stage_kernel<P, double, true><<<ls.grid, ls.threads, ls.smem, st>>>(sp, ph);
        else
            stage_kernel<P, double, false><<<ls.grid, ls.threads, ls.smem, st>>>(sp, ph);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ls.grid);
    cfg.blockDim = dim3(ls.threads);
    cfg.dynamicSmemBytes = ls.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (ls.theta) return cudaLaunchKernelEx(&cfg, stage64_kernel<P, true>, sp, x, ph);
    return cudaLaunchKernelEx(&cfg, stage64_kernel<P, false>, sp, x, ph);
}

// Whether the symmetric contraction is taken.  It costs fewer FP64
// instructions from p = 2 on (about, per node, with the plain rows and by symmetry:
// p = 1 40 and 56, p = 2 64 and 54, p = 3 96 and 70, p = 4 136 and 96); at p = 2
// its sums and differences round more than they save (RMS error 1.03 times that
// of the plain rows), and below some thousand elements its two passes through
// shared memory cost more than the pipe.  us, plain and symmetric: p = 1, 256^2
// quads 42 and 60; p = 2 101 and 95; p = 3, 16^2 18.0 and 19.0, 32^2 20.2 and
// 18.8, 256^2 226 and 186.
template <int P>
constexpr bool grad_by_symmetry(long long K)
{
    return P > 3 || (P == 3 && K >= 1500);
}

// blocks of the FP64 gradient: those resident at once, capped by the tiles
template <int P>
cudaError_t grad64_grid_p(long long K, int &grid)
{
    if (!grad_by_symmetry<P>(K)) {
        grid = static_cast<int>((K * Sym64<P>::Np + 127) / 128);
        return cudaSuccess;
    }
    using S = Sym64<P>;
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grad64_kernel<P>, S::NT, 0);
    if (e != cudaSuccess) return e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (K + S::EB - 1) / S::EB, most = static_cast<long long>(sms) * (per_sm < 1 ? 1 : per_sm);
    grid = static_cast<int>(tiles < most ? tiles : most);
    return cudaSuccess;
}

template <int P>
cudaError_t grad64_p(const Grad64Args &a, cudaStream_t st)
{
    if (grad_by_symmetry<P>(a.K))
        grad64_kernel<P><<<a.grid, Sym64<P>::NT, 0, st>>>(a.U, a.geo, reinterpret_cast<const double2 *>(a.ops), a.nodes,
                                                         a.K, a.gx, a.gy);
    else
        grad64_rows_kernel<P><<<a.grid, 128, 0, st>>>(a.U, a.Dr, a.Ds, a.geo, a.K, a.gx, a.gy);
    return cudaGetLastError();
}

template <int P>
bool sym64_tables_p(const RefOps &o, bool theta, std::vector<double> &tab, std::vector<int> &nodes)
{
    using S = Sym64<P>;
    constexpr int Np = S::Np, NF = S::NF, NO = S::NO, NE = S::NE, TPE = S::TPE, NEF = S::NEF;
    // mirrored nodes: (r, s) -> (s, r)
    int mirror[Np];
    for (int i = 0; i < Np; ++i) {
        mirror[i] = -1;
        for (int j = 0; j < Np; ++j)
            if (std::fabs(o.r[i] - o.s[j]) < 1e-10 && std::fabs(o.s[i] - o.r[j]) < 1e-10) mirror[i] = j;
        if (mirror[i] < 0) return false;
    }
    std::vector<int> pair, axis;
    for (int i = 0; i < Np; ++i) {
        if (mirror[i] == i) axis.push_back(i);
        else if (i < mirror[i]) pair.push_back(i);
    }
    if (static_cast<int>(pair.size()) != NO || static_cast<int>(axis.size()) != NE - NO) return false;
    // the reflection exchanges Dr and Ds (and Wr, Ws) and mirrors the face slots
    double worst = 0.0;
    for (int i = 0; i < Np; ++i) {
        for (int j = 0; j < Np; ++j) {
            worst = std::fmax(worst, std::fabs(o.Dr[i * Np + j] - o.Ds[mirror[i] * Np + mirror[j]]));
            worst = std::fmax(worst, std::fabs(o.Wr[i * Np + j] - o.Ws[mirror[i] * Np + mirror[j]]));
        }
        for (int m = 0; m < NF; ++m)
            worst = std::fmax(worst, std::fabs(o.LIFT[i * NF + m] - o.LIFT[mirror[i] * NF + NF - 1 - m]));
    }
    if (!(worst < 1e-9)) return false;
    // The rows of a pair serve both of its nodes, so they are the mean of the
    // two; and the derivative of a constant is zero.  The tables then carry
    // less of the operators' own rounding than the operators do (RMS error of
    // a gradient against exact operators, vortex, p = 4, energy: 0.55e-14 with
    // them, 1.0e-14 with the plain rows, 1.6e-14 with the rows of one node).
    std::vector<double> Dr(o.Dr), Ds(o.Ds), LIFT(o.LIFT), Wr(o.Wr), Ws(o.Ws);
    for (int i = 0; i < Np; ++i) {
        double sum = 0.0;
        for (int j = 0; j < Np; ++j) {
            Dr[i * Np + j] = 0.5 * (o.Dr[i * Np + j] + o.Ds[mirror[i] * Np + mirror[j]]);
            Wr[i * Np + j] = 0.5 * (o.Wr[i * Np + j] + o.Ws[mirror[i] * Np + mirror[j]]);
            sum += Dr[i * Np + j];
        }
        Dr[i * Np + i] -= sum;
        for (int m = 0; m < NF; ++m)
            LIFT[i * NF + m] = 0.5 * (o.LIFT[i * NF + m] + o.LIFT[mirror[i] * NF + NF - 1 - m]);
    }
    for (int i = 0; i < Np; ++i)
        for (int j = 0; j < Np; ++j) {
            Ds[mirror[i] * Np + mirror[j]] = Dr[i * Np + j];
            Ws[mirror[i] * Np + mirror[j]] = Wr[i * Np + j];
        }
    // Q = W LIFT for the theta terms
    std::vector<double> Pm(Np * Np), Mm(Np * Np), Qp(Np * NF, 0.0), Qm(Np * NF, 0.0);
    for (int i = 0; i < Np * Np; ++i) {
        Pm[i] = 0.5 * (Dr[i] + Ds[i]);
        Mm[i] = 0.5 * (Dr[i] - Ds[i]);
    }
    for (int i = 0; theta && i < Np; ++i)
        for (int m = 0; m < NF; ++m)
            for (int j = 0; j < Np; ++j) {
                Qp[i * NF + m] += 0.5 * (Wr[i * Np + j] + Ws[i * Np + j]) * LIFT[j * NF + m];
                Qm[i * NF + m] += 0.5 * (Wr[i * Np + j] - Ws[i * Np + j]) * LIFT[j * NF + m];
            }
    // even (sign +1) and odd (-1) rows of a matrix over nodes, and over face slots
    auto node_row = [&](const std::vector<double> &A, int i, int l, double sign) {
        if (l >= NO) return sign > 0 ? A[i * Np + axis[l - NO]] : 0.0;
        return 0.5 * (A[i * Np + pair[l]] + sign * A[i * Np + mirror[pair[l]]]);
    };
    auto face_row = [&](const std::vector<double> &A, int i, int m, double sign) {
        if (m == NF - 1 - m) return sign > 0 ? A[i * NF + m] : 0.0;
        return 0.5 * (A[i * NF + m] + sign * A[i * NF + NF - 1 - m]);
    };
    tab.assign(2 * S::NTAB, 0.0);
    nodes.assign(2 * TPE, -1);
    for (int t = 0; t < TPE; ++t) {
        const bool pr = t < NO;
        const int a = pr ? pair[t] : axis[2 * (t - NO)];
        const int b = pr ? mirror[pair[t]] : (2 * (t - NO) + 1 < NE - NO ? axis[2 * (t - NO) + 1] : -1);
        nodes[2 * t] = a;
        nodes[2 * t + 1] = b;
        auto put = [&](int at, double x, double y) {
            tab[2 * (at + t)] = x;
            tab[2 * (at + t) + 1] = y;
        };
        for (int l = 0; l < NE; ++l)
            put(l * TPE, node_row(Pm, a, l, 1), pr ? node_row(Mm, a, l, 1) : (b < 0 ? 0.0 : node_row(Pm, b, l, 1)));
        for (int l = 0; l < NO; ++l)
            put(S::oB + l * TPE, pr ? node_row(Pm, a, l, -1) : (b < 0 ? 0.0 : node_row(Mm, b, l, -1)),
                node_row(Mm, a, l, -1));
        for (int m = 0; m < NEF; ++m) {
            put(S::oL + m * TPE, -face_row(LIFT, a, m, 1),
                pr ? -face_row(LIFT, a, m, -1) : (b < 0 ? 0.0 : -face_row(LIFT, b, m, 1)));
            put(S::oQA + m * TPE, -face_row(Qp, a, m, 1),
                pr ? -face_row(Qm, a, m, 1) : (b < 0 ? 0.0 : -face_row(Qp, b, m, 1)));
            put(S::oQB + m * TPE, pr ? -face_row(Qp, a, m, -1) : (b < 0 ? 0.0 : -face_row(Qm, b, m, -1)),
                -face_row(Qm, a, m, -1));
        }
    }
    return true;
}

}  // namespace

#define DG_SWITCH_P(p, CALL)                      \
    switch (p) {                                  \
    case 1: return CALL(1);                       \
    case 2: return CALL(2);                       \
    case 3: return CALL(3);                       \
    case 4: return CALL(4);                       \
    case 5: return CALL(5);                       \
    case 6: return CALL(6);                       \
    default: return cudaErrorInvalidValue;        \
    }

cudaError_t stage_shape_fp64(int p, long long K, bool theta, LaunchShape &out, bool overint, bool phases)
{
#define C_(P) (overint  ? shape_alone_p<P, false, true>(K, out)                                                  \
               : phases ? (theta ? shape64_p<P, true>(K, out) : shape64_p<P, false>(K, out))                     \
                        : (theta ? shape_alone_p<P, true, false>(K, out) : shape_alone_p<P, false, false>(K, out)))
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_stage_fp64(int p, const LaunchShape &ls, const StageParams &sp, const Stage64Args &a,
                              const Phys<double> &ph, cudaStream_t st)
{
    const Stage64 x{reinterpret_cast<const double2 *>(a.ops), a.nodes, a.faces, a.nfaces, a.flux, a.dh, a.th};
#define C_(P) launch64_p<P>(ls, sp, x, ph, st)
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t grad64_grid(int p, long long K, int &grid)
{
#define C_(P) grad64_grid_p<P>(K, grid)
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_grad64(int p, const Grad64Args &a, cudaStream_t st)
{
#define C_(P) grad64_p<P>(a, st)
    DG_SWITCH_P(p, C_)
#undef C_
}

bool build_sym64_tables(const RefOps &o, bool theta, std::vector<double> &tab, std::vector<int> &nodes)
{
    switch (o.p) {
    case 1: return sym64_tables_p<1>(o, theta, tab, nodes);
    case 2: return sym64_tables_p<2>(o, theta, tab, nodes);
    case 3: return sym64_tables_p<3>(o, theta, tab, nodes);
    case 4: return sym64_tables_p<4>(o, theta, tab, nodes);
    case 5: return sym64_tables_p<5>(o, theta, tab, nodes);
    case 6: return sym64_tables_p<6>(o, theta, tab, nodes);
    default: return false;
    }
}

namespace {

template <int P>
void sym32_tables_p(const RefOps &o, const std::vector<double> &tab, const std::vector<int> &nodes,
                    std::vector<float> &tab32, std::vector<int> &slots)
{
    using S = Sym64<P>;
    tab32.resize(4 * S::oQA);
    for (int i = 0; i < S::oQA; ++i) {
        tab32[4 * i] = tab32[4 * i + 1] = static_cast<float>(tab[2 * i]);
        tab32[4 * i + 2] = tab32[4 * i + 3] = static_cast<float>(tab[2 * i + 1]);
    }
    slots.assign(6 * S::TPE, -1);
    for (int t = 0; t < S::TPE; ++t)
        for (int q = 0; q < 2; ++q) {
            const int n = nodes[2 * t + q];
            slots[6 * t + q] = n;
            int at = 6 * t + 2 + 2 * q;
            for (int m = 0; m < S::NF; ++m)
                if (n >= 0 && o.Fmask[m] == n) slots[at++] = m;      // a vertex belongs to two faces
        }
}

}  // namespace

void build_sym32_tables(const RefOps &o, const std::vector<double> &tab, const std::vector<int> &nodes,
                        std::vector<float> &tab32, std::vector<int> &slots)
{
    switch (o.p) {
    case 1: return sym32_tables_p<1>(o, tab, nodes, tab32, slots);
    case 2: return sym32_tables_p<2>(o, tab, nodes, tab32, slots);
    case 3: return sym32_tables_p<3>(o, tab, nodes, tab32, slots);
    case 4: return sym32_tables_p<4>(o, tab, nodes, tab32, slots);
    case 5: return sym32_tables_p<5>(o, tab, nodes, tab32, slots);
    case 6: return sym32_tables_p<6>(o, tab, nodes, tab32, slots);
    default: return;
    }
}

void unique_faces(const int4 *conn, long long K, std::vector<int4> &faces)
{
    std::vector<int4> edge;
    faces.clear();
    faces.reserve(static_cast<size_t>(K) * 3 / 2 + 3);
    for (long long k = 0; k < K; ++k) {
        const int4 cn = conn[k];
        for (int f = 0; f < 3; ++f) {
            const int nb = f == 0 ? cn.x : (f == 1 ? cn.y : cn.z);
            const int f2 = (cn.w >> (2 * f)) & 3, bt = (cn.w >> (8 + 2 * f)) & 3;
            const int4 fc = make_int4(static_cast<int>(k), nb, f | (f2 << 2) | (bt << 4), 0);
            if (bt != BCT_INTERIOR) edge.push_back(fc);
            else if (k < nb) faces.push_back(fc);
        }
    }
    faces.insert(faces.end(), edge.begin(), edge.end());
}

}  // namespace dg
