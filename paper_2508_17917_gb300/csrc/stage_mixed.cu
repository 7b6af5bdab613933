// stage_mixed.cu -- mixed-precision stage kernel instantiations (p = 1..6):
// FP32 arithmetic, FP64 state in HBM, FP64 pressure recovery and registers.
#include "dg_dt.cuh"
#include "dg_stage_mixed.cuh"
#include "dg_stage_handoff.cuh"
#include "dg_stage_mixed2.cuh"
#include "handoff_grid.h"
#include "launch.h"

namespace dg {

namespace {

template <int P, bool TH>
cudaError_t shape_p(long long K, LaunchShape &ls)
{
    using L = MixedLayout<P, TH>;
    auto kern = stage_mixed_kernel<P, TH>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
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
    return cudaSuccess;
}

template <int P>
cudaError_t launch_p(const LaunchShape &ls, const StageParams &sp, const Phys<float> &ph, cudaStream_t st)
{
    if (ls.theta) return launch_pdl(stage_mixed_kernel<P, true, false, false>, ls, st, sp, ph);
    return launch_pdl(stage_mixed_kernel<P, false, false, false>, ls, st, sp, ph);
}

template <int P>
cudaError_t shape_batch_p(long long ntiles, LaunchShape &ls)
{
    using L = MixedLayout<P, false>;
    auto kern = stage_mixed_kernel<P, false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Shape<P>::NT, L::bytes);
    if (e != cudaSuccess) return e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (per_sm < 1) per_sm = 1;
    long long grid = static_cast<long long>(sms) * per_sm;
    ls.grid = static_cast<int>(ntiles < grid ? ntiles : grid);
    ls.threads = Shape<P>::NT;
    ls.smem = L::bytes;
    ls.elems_per_tile = Shape<P>::E;
    ls.theta = false;
    return cudaSuccess;
}

template <int P>
cudaError_t launch_batch_p(const LaunchShape &ls, const StageParams &sp, const Phys<float> &ph, cudaStream_t st)
{
    // batch stage launches are graph-captured next to the batch's other
    // kernels: ordinary launches (overlapping launches measured slower there)
    stage_mixed_kernel<P, false, true><<<ls.grid, ls.threads, ls.smem, st>>>(sp, ph);
    return cudaGetLastError();
}

// Cooperative launch: the blocks are resident together
template <typename... KArgs, typename... Args>
cudaError_t launch_coop(void (*kern)(KArgs...), const LaunchShape &ls, cudaStream_t st, Args... args)
{
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
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// two nodes per thread (IIP), hand-off kernel: resident blocks per SM of the
// build for at least M
template <int P, bool BATCH, bool FUSE, int M>
cudaError_t handoff_occupancy_p(int &per_sm)
{
    using L = Layout2<P>;
    auto kern = stage_handoff_kernel<P, BATCH, FUSE, M>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Sym64<P>::NT, L::bytes);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
    return e;
}

template <int P, bool BATCH, bool FUSE>
cudaError_t handoff_shape_p(long long K, LaunchShape &ls)
{
    using L = Layout2<P>;
    int occ4 = 0, occ5 = 0, dev = 0, sms = 0;
    cudaError_t e = handoff_occupancy_p<P, BATCH, FUSE, 4>(occ4);
    if constexpr (!FUSE && P != 6)
        if (e == cudaSuccess) e = handoff_occupancy_p<P, BATCH, FUSE, 5>(occ5);
    if (e != cudaSuccess) return e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long per_block = L::EG * L::NG;
    const HandoffGrid h = handoff_grid(sms, occ4, occ5, (K + per_block - 1) / per_block);
    ls.minb = h.minb;
    ls.grid = h.grid;
    ls.threads = Sym64<P>::NT;
    ls.smem = L::bytes;
    ls.elems_per_tile = L::EG;
    ls.theta = false;
    ls.variant = 2;
    ls.handoff = true;
    return cudaSuccess;
}

template <int P, bool BATCH, bool FUSE, int M>
cudaError_t handoff_launch_p(const LaunchShape &ls, const StageParams &sp, const Stage2 &x, const Phys<float> &ph,
                             cudaStream_t st)
{
    auto kern = stage_handoff_kernel<P, BATCH, FUSE, M>;
    if (!FUSE && !x.first) {
        if (!BATCH) return launch_pdl(kern, ls, st, sp, x, ph);
        kern<<<ls.grid, ls.threads, ls.smem, st>>>(sp, x, ph);
        return cudaGetLastError();
    }
    return launch_coop(kern, ls, st, sp, x, ph);
}

template <int P, bool BATCH, bool FUSE>
cudaError_t launch2_p(const LaunchShape &ls, const StageParams &sp, const Stage2 &x, const Phys<float> &ph, cudaStream_t st)
{
    if constexpr (!FUSE && P != 6)
        if (ls.minb == 5) return handoff_launch_p<P, BATCH, FUSE, 5>(ls, sp, x, ph, st);
    return handoff_launch_p<P, BATCH, FUSE, 4>(ls, sp, x, ph, st);
}

// ... and the kernel whose stages stand alone (single mesh)
template <int P, bool FUSE>
cudaError_t alone_shape_p(long long K, LaunchShape &ls)
{
    using S2 = Shape2<P>;
    using L = MixedLayout<P, false, S2::E>;
    auto kern = stage_mixed2_kernel<P, FUSE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(L::bytes));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, S2::NT, L::bytes);
    if (e != cudaSuccess) return e;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (per_sm < 1) {
        if (FUSE) return cudaErrorInvalidConfiguration;
        per_sm = 1;
    }
    const long long ntiles = (K + S2::E - 1) / S2::E, grid = static_cast<long long>(sms) * per_sm;
    ls.grid = static_cast<int>(ntiles < grid ? ntiles : grid);
    ls.threads = S2::NT;
    ls.smem = L::bytes;
    ls.elems_per_tile = S2::E;
    ls.theta = false;
    ls.variant = 2;
    ls.handoff = false;
    return cudaSuccess;
}

template <int P>
cudaError_t alone_launch_p(bool fused, const LaunchShape &ls, const StageParams &sp, const Phys<float> &ph, cudaStream_t st)
{
    if (!fused) return launch_pdl(stage_mixed2_kernel<P, false>, ls, st, sp, ph);
    return launch_coop(stage_mixed2_kernel<P, true>, ls, st, sp, ph);
}

// fused variant of the one-node shape: five stages per cooperative launch;
// the grid is the number of co-resident blocks (capped by the tile count)
template <int P, bool BATCH>
cudaError_t fused_shape_p(long long units, LaunchShape &ls)
{
    auto kern = stage_mixed_kernel<P, false, BATCH, true>;
    const int nt = Shape<P>::NT;
    const size_t smem = MixedLayout<P, false>::bytes;
    const long long ntiles = BATCH ? units : (units + Shape<P>::E - 1) / Shape<P>::E;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long grid = static_cast<long long>(sms) * per_sm;
    ls.grid = static_cast<int>(ntiles < grid ? ntiles : grid);
    ls.threads = nt;
    ls.smem = smem;
    ls.elems_per_tile = Shape<P>::E;
    ls.theta = false;
    ls.variant = 1;
    return cudaSuccess;
}

template <int P, bool BATCH>
cudaError_t fused_launch_p(const LaunchShape &ls, const StageParams &sp, const Phys<float> &ph, cudaStream_t st)
{
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
    return cudaLaunchKernelEx(&cfg, stage_mixed_kernel<P, false, BATCH, true>, sp, ph);
}

template <int P>
cudaError_t shadow_p(const double *K0, long long K, double gm1, float4 *S, float *Pr, cudaStream_t st)
{
    constexpr int Np = (P + 1) * (P + 2) / 2;
    const long long n = K * Np;
    const int threads = 256;
    make_shadow_kernel<P><<<static_cast<unsigned>((n + threads - 1) / threads), threads, 0, st>>>(K0, K, gm1, S, Pr);
    return cudaGetLastError();
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

cudaError_t stage_shape_mixed(int p, long long K, bool theta, LaunchShape &out)
{
#define C_(P) (theta ? shape_p<P, true>(K, out) : shape_p<P, false>(K, out))
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_stage_mixed(int p, const LaunchShape &ls, const StageParams &sp,
                               const Phys<float> &ph, cudaStream_t st)
{
#define C_(P) launch_p<P>(ls, sp, ph, st)
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t stage_shape_mixed_batch(int p, long long ntiles, LaunchShape &out)
{
#define C_(P) shape_batch_p<P>(ntiles, out)
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_stage_mixed_batch(int p, const LaunchShape &ls, const StageParams &sp,
                                     const Phys<float> &ph, cudaStream_t st)
{
#define C_(P) launch_batch_p<P>(ls, sp, ph, st)
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_dt_lambda_mixed_multi(const DtGroups &dgs, const BatchCase *cases, const Phys<float> &ph,
                                         float sig_fac, cudaStream_t st)
{
    if (dgs.blocks < 1) return cudaSuccess;
    dt_lambda_mixed_multi_kernel<1, 2, 3, 4, 5, 6><<<static_cast<unsigned>(dgs.blocks), 256, 0, st>>>(
        dgs, cases, ph, sig_fac);
    return cudaGetLastError();
}

template <int P>
cudaError_t dt_screen_p(const AuxMesh &m, const Phys<float> &ph, double gm1d, float sig_fac, float *lam,
                        unsigned *words, cudaStream_t st)
{
    const long long blocks = (m.K + Shape<P>::E - 1) / Shape<P>::E;
    dt_screen_kernel<P><<<static_cast<unsigned>(blocks), Shape<P>::NT, 0, st>>>(m.U, m.geo, m.conn, m.fmask, m.K, ph,
                                                                               gm1d, sig_fac, lam, words);
    return cudaGetLastError();
}

cudaError_t launch_dt_screen(const AuxMesh &m, const Phys<float> &ph, double gm1d, float sig_fac, float *lam,
                             unsigned *words, cudaStream_t st)
{
#define C_(P) dt_screen_p<P>(m, ph, gm1d, sig_fac, lam, words, st)
    DG_SWITCH_P(m.p, C_)
#undef C_
}

cudaError_t stage_shape_mixed2(int p, long long K, bool batch, bool fused, bool handoff, LaunchShape &out)
{
    // Measured, us for two steps of a single mesh, fastest of the shapes of each
    // side: p = 3, 76^2 quads 138 (stages alone) and 147 (hand-off), 110^2 231
    // and 245, 119^2 295 and 247; p = 5, 50^2 140 and 172, 70^2 235 and 274, 86^2
    // 329 and 341, 90^2 393 and 346.  Other degrees: hand-off ahead or neither
    // the fastest shape.
    const bool alone = !handoff || (p == 3 && K < 25000) || (p == 5 && K < 15000);
#define C_(P) (batch   ? (fused ? handoff_shape_p<P, true, true>(K, out) : handoff_shape_p<P, true, false>(K, out)) \
               : alone ? (fused ? alone_shape_p<P, true>(K, out) : alone_shape_p<P, false>(K, out))                 \
                       : (fused ? handoff_shape_p<P, false, true>(K, out) : handoff_shape_p<P, false, false>(K, out)))
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_stage_mixed2(int p, bool batch, bool fused, const LaunchShape &ls, const StageParams &sp,
                                const Stage2Args &a, const Phys<float> &ph, cudaStream_t st)
{
    if (!ls.handoff) {
#define C_(P) alone_launch_p<P>(fused, ls, sp, ph, st)
        DG_SWITCH_P(p, C_)
#undef C_
    }
    const Stage2 x{reinterpret_cast<const float4 *>(a.ops), a.nodes, a.fin, a.fout, a.rv, a.elem_case, a.first, a.next};
#define C_(P) (batch ? (fused ? launch2_p<P, true, true>(ls, sp, x, ph, st) : launch2_p<P, true, false>(ls, sp, x, ph, st)) \
                     : (fused ? launch2_p<P, false, true>(ls, sp, x, ph, st) : launch2_p<P, false, false>(ls, sp, x, ph, st)))
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t stage_shape_mixed_fused(int p, bool batch, long long units, LaunchShape &out)
{
#define C_(P) (batch ? fused_shape_p<P, true>(units, out) : fused_shape_p<P, false>(units, out))
    DG_SWITCH_P(p, C_)
#undef C_
}

cudaError_t launch_stage_mixed_fused(int p, bool batch, const LaunchShape &ls, const StageParams &sp,
                                     const Phys<float> &ph, cudaStream_t st)
{
#define C_(P) (batch ? fused_launch_p<P, true>(ls, sp, ph, st) : fused_launch_p<P, false>(ls, sp, ph, st))
    DG_SWITCH_P(p, C_)
#undef C_
}

int stage_tile_elems(int p)
{
    switch (p) {
    case 1: return Shape<1>::E;
    case 2: return Shape<2>::E;
    case 3: return Shape<3>::E;
    case 4: return Shape<4>::E;
    case 5: return Shape<5>::E;
    case 6: return Shape<6>::E;
    default: return 0;
    }
}

cudaError_t launch_make_shadow(int p, const double *K0, long long K, double gm1, float4 *S, float *Pr,
                               cudaStream_t st)
{
#define C_(P) shadow_p<P>(K0, K, gm1, S, Pr, st)
    DG_SWITCH_P(p, C_)
#undef C_
}

}  // namespace dg
