// launch.h -- host-side launch wrappers for the library's kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "dg_device.cuh"

namespace dg {

struct StageParams;
struct BatchCase;

struct LaunchShape {
    bool theta = false;      // kernel variant with the theta terms of the IP flux
    int variant = 1;         // mixed IIP kernel: 1 node per thread (1), 2 nodes per thread (2),
                             // tensor-core warp tiles (3)
    bool overint = false;    // FP64 kernel: volume flux integrated with a cubature rule
    int grid = 0;
    int threads = 0;
    size_t smem = 0;
    int elems_per_tile = 0;
    bool phases = false;     // FP64: the three-phase kernel (arrays between its phases, cooperative launch)
    bool handoff = false;    // two nodes per thread: the kernel that hands volume parts from stage to stage
    int minb = 0;            // ... and which of its builds (handoff_grid.h)
};

// Launch `kern` with programmatic stream serialization: its blocks may be
// scheduled while the previous kernel of the stream drains; the kernel waits
// for that kernel (pdl_wait_then_release) before touching the state.
template <typename... Args>
inline cudaError_t launch_pdl(void (*kern)(Args...), const LaunchShape &ls, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ls.grid);
    cfg.blockDim = dim3(ls.threads);
    cfg.dynamicSmemBytes = ls.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}


// Launch configuration of the fused stage kernel for degree p and K elements
// on the current device (persistent grid: SMs x resident CTAs, capped by tiles).
// FP64: over-integrated, in three phases, or the kernel that needs neither
// memory of its own nor a cooperative launch
cudaError_t stage_shape_fp64(int p, long long K, bool theta, LaunchShape &out, bool overint, bool phases);
cudaError_t stage_shape_mixed(int p, long long K, bool theta, LaunchShape &out);
// what the three-phase FP64 stage kernel reads and keeps besides StageParams:
// the symmetric operator tables of build_sym64_tables, every face once as
// (element, neighbour, face | its face << 2 | boundary type << 4, 0) with the
// interior ones first, and its arrays (fluxes [K][Np][8], face terms
// [K][3 Nfp][4], with theta terms [K][3 Nfp][8])
struct Stage64Args {
    const double *ops;
    const int *nodes;
    const int4 *faces;
    int nfaces;
    double *flux, *dh, *th;
};
cudaError_t launch_stage_fp64(int p, const LaunchShape &ls, const StageParams &sp, const Stage64Args &a,
                              const Phys<double> &ph, cudaStream_t st);
// false if the operators are not symmetric under r <-> s; theta: with the rows
// of the theta terms (zero otherwise)
struct RefOps;
bool build_sym64_tables(const RefOps &o, bool theta, std::vector<double> &tab, std::vector<int> &nodes);
// broken gradient [K][4][Np] x 2 in FP64, from those tables or the plain rows
// (both on the device), on `grid` blocks (asked for once per mesh: the query
// costs as much as the launch)
struct Grad64Args {
    int grid;
    const double *U, *geo, *ops;
    const int *nodes;
    const double *Dr, *Ds;
    long long K;
    double *gx, *gy;
};
cudaError_t grad64_grid(int p, long long K, int &grid);
cudaError_t launch_grad64(int p, const Grad64Args &a, cudaStream_t st);
cudaError_t launch_stage_mixed(int p, const LaunchShape &ls, const StageParams &sp,
                               const Phys<float> &ph, cudaStream_t st);
// batch variant of the mixed kernel (IIP): grid for `ntiles` tiles of a tile table
cudaError_t stage_shape_mixed_batch(int p, long long ntiles, LaunchShape &out);
cudaError_t launch_stage_mixed_batch(int p, const LaunchShape &ls, const StageParams &sp,
                                     const Phys<float> &ph, cudaStream_t st);
// Lambda_K of every degree group of a batch in one launch (one block per tile)
cudaError_t launch_dt_lambda_mixed_multi(const DtGroups &dgs, const BatchCase *cases, const Phys<float> &ph,
                                         float sig_fac, cudaStream_t st);
// The mixed IIP kernel with two nodes per thread for K elements: one stage, or
// the five of a step (fused).  The hand-off kernel (LaunchShape::handoff) has
// the tables of build_sym32_tables and hands a record per face node (pressure,
// viscous normal flux) [K][3 Nfp] and the divergence [K][Np] from stage to
// stage; a launch with `first` (and a fused one) is cooperative.  A single
// mesh without memory for those, or on a stream that cannot hold its grid,
// takes the kernel whose stages stand alone (handoff = false), and so do
// small meshes at some degrees.
struct Stage2Args {
    const float *ops;
    const int *nodes;
    const float4 *fin;         // trace records this stage reads (first: written to fout, then swapped)
    float4 *fout;              // ... and the next one's
    float4 *rv;
    const int *elem_case;      // batch: case of every element
    int first, next;           // a step's first stage (or a residual); not its last (residual: 1, 0)
};
// those of stage s of a step (-1: a residual; 0 also for a fused step) with the
// two flux buffers of n records each at fd: the first stage fills the first
// buffer, and the buffers change roles from stage to stage
inline Stage2Args stage2_args(const float *ops, const int *nodes, float4 *fd, float4 *rv, const int *elem_case, size_t n, int s)
{
    const bool second = s <= 0 || (s & 1);
    return {ops, nodes, second ? fd + n : fd, second ? fd : fd + n, rv, elem_case, s <= 0 ? 1 : 0, s >= 0 && s < 4 ? 1 : 0};
}
cudaError_t stage_shape_mixed2(int p, long long K, bool batch, bool fused, bool handoff, LaunchShape &out);
cudaError_t launch_stage_mixed2(int p, bool batch, bool fused, const LaunchShape &ls, const StageParams &sp,
                                const Stage2Args &a, const Phys<float> &ph, cudaStream_t st);
// FP32 rows (each twice) from the FP64 tables, and per thread its two nodes
// and up to two face slots of each
void build_sym32_tables(const RefOps &o, const std::vector<double> &tab, const std::vector<int> &nodes,
                        std::vector<float> &tab32, std::vector<int> &slots);
// every face of K elements once, as Stage64Args has them
void unique_faces(const int4 *conn, long long K, std::vector<int4> &faces);
// five stages per cooperative launch (mixed IIP, one node per thread): grid of
// co-resident blocks for `units` (K, or the tile count of a batch table)
cudaError_t stage_shape_mixed_fused(int p, bool batch, long long units, LaunchShape &out);
cudaError_t launch_stage_mixed_fused(int p, bool batch, const LaunchShape &ls, const StageParams &sp,
                                     const Phys<float> &ph, cudaStream_t st);
// elements per tile of the mixed kernel for degree p
int stage_tile_elems(int p);
// the tensor-core mixed IIP kernel (p = 1..6): warp tiles of 2 elements;
// its `ops` is the operator table of build_tc_fragments
bool stage_tc_supported(int p);
// elements per warp tile of the tensor-core kernel (any p)
int stage_tile_elems_tc();
// units = K elements (single mesh) or the tile count of a batch tile table;
// fused: five stages per cooperative launch with grid barriers
// theta: the SIP / NIPG variant (single mesh, stage-wise launches only)
cudaError_t stage_shape_tc(int p, long long units, bool batch, bool fused, LaunchShape &out, bool theta = false);
// the fused batch body of every degree group in one cooperative launch:
// blocks that fit the GPU at once and the shared memory per block (the
// largest group's layout), then the launch with nblk[g] blocks for group g
cudaError_t stage_tc_multi_capacity(const int *ps, int ngroups, int &blocks, size_t &smem);
cudaError_t launch_stage_tc_multi(int ngroups, const int *ps, const StageParams *sps, const unsigned *nblk,
                                  size_t smem, const Phys<float> &ph, cudaStream_t st);
cudaError_t launch_stage_tc(int p, bool batch, bool fused, const LaunchShape &ls, const StageParams &sp,
                            const Phys<float> &ph, cudaStream_t st);
// Dr, Ds [Np][Np], LIFT [Np][NF], Wr, Ws [Np][Np] (FP64, row-major) -> the kernel's
// operator table (TF32 hi / lo fragments of 16-row tiles, then (Dr, Ds) as
// FP32 pairs [Np][Np])
void build_tc_fragments(int Np, int NF, const double *Dr, const double *Ds, const double *LIFT,
                        const double *Wr, const double *Ws, std::vector<float> &out);
// FP32 copy [K][Np] float4 and FP64-recovered pressure [K][NpP] of a state
cudaError_t launch_make_shadow(int p, const double *K0, long long K, double gm1, float4 *S,
                               float *Pr, cudaStream_t st);
// padded pressure row length: Np rounded up to a multiple of 4
inline int pressure_row(int p) { return (((p + 1) * (p + 2) / 2) + 3) & ~3; }

struct BatchCase;

struct AuxMesh {
    const double *U;          // [K][4][Np]
    const int *elem_case = nullptr;         // batch: case of every element (mu, v_b)
    const BatchCase *cases = nullptr;
    const double *geo;        // double[16] per element
    const int4 *conn;
    const double *Dr, *Ds;    // Np*Np
    const int *fmask;         // 3*Nfp
    long long K;
    int p;
};

// max_K Lambda_K of Eq. rayleigh_bound in FP64: an FP32 screen of every
// element into lam[K], then FP64 on the elements that can hold the maximum,
// whose value goes to *out (NaN if one is not finite).  sig_fac = C1
// (1+theta)^2 (d+1) of Eq. penalty_final; words: 8 words, zero between calls.
cudaError_t launch_dt_screen(const AuxMesh &m, const Phys<float> &ph, double gm1d, float sig_fac, float *lam,
                             unsigned *words, cudaStream_t st);
cudaError_t launch_dt_confirm(const AuxMesh &m, const Phys<double> &ph, double sig_fac, const float *lam,
                              unsigned *words, double *out, cudaStream_t st);

// per-wall-face force/moment partials and their sum (fixed order) into out[3],
// one launch; *ticket counts finished blocks, zero before and after it
cudaError_t launch_wall_forces(const AuxMesh &m, const Phys<double> &ph, const int2 *faces, const double *face_xy,
                               const double *wface, int nwall, double xc, double yc, double *partial,
                               unsigned *ticket, double *out, cudaStream_t st);

// batch: one block per case, max of lam over the case's element range
// [seg[2i], seg[2i+1]) -> cases[i].lam and dt = cfl / lam, or fixed[i] when
// fixed is not null (0 and bad = 1 if the bound is not finite); then the
// case's Newmark step with its lagged lift: sets v_b, advances t
cudaError_t launch_batch_dt_newmark(const double *lam, const long long *seg, BatchCase *cases, int ncases,
                                    double cfl, const double *fixed, cudaStream_t st);
// batch: the wall faces of every degree group in one launch (group g's faces
// numbered from g.base); partial[w] = (Fx, Fy, Mz) of face w, moment about 0
struct WallGroup {
    AuxMesh m;
    const int2 *faces;        // (element, face) of the group's wall faces
    const double *face_xy;    // their face nodes' coordinates, [nwall][Nfp][2]
    const double *wface;      // LGL weights [Nfp]
    int base, nwall;
};
struct WallGroups {
    WallGroup g[8];
    int n = 0, total = 0;
};
cudaError_t launch_batch_wall_forces(const WallGroups &wg, const Phys<double> &ph, double *partial,
                                     cudaStream_t st);
// batch: one block per case, sum of the wall-face partials [wseg[2i], wseg[2i+1]) -> Fx, Fy, Mz, and
// with hist: (t, dt, y, y', v_b, Fx, Fy, lam) of every case at row *counter, then ++*counter
// (ticket: a zeroed counter of finished blocks)
cudaError_t launch_batch_forces_record(const double *partial, const int *wseg, BatchCase *cases, int ncases,
                                       double *hist, int cap, int *counter, unsigned *ticket, cudaStream_t st);

// *flag = 1 if any of x[0..n) is not finite (flag must be zeroed first)
cudaError_t launch_nonfinite(const double *x, long long n, int *flag, cudaStream_t st);

// viscous source of the advected isentropic vortex (dg_set_source kind 2)
struct VortexSource {
    double beta, x0, y0, L, u0, v0;   // strength, centre at t = 0, period, advection velocity
    double mu, Pr;
    double invL, f0, c2, invPr;       // 1/L, beta/(2 pi), beta^2/(2 pi^2), 1/Pr
};
// broken gradient of every element (dg_broken_gradient), impl 1: split TF32
// on tcgen05 with the tiles staged by TMA
struct GradTc05Args {
    const double *U;            // [K][4][Np] FP64 state (device)
    const double *Dr, *Ds;      // Np x Np operators (host, for the split image)
    const double *geo;          // double[16] per element
    long long K;
    double *gx, *gy;            // [K][4][Np] outputs (device)
    float *bimg;                // device buffer of grad_tc05_bimg_floats(p) floats
    bool upload_ops;            // (re)write the split operator image into bimg first
    int *err;                   // set to 1 if a bounded wait gave up
    unsigned wait_limit;
};
size_t grad_tc05_bimg_floats(int p);
cudaError_t launch_grad_tc05(int p, const GradTc05Args &a, cudaStream_t st);

struct VortexCentres {
    double xc[5], yc[5];
    int ns;
};
// S[s][K][4][Np] at the times t[s], s < ns <= 5, from node coordinates
// xy = (x[K*Np], y[K*Np]) in one launch; fp64: double arithmetic, else float
// after the offsets
cudaError_t launch_vortex_source(bool fp64, const double *xy, long long nn, int Np, const VortexSource &v,
                                 const double *t, int ns, double *S, cudaStream_t st);

}  // namespace dg
