// hj_internal.h -- host/device shared declarations of the GB300 level-set
// library (not part of the public ABI; the ABI is include/hj.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include <vector>
#include <nvtx3/nvToolsExt.h>

namespace hj {

constexpr int kMaxDim = 4;

// WENO5 epsilon floor of FP32 kernels, in raw-difference units: 1e-99 (the
// FP64 floor) underflows in FP32; with 1e-18 the squared sums stay normal.
constexpr float kWenoFloorF32 = 1e-18f;

// Row and batch kernels take the dynamics as a template parameter. For the
// Hamiltonians whose |dHg/dp_d| depends on p (norm, air3D, rockets), the
// variant with Lax-Friedrichs dissipation local in p (HJ_ALPHA_BOX) is the
// dynamics id plus kDynBox; the other dynamics need no such variant (their
// box maximum is the maximum over every p).
constexpr int kDynBox = 8;
__host__ __device__ constexpr int dyn_base(int dyn) { return dyn & (kDynBox - 1); }
__host__ __device__ constexpr bool dyn_is_box(int dyn) { return (dyn & kDynBox) != 0; }
__host__ __device__ inline bool box_differs(int dyn) {
    return dyn == 4 /* HJ_DYN_NORM */ || dyn == 2 /* HJ_DYN_AIR3D */ || dyn == 7 /* HJ_DYN_ROCKETS */;
}

// A named NVTX range for the lifetime of the object: solves, steps, batched
// graph replays and server admissions show up as ranges in a profiler's
// timeline (header-only NVTX: inert unless a tool is attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// Rows of at most this many threads' worth of nodes (n0 + 1 <= 1024 in FP32,
// 512 in FP64) are the row kernel's; a pinned launch shape may ask for up to
// this many nodes a block.
inline int rows_max_nodes(int dtype_is_f64) { return dtype_is_f64 ? 512 : 1024; }
// Largest block of the row-tiled kernels, and the share its node threads may
// take (two nodes a thread; at least one warp is left for the tile's edges).
// FP64 blocks of 384 threads may use 168 registers a thread; what FP32 may use
// is RowsBounds (rows_kernel.cuh).
constexpr int kRowsThreadsF32 = 640, kRowsThreadsF64 = 384;
inline int rows_max_threads(int dtype_is_f64) { return dtype_is_f64 ? kRowsThreadsF64 : kRowsThreadsF32; }
inline int rows_max_node_threads(int dtype_is_f64) { return dtype_is_f64 ? 256 : 512; }

// Grid as the kernels see it. Spacing and its inverse are computed once on
// the host from the hj_grid (periodic: (hi-lo)/n, else (hi-lo)/(n-1)).
struct GridDev {
    int ndim;
    int n[kMaxDim];
    long long stride[kMaxDim];
    long long total;
    double lo[kMaxDim];
    double dx[kMaxDim];
    double inv_dx[kMaxDim];
    unsigned periodic_mask;
    int extrap;  // HJ_EXTRAP_*
};

// What one launch of the fused stage kernel computes at every node:
//   w   = U + dt * ydot(U)            (mode kStage*)  or  w = ydot(U)  (mode kTerm)
//   out = cv * Vn + cu * w            (cv == 0: out = w)
//   out = min(out, Vn)                (minv_after: BRT "min(V, V_prev)" rule)
enum StageMode { kTerm = 0, kStage = 1 };

struct StageParams {
    GridDev g;
    int dynamics;
    double params[8];
    int brt_min0;     // clamp ydot at zero (BRT min(0, H))
    int minv_after;   // out = min(out, Vn)
    int mode;         // StageMode
    int scheme;       // HJ_ENO1/2/3 or HJ_WENO5 (row kernel); the one-node kernel takes it as an argument
    double dt;
    double cv, cu;    // stage combination coefficients
    const void* u;    // stencil input
    const void* vn;   // V^n (read at the node only); may be null when cv == 0 and !minv_after
    void* out;
    const double* trig_d;  // cos, sin of the dimension-2 coordinate: [cos(0..n2-1), sin(0..n2-1)]
    const float* trig_f;
    double weno_floor[kMaxDim];   // additive floor of the WENO5 epsilon per dimension, in raw-difference units
    double weno_floor12[kMaxDim]; // 12 times that (the FP64 smoothness sums are scaled by 12)
    double half_inv_dx[kMaxDim];  // 1 / (2 dx): raw differences to (p- + p+)/2 and (p+ - p-)/2
    double half_inv_dx6[kMaxDim]; // 1 / (12 dx): the same from six times the raw differences (WENO5)
    int alpha_global;             // dissipation alpha_d = alpha_g[d] (global LF) instead of alpha_d(x)
    double alpha_g[kMaxDim];
    int alpha_box;                // dissipation alpha_d = max |dHg/dp_d| over the node's box of gradients
    // FP32 copies of the scalars above, so that FP32 kernels do no FP64 arithmetic
    float lo_f[kMaxDim], dx_f[kMaxDim], half_inv_dx_f[kMaxDim], half_inv_dx6_f[kMaxDim];
    float alpha_g_f[kMaxDim];
    float params_f[8];
    float dt_f, cv_f, cu_f;
    int has_vn;            // the stage reads Vn (cv != 0 or minv_after)
};

// Whether a row-kernel launch takes a variant with dissipation local in p
// (rows_f32_box.cu, rows_f64_box.cu).
inline bool rows_box_variant(const StageParams& p) { return p.alpha_box && box_differs(p.dynamics); }

// Fills the FP32 copies and has_vn from the FP64 fields (call before launching).
inline StageParams finalize(StageParams p) {
    for (int d = 0; d < kMaxDim; ++d) {
        p.lo_f[d] = (float)p.g.lo[d];
        p.dx_f[d] = (float)p.g.dx[d];
        p.half_inv_dx[d] = 0.5 * p.g.inv_dx[d];
        p.half_inv_dx6[d] = p.half_inv_dx[d] / 6.0;
        p.half_inv_dx6_f[d] = (float)p.half_inv_dx6[d];
        p.half_inv_dx_f[d] = (float)p.half_inv_dx[d];
        p.alpha_g_f[d] = (float)p.alpha_g[d];
        p.weno_floor12[d] = 12.0 * p.weno_floor[d];
    }
    for (int k = 0; k < 8; ++k) p.params_f[k] = (float)p.params[k];
    p.dt_f = (float)p.dt;
    p.cv_f = (float)p.cv;
    p.cu_f = (float)p.cu;
    p.has_vn = (p.mode == kStage) && (p.cv != 0.0 || p.minv_after);
    return p;
}

// What the row kernels store per node, by launch (a template parameter, so
// that no per-node branch remains): the stage term alone, the first RK
// stage (no V^n), or a combination with V^n (stages 2 and 3).
enum StageKind { kKindTerm = 0, kKindFirst = 1, kKindCombine = 2 };
inline int stage_kind(const StageParams& p) {  // p finalized
    return p.mode == kTerm ? kKindTerm : (p.has_vn ? kKindCombine : kKindFirst);
}

struct UpwindParams {
    GridDev g;
    int dim;
    const void* u;
    void* pm;
    void* pp;
    double weno_floor;  // FP64: times 12 (see StageParams)
    double dx;
    double inv_6dx;     // 1 / (6 dx)
};

// Launch configuration of the row-tiled stage kernel (rows_kernel.cuh).
constexpr int kRowsMaxTy = 8;    // rows of a tile
constexpr int kRowsMaxSx = 124;  // nodes along dimension 0 of a tile (at most four edge warps)
constexpr int kRowsPitch = 30;  // values of one column of a shared buffer (rows_kernel.cuh says which)
struct RowsCfg {
    int sx;       // nodes along dimension 0 of a tile
    int ty;       // node rows per tile, at most kRowsMaxTy
    int nt;       // threads per block (1-D), a multiple of 32
    int tz;       // planes per chunk along the streamed (last) dimension
    int nchunks;  // chunks along the streamed dimension
    int tiles;    // ceil(n0 / sx) * ceil(n1 / ty)
    int plane;    // 1: the kernel of one interface a thread (2-D grids, plane_kernel.cuh)
};
// threads of the node warps (two rows each)
__host__ __device__ inline int rows_node_threads(int sx, int ty) { return (sx * ((ty + 1) / 2) + 31) / 32 * 32; }
__host__ __device__ inline int rows_buf_elems(int sx) { return (sx + 6) * kRowsPitch; }
// Dynamic shared memory of a block (element size es).
inline size_t rows_smem(int sx, size_t es) { return 2 * es * (size_t)rows_buf_elems(sx); }
// The widest segment (nodes along dimension 0, as equal as possible) with which
// ty rows of n0 nodes fit node_threads node threads.
inline int rows_segment(int n0, int ty, int node_threads) {
    const int fit = node_threads / ((ty + 1) / 2);
    const int most = fit < kRowsMaxSx ? fit : kRowsMaxSx;
    const int nseg = (n0 + most - 1) / most;
    return (n0 + nseg - 1) / nseg;
}
// Edge threads beside a tile's node threads (the tile's last interfaces, one per
// two columns and per row pair, and the halos). A block waits for its edge warps
// in every plane: with one column of halo a thread the FP32 stage of 101^3 took
// 15.6 us, with two (and half the threads) 21; in FP64, whose planes take longer,
// 240 and 231 us (now 14.4 and 206).
__host__ __device__ constexpr int rows_edge_cols(bool f64) { return f64 ? 2 : 1; }
inline int rows_edge_threads(int sx, bool f64) {
    const int need = f64 ? (sx + 1) / 2 + 4 : sx + 4;
    return (need + 31) / 32 * 32;
}
inline RowsCfg make_rows_cfg(const GridDev& G, int sx, int ty, int tz, int nt) {
    RowsCfg c;
    c.sx = sx;
    c.ty = ty;
    c.nt = nt;
    c.tiles = ((G.n[0] + sx - 1) / sx) * ((G.n[1] + ty - 1) / ty);
    const int ns = G.ndim >= 3 ? G.n[G.ndim - 1] : 1;
    c.tz = G.ndim >= 3 ? tz : 1;
    c.nchunks = (ns + c.tz - 1) / c.tz;
    c.plane = 0;
    return c;
}

// The row kernel's launch shapes for this stage, the cheapest by a cost model first
// (hj_api.cu; P finalized or not: its grid, dynamics and scheme count).
std::vector<RowsCfg> rows_ranked(const StageParams& P, int dtype, int sm_count, bool quick);

// The plane kernel's block: threads for the items of a tile (FP32: pairs of
// interfaces), at most kPlaneThreads; and its shared memory.
constexpr int kPlaneThreads = 384;
inline RowsCfg make_plane_cfg(const GridDev& G, int sx, int ty, int dtype_is_f64) {
    const int w = dtype_is_f64 ? 1 : 2;
    const int items = (sx + 1) * ((ty + w - 1) / w) + sx * ((ty + w) / w);
    const int nt = (items + 31) / 32 * 32;
    RowsCfg c = make_rows_cfg(G, sx, ty, 1, nt < kPlaneThreads ? nt : kPlaneThreads);
    c.plane = 1;
    return c;
}
inline size_t plane_smem(int sx, int ty, size_t es) {
    return es * ((size_t)(ty + 8) * (sx + 6) + 2 * (size_t)(ty + 1) * (sx + 1) + 2 * (size_t)(ty + 2) * sx);
}

// Launchers (one translation unit per element type). Return the launch error.
cudaError_t launch_stage_f64(const StageParams& p, int scheme, cudaStream_t s);
cudaError_t launch_stage_f32(const StageParams& p, int scheme, cudaStream_t s);
cudaError_t launch_upwind_f64(const UpwindParams& p, int scheme, cudaStream_t s);
cudaError_t launch_upwind_f32(const UpwindParams& p, int scheme, cudaStream_t s);

// Row-tiled stage kernel (every scheme): defined for D = 2 (double integrator, norm,
// advection, rotation), D = 3 (air3D, rockets, norm, advection, rotation), D = 4 (Dubins4D).
bool rows_supported(int ndim, int dynamics);
cudaError_t launch_rows_f64(const StageParams& p, const RowsCfg& c, cudaStream_t s);
cudaError_t launch_rows_f32(const StageParams& p, const RowsCfg& c, cudaStream_t s);
// resident blocks per SM of a configuration (0 if it cannot launch)
int rows_blocks_per_sm_f64(const StageParams& p, const RowsCfg& c);
int rows_blocks_per_sm_f32(const StageParams& p, const RowsCfg& c);

// ---------------------------------------------------------------------------
// Batched solves: many instances advanced together by one launch per stage
// over a list of tiles (batch.cuh).
// ---------------------------------------------------------------------------
struct BatchTile {
    int inst;      // instance index
    int tile;      // tile of the instance's planes: segment + segments * row tile
    int i2;        // dimension-2 index (4-D instances)
    int chunk;     // chunk along the streamed dimension
};

struct BatchInst {
    StageParams P;            // grid, dynamics, parameters (FP64 + FP32), angle tables, WENO floor
    int sx, ty, tz;           // tile shape of this instance
    int steps_total;          // RK3 steps of the whole solve
    int k;                    // steps completed (advanced on the device)
    double dt;                // dt of the current step
    float dt_f;
    int brt;                  // HJ_BRT_*
    void* V;                  // value function (in place)
    void* V1;                 // stage buffers
    void* V2;
    void* slice_out;          // stage 3 of the current step also writes here, or null
    double dt_full;           // dt of every step that does not end a slice: min(max_step, cfl/stepBoundInv)
    const long long* ends;    // distinct positive step counts at which slices are taken, ascending
    const int* end_slice;     // slice index written at each of those
    const double* end_dt;     // dt of the step that completes each of those (clipped to the slice time)
    int n_ends;
    int cursor;               // next entry of ends not yet scheduled
    void* out;                // slice outputs: n_slices x nodes elements
    long long nodes;
    int elem;                 // element size in bytes
};

cudaError_t launch_batch_stage_f32(const BatchTile* tiles, int ntiles, const BatchInst* insts, int stage, int ndim,
                                   int dynamics, int scheme, int threads, size_t smem, cudaStream_t s);
cudaError_t launch_batch_stage_f64(const BatchTile* tiles, int ntiles, const BatchInst* insts, int stage, int ndim,
                                   int dynamics, int scheme, int threads, size_t smem, cudaStream_t s);
// Advances the instances of these tiles.
cudaError_t launch_batch_advance(const BatchTile* tiles, int ntiles, BatchInst* insts, cudaStream_t s);

// max over nodes of sum_d alpha_d(x)/dx_d, as the FP64 bit pattern, atomically
// max-ed into *acc (which the caller zeroes first).
cudaError_t launch_step_bound(const GridDev& g, int dynamics, const double* params, const double* trig_d,
                              unsigned long long* acc, int per_dim, cudaStream_t s);
// Sets *flag to 1 if any of the n elements is NaN or +-Inf.
cudaError_t launch_nonfinite_f64(const double* v, long long n, int* flag, cudaStream_t s);
cudaError_t launch_nonfinite_f32(const float* v, long long n, int* flag, cudaStream_t s);

}  // namespace hj
