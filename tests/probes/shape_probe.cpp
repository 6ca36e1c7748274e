// Test probe: one launch of the stage kernels with a chosen launch shape (which
// kernel, segment, rows, planes), so that tests can hold shapes against each
// other that the public interface leaves to the library. Linked with libhj.so.
#include <cstring>

#include "../../include/hj.h"
#include "hj_internal.h"

using namespace hj;

namespace {
StageParams params(const hj_grid* grid, const hj_method* m, int dtype) {
    StageParams P;
    std::memset(&P, 0, sizeof P);
    GridDev& G = P.g;
    G.ndim = grid->ndim;
    long long stride = 1;
    for (int d = 0; d < 4; ++d) {
        const bool in = d < grid->ndim, periodic = in && ((grid->periodic_mask >> d) & 1u);
        G.n[d] = in ? (int)grid->n[d] : 1;
        G.stride[d] = stride;
        stride *= G.n[d];
        G.lo[d] = in ? grid->lo[d] : 0.0;
        G.dx[d] = in ? (grid->hi[d] - grid->lo[d]) / (double)(periodic ? G.n[d] : G.n[d] - 1) : 1.0;
        G.inv_dx[d] = 1.0 / G.dx[d];
    }
    G.total = stride;
    G.periodic_mask = grid->periodic_mask;
    G.extrap = m->extrap;
    P.dynamics = m->dynamics;
    P.scheme = m->scheme;
    for (int k = 0; k < 8; ++k) P.params[k] = m->params[k];
    P.brt_min0 = m->brt == HJ_BRT_MIN0;
    P.alpha_box = m->alpha_mode == HJ_ALPHA_BOX;
    for (int d = 0; d < 4; ++d)
        P.weno_floor[d] = dtype == HJ_F32 ? (double)kWenoFloorF32 : 1e-99 * G.dx[d] * G.dx[d];
    return P;
}
int blocks_per_sm(const StageParams& Q, const RowsCfg& c, bool f64) {
    return f64 ? rows_blocks_per_sm_f64(Q, c) : rows_blocks_per_sm_f32(Q, c);
}
}  // namespace

extern "C" int shape_bps(const hj_grid* grid, const hj_method* m, int dtype, int sx, int ty) {
    const StageParams P = params(grid, m, dtype);
    const bool f64 = dtype == HJ_F64;
    return blocks_per_sm(finalize(P), make_rows_cfg(P.g, sx, ty, 1, rows_node_threads(sx, ty) + rows_edge_threads(sx, f64)), f64);
}

// stage 0: the term; 1..3: a stage of the RK3 step. plane: plane_kernel (2-D),
// else the row kernel. sx, ty, tz: nodes of a segment, rows, planes of a chunk.
// trig: cos and sin of the dimension-2 coordinate in both precisions, or null.
// Returns a CUDA error, or -1 where the kernel has no such shape.
extern "C" int shape_stage(const hj_grid* grid, const hj_method* m, int dtype, int plane, int sx, int ty, int tz,
                           int stage, const void* u, const void* vn, void* out, const double* trig_d,
                           const float* trig_f, double dt, void* stream) {
    StageParams P = params(grid, m, dtype);
    const GridDev& G = P.g;
    P.trig_d = trig_d;
    P.trig_f = trig_f;
    P.mode = stage == 0 ? kTerm : kStage;
    P.dt = dt;
    P.u = u;
    P.vn = stage > 1 ? vn : nullptr;
    P.out = out;
    P.cv = stage == 2 ? 0.75 : stage == 3 ? 1.0 / 3.0 : 0.0;
    P.cu = stage == 2 ? 0.25 : stage == 3 ? 2.0 / 3.0 : 1.0;
    P.minv_after = stage == 3 && m->brt == HJ_BRT_MINV;
    const bool f64 = dtype == HJ_F64;
    if (sx < 1 || ty < 1 || tz < 1 || sx > G.n[0] || ty > G.n[1]) return -1;
    RowsCfg c;
    if (plane) {
        if (G.ndim != 2 || sx > 64 || ty > 64) return -1;
        c = make_plane_cfg(G, sx, ty, f64);
    } else {
        if (sx > kRowsMaxSx || ty > kRowsMaxTy || rows_node_threads(sx, ty) > rows_max_node_threads(f64)) return -1;
        c = make_rows_cfg(G, sx, ty, tz, rows_node_threads(sx, ty) + rows_edge_threads(sx, f64));
    }
    const StageParams Q = finalize(P);
    if (blocks_per_sm(Q, c, f64) <= 0) return -1;
    return (int)(f64 ? launch_rows_f64(Q, c, static_cast<cudaStream_t>(stream))
                     : launch_rows_f32(Q, c, static_cast<cudaStream_t>(stream)));
}
