// plane_kernel.cuh -- the fused RK stage kernel on 2-D grids that leave the chip
// mostly idle: one interface per thread, then one node per thread.
//
// An FP64 2-D stage of 101^2 nodes is one short chain of dependent operations per
// thread, and with two rows a thread (rows_kernel.cuh) a chain of 11.4 us: one
// warp's FP64 instructions follow each other in 64 cycles each on its quarter of
// the SM, while the other quarters have no warp. Here the interfaces along both
// dimensions of a small tile are dealt out to the threads of a block (FP32: two
// rows' or two gaps' at a time, packed as in the row kernel), both halves go
// through shared memory, and each node is updated by a thread of its own: 6.2 us
// (5 x 12 nodes a block, two blocks an SM), 44 us instead of 50 on 511^2; a whole
// solve of 101^2 then took 2592 us, with the smoothness sums in integers 2438, and
// with indices and cells ready before the wait for the kernel in front 2275, with
// the next kernel let in only after that wait 1800. FP32, whose stage is launch latency up to 301^2 (2.5 to 2.8 us with either kernel),
// keeps the row kernel where that is faster: the launch-shape tuner times both.
// Both evaluate an interface and a node with the same functions, so that the
// results are the same bits.
#pragma once

#include "rows_kernel.cuh"

namespace hj {

// Shared memory: the tile with three halo cells on each side (and two rows
// that only the second lane of a last pair reads), then p+ and p- of the
// interfaces along dimension 0 (TY + 1 rows of SX + 1) and along dimension 1
// (TY + 2 gaps of SX).
template <typename T, int DYN, int SCHEME, int KIND>
__global__ void __launch_bounds__(kPlaneThreads, 1) plane_kernel(const StageParams P, const RowsCfg C) {
    constexpr int kW = sizeof(T) == 4 ? 2 : 1;  // interfaces of an item
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const StageRun<T> R = stage_run<T>(P);
    const GridDev& g = P.g;
    const int nx = g.n[0], ny = g.n[1];
    const bool per0 = g.periodic_mask & 1u, per1 = (g.periodic_mask >> 1) & 1u;
    const int nseg = (nx + C.sx - 1) / C.sx;
    const int row_tile = blockIdx.x / nseg, seg = blockIdx.x - row_tile * nseg;
    const int x0 = seg * C.sx, sx = min(C.sx, nx - x0);
    const int y0 = row_tile * C.ty, rv = min(C.ty, ny - y0);
    const int t = threadIdx.x;
    const int W = C.sx + 6;
    T* const V = reinterpret_cast<T*>(smem_raw);
    T* const xp = V + (C.ty + 8) * W;
    T* const xm = xp + (C.ty + 1) * (C.sx + 1);
    T* const yp = xm + (C.ty + 1) * (C.sx + 1);
    T* const ym = yp + (C.ty + 2) * C.sx;
    const T fl0 = SP<T>::floor(P, 0), fl1 = SP<T>::floor(P, 1);

    // One cell of the tile: where it goes, and its source or, of a ghost cell, the
    // two outermost values and its distance from them.
    struct Cell {
        int to, a, b, m;  // to < 0: none; b < 0: no ghost cell
    };
    auto make_cell = [&](int c) {
        Cell q{-1, 0, -1, 0};
        const int r = c / (sx + 6) - 3, x = c - (r + 3) * (sx + 6) - 3;
        const bool in_x = x >= 0 && x < sx, in_y = r >= 0 && r < rv;
        if (r >= rv + 3 || !(in_x || in_y)) return q;
        q.to = (r + 3) * W + x + 3;
        const int n = in_y ? nx : ny, s = in_y ? 1 : nx, base = in_y ? (y0 + r) * nx : x0 + x;
        int i = in_y ? x0 + x : y0 + r;
        if (in_y ? per0 : per1) i += i < 0 ? n : i >= n ? -n : 0;
        if (i >= 0 && i < n) {
            q.a = base + i * s;
        } else {
            q.a = base + (i < 0 ? 0 : n - 1) * s;
            q.b = base + (i < 0 ? 1 : n - 2) * s;
            q.m = i < 0 ? -i : i - (n - 1);
        }
        return q;
    };
    // One item of interfaces: its first row or gap, its column, and where its values begin.
    const int n_x = (sx + 1) * ((rv + kW - 1) / kW), n_y = sx * ((rv + kW) / kW);
    struct Item {
        bool along_x;
        int from, to;
    };
    auto make_item = [&](int i) {
        Item q;
        q.along_x = i < n_x;
        const int k = q.along_x ? i : i - n_x, width = q.along_x ? sx + 1 : sx;
        const int line = k / width, x = k - line * width;
        q.from = q.along_x ? (line * kW + 3) * W + x : line * kW * W + x + 3;
        q.to = line * kW * (q.along_x ? C.sx + 1 : C.sx) + x;
        return q;
    };

    // A stage is a chain of latencies: what needs no values is done before the
    // wait for the kernel in front (this thread's first cells, interface and node),
    // and both cells are loaded before the first is used.
    constexpr int kCells = 2;
    Cell cell[kCells];
#pragma unroll
    for (int k = 0; k < kCells; ++k) cell[k] = make_cell(t + k * C.nt);
    Item item = make_item(t);
    const int r_own = t / C.sx, x_own = t - r_own * C.sx;
    const bool own = x_own < sx && r_own < rv;

    grid_wait_only();
    const T* __restrict__ u = R.u;
    T va[kCells], vb[kCells];
#pragma unroll
    for (int k = 0; k < kCells; ++k) {
        va[k] = vb[k] = T(0);
        if (cell[k].to >= 0) va[k] = ld(u + cell[k].a);
        if (cell[k].b >= 0) vb[k] = ld(u + cell[k].b);
    }
    // V^n of this thread's (first) node, ahead of its use
    T old = T(0);
    if (KIND == kKindCombine && own) old = ld(R.vn + (y0 + r_own) * nx + x0 + x_own);
#pragma unroll
    for (int k = 0; k < kCells; ++k)
        if (cell[k].to >= 0) V[cell[k].to] = cell[k].b >= 0 ? ghost_value(va[k], vb[k], cell[k].m, g.extrap) : va[k];
    for (int c = t + kCells * C.nt; c < (rv + 6) * (sx + 6); c += C.nt) {
        const Cell q = make_cell(c);
        if (q.to >= 0) V[q.to] = q.b >= 0 ? ghost_value(ld(u + q.a), ld(u + q.b), q.m, g.extrap) : ld(u + q.a);
    }
    __syncthreads();
    grid_next();

    for (int i = t; i < n_x + n_y; i += C.nt) {
        if (i != t) item = make_item(i);
        const bool along_x = item.along_x;
        const T* w0 = V + item.from;
        const int step = along_x ? 1 : W;
        T v[kW][6], pp[kW], pm[kW];
#pragma unroll
        for (int l = 0; l < kW; ++l)
#pragma unroll
            for (int k = 0; k < 6; ++k) v[l][k] = w0[l * W + k * step];
        iface_item<SCHEME>(v, along_x ? fl0 : fl1, pp, pm);
#pragma unroll
        for (int l = 0; l < kW; ++l) {
            const int o = item.to + l * (along_x ? C.sx + 1 : C.sx);
            (along_x ? xp : yp)[o] = pp[l];
            (along_x ? xm : ym)[o] = pm[l];
        }
    }
    __syncthreads();

    const auto half_inv = [&P](int d) -> T {
        if constexpr (iface_times6<T, SCHEME>()) return SP<T>::half_inv_dx6(P, d);
        else return SP<T>::half_inv_dx(P, d);
    };
    const T hh[2] = {half_inv(0), half_inv(1)};
    T par[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) par[k] = SP<T>::param(P, k);
    for (int i = t; i < C.sx * rv; i += C.nt) {
        const int r = i == t ? r_own : i / C.sx, x = i - r * C.sx;
        if (x >= sx) continue;
        const int flat = (y0 + r) * nx + x0 + x;
        if (KIND == kKindCombine && i != t) old = ld(R.vn + flat);
        const T pmx = xm[r * (C.sx + 1) + x], ppx = xp[r * (C.sx + 1) + x + 1];
        const T pmy = ym[r * C.sx + x], ppy = yp[(r + 1) * C.sx + x];
        const T S[2] = {add_rn(pmx, ppx), add_rn(pmy, ppy)}, Q[2] = {add_rn(ppx, -pmx), add_rn(ppy, -pmy)};
        T xc[2] = {T(0), T(0)};
        if constexpr (uses_coord<2, DYN>(0)) xc[0] = coord(SP<T>::lo(P, 0), x0 + x, SP<T>::dx(P, 0));
        if constexpr (uses_coord<2, DYN>(1)) xc[1] = coord(SP<T>::lo(P, 1), y0 + r, SP<T>::dx(P, 1));
        T res[1], w[1];
        const T vn[1] = {old};
        res[0] = stage_value<T, 2, DYN, KIND>(P, R, par, xc, T(0), T(0), S, Q, hh, P.alpha_global,
                                              V[(r + 3) * W + x + 3], old, w[0]);
        finish_values<T, 2, KIND>(R, res, w, vn);
        R.out[flat] = res[0];
    }
}

template <typename T, int DYN, int SCHEME, int KIND>
inline cudaError_t plane_prepare() {
    static std::atomic<unsigned long long> done{0};
    return smem_optin(plane_kernel<T, DYN, SCHEME, KIND>, done);
}
template <typename T, int DYN, int SCHEME, int KIND>
cudaError_t launch_plane(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    cudaError_t e = plane_prepare<T, DYN, SCHEME, KIND>();
    if (e != cudaSuccess) return e;
    return launch_dependent(plane_kernel<T, DYN, SCHEME, KIND>, dim3((unsigned)c.tiles), dim3((unsigned)c.nt),
                            plane_smem(c.sx, c.ty, sizeof(T)), s, p, c);
}

}  // namespace hj
