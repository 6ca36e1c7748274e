// plane_kernel.cuh -- the fused RK stage kernel on 2-D grids that leave the chip
// mostly idle: one interface per thread, then one node per thread.
//
// An FP64 2-D stage of 101^2 nodes is one short chain of dependent operations per
// thread, and with two rows a thread (rows_kernel.cuh) a chain of 11.4 us: one warp's FP64 instructions follow each other in 64 cycles each on its
// quarter of the SM, while the other quarters have no warp. Here the
// interfaces along both dimensions of a small tile are dealt out to the
// threads of a block (FP32: two rows' or two gaps' at a time, packed as in the
// row kernel), both halves go through shared memory, and each node is updated
// by a thread of its own: 6.2 us (5 x 12 nodes a block, two blocks an SM), 44 us
// instead of 50 on 511^2. FP32, whose stage is launch latency up to 301^2 (2.5 to
// 2.8 us with either kernel), keeps the row kernel where that is faster: the
// launch-shape tuner times both.
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

    grid_wait();
    const T* __restrict__ u = R.u;
    // V^n of this thread's (first) node, ahead of its use
    T old = T(0);
    const int x_own = t % C.sx, r_own = t / C.sx;
    const bool own = x_own < sx && r_own < rv;
    if (KIND == kKindCombine && own) old = ld(R.vn + (y0 + r_own) * nx + x0 + x_own);

    // value at offset i of a line (n nodes from base, stride s), ghosts included
    auto at = [&](int base, int i, int n, int s, bool periodic) -> T {
        if (i >= 0 && i < n) return ld(u + base + i * s);
        if (periodic) return ld(u + base + (i + (i < 0 ? n : -n)) * s);
        const int e = i < 0 ? 0 : n - 1, inner = i < 0 ? 1 : n - 2;
        return ghost_value(ld(u + base + e * s), ld(u + base + inner * s), i < 0 ? -i : i - (n - 1), g.extrap);
    };
    for (int c = t; c < (rv + 6) * (sx + 6); c += C.nt) {
        const int r = c / (sx + 6) - 3, x = c - (r + 3) * (sx + 6) - 3;
        const bool in_x = x >= 0 && x < sx, in_y = r >= 0 && r < rv;
        if (in_y) V[(r + 3) * W + x + 3] = at((y0 + r) * nx, x0 + x, nx, 1, per0);
        else if (in_x) V[(r + 3) * W + x + 3] = at(x0 + x, y0 + r, ny, nx, per1);
    }
    __syncthreads();

    const int n_x = (sx + 1) * ((rv + kW - 1) / kW), n_y = sx * ((rv + kW) / kW);
    for (int i = t; i < n_x + n_y; i += C.nt) {
        const bool along_x = i < n_x;
        int line, x;  // first row, or first gap, and column
        if (along_x) {
            line = i / (sx + 1);
            x = i - line * (sx + 1);
        } else {
            line = (i - n_x) / sx;
            x = i - n_x - line * sx;
        }
        line *= kW;
        const T* w0 = along_x ? V + (line + 3) * W + x : V + line * W + x + 3;
        const int step = along_x ? 1 : W;
        T v[kW][6], pp[kW], pm[kW];
#pragma unroll
        for (int l = 0; l < kW; ++l)
#pragma unroll
            for (int k = 0; k < 6; ++k) v[l][k] = w0[l * W + k * step];
        iface_item<SCHEME>(v, along_x ? fl0 : fl1, pp, pm);
#pragma unroll
        for (int l = 0; l < kW; ++l) {
            const int o = along_x ? (line + l) * (C.sx + 1) + x : (line + l) * C.sx + x;
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
        const int r = i / C.sx, x = i - r * C.sx;
        if (x >= sx) continue;
        const int flat = (y0 + r) * nx + x0 + x;
        if (KIND == kKindCombine && i != t) old = ld(R.vn + flat);
        const T pmx = xm[r * (C.sx + 1) + x], ppx = xp[r * (C.sx + 1) + x + 1];
        const T pmy = ym[r * C.sx + x], ppy = yp[(r + 1) * C.sx + x];
        const T S[2] = {add_rn(pmx, ppx), add_rn(pmy, ppy)}, Q[2] = {add_rn(ppx, -pmx), add_rn(ppy, -pmy)};
        T xc[2] = {T(0), T(0)};
        if constexpr (uses_coord<2, DYN>(0)) xc[0] = coord(SP<T>::lo(P, 0), x0 + x, SP<T>::dx(P, 0));
        if constexpr (uses_coord<2, DYN>(1)) xc[1] = coord(SP<T>::lo(P, 1), y0 + r, SP<T>::dx(P, 1));
        const T res = stage_value<T, 2, DYN, KIND>(P, R, par, xc, T(0), T(0), S, Q, hh, P.alpha_global,
                                                         V[(r + 3) * W + x + 3], old);
        R.out[flat] = res;
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
