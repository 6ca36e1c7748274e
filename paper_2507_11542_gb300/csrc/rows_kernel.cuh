// rows_kernel.cuh -- the fused RK stage kernel (WENO5, ENO1/2/3) on 2-4 dimensional
// grids, tiled for GB300:
//
//  * A thread block owns a tile of one plane of dimensions (0, 1): a segment of
//    SX nodes along dimension 0 by TY <= 8 rows, with three halo cells on each
//    side. Each node thread works on two neighbouring rows of its column (one
//    per lane of a pair, lanes.cuh): one walk through addresses, predicates and
//    loop control serves two nodes, and FP32 arithmetic is packed.
//  * The upwind scheme (WENO5, ENO1/2/3) is evaluated per interface (one
//    interface gives p+ of a node and p- of the next). Along dimension 0 the
//    node thread of column x computes the interfaces between x-1 and x of its
//    two rows; along dimension 1 the one below its first row and the one
//    between its two rows. So each node pays for about one interface per
//    dimension instead of two.
//  * Whole warps have one role: node warps hold the node threads; edge warps
//    copy the halos two planes ahead and compute what is left over at the
//    tile's edges (the last interface of every row, the gap above the last row).
//  * For 3-D and 4-D grids the block streams along the last dimension through
//    a chunk of planes: each thread keeps its columns' values in registers and
//    carries the interface result p- to the next plane. One barrier per plane.
//  * In 4-D, dimension 2 is differentiated two-sided from 7-point loads.
//  * Ghost values (periodic wrap or slope continued away from zero, Sec. 2.1)
//    are produced where values are staged; no padded array exists.
// Then: Hamiltonian + Lax-Friedrichs dissipation (Sec. 4), BRT clamp (Sec.
// 6.1) and the TVD-RK3 stage combination (Sec. 5), one store per node.
#pragma once

#include <atomic>
#include <type_traits>

#include "stencil.cuh"
#include "weno_iface.cuh"

namespace hj {

// Launch bounds, i.e. registers a thread (blocks have at most rows_max_threads).
// FP32 stage of 101^3 / 161x113x79 at 640, 768, 896, 1024 threads (96, 80, 72, 64
// registers): 16.7, 16.1, 15.7, 16.2 / 22.6, 20.5, 20.0, 20.7 us (now 14.4 / 18.5 at
// 896); of 81^4 at 768 and 896: 0.69 and 0.71 ms, and with the lines of dimension 2
// loaded a phase ahead 0.66 at 896 (now 0.636).
template <typename T, int D> struct RowsBounds { static constexpr int kThreads = D == 2 ? 768 : 896; };
template <int D> struct RowsBounds<double, D> { static constexpr int kThreads = kRowsThreadsF64; };

// The slope that ghost values continue outward, and the m-th ghost value.
template <typename T>
__device__ __forceinline__ T outward_slope(T edge, T inner, int extrap) {
    const T d = edge - inner;
    if (extrap == HJ_EXTRAP_LINEAR) return d;
    return edge == T(0) ? fabs(d) * T(0) : copysign(d, edge);
}
template <typename T>
__device__ __forceinline__ T ghost_value(T edge, T inner, int m, int extrap) {
    return add_rn(edge, mul_rn(T(m), outward_slope(edge, inner, extrap)));
}

// Values of one stage launch that differ between the three RK stages, in the
// kernel's precision (kept in registers).
template <typename T>
struct StageRun {
    const T* u;        // stencil input
    const T* vn;       // V^n (stages 2 and 3)
    T* out;            // result
    T* also_out;       // if not null, the result is written here as well (a time slice)
    T dt, cv, cu;
    bool minv, brt0;
};

template <typename T>
__device__ __forceinline__ StageRun<T> stage_run(const StageParams& P) {
    StageRun<T> R;
    R.u = static_cast<const T*>(P.u);
    R.vn = static_cast<const T*>(P.vn);
    R.out = static_cast<T*>(P.out);
    R.also_out = nullptr;
    R.dt = SP<T>::dt(P);
    R.cv = SP<T>::cv(P);
    R.cu = SP<T>::cu(P);
    R.minv = P.minv_after;
    R.brt0 = P.brt_min0;
    return R;
}

// What a stage stores at a node, from the raw sums and differences of its
// one-sided derivatives (lf_node), its stage input `center` and its V^n `old`;
// finish_values() completes it (w: center + dt times the term).
template <typename T, int D, int DYN, int KIND>
__device__ __forceinline__ T stage_value(const StageParams& P, const StageRun<T>& R, const T* par, const T* x, T c, T s,
                                         const T* S, const T* Q, const T* h, bool alpha_global, T center, T old, T& w) {
    T yd = lf_node<T, D, DYN>(P, par, x, c, s, S, Q, h, alpha_global);
    // BRT min(0, .) as a clamp (+inf: none); FP64 on the high word: what is positive
    // becomes 0, NaN of either sign (quiet: high word above infinity's) stays, since
    // its sign depends on how it came about
    if constexpr (std::is_same<T, double>::value) {
        if (R.brt0 && (unsigned)__double2hiint(yd) <= 0x7ff00000u) yd = 0.0;
    } else {
        yd = fminf(yd, R.brt0 ? 0.0f : INFINITY);
    }
    if constexpr (KIND == kKindTerm) return yd;
    w = fma_rn(R.dt, yd, center);
    if constexpr (KIND != kKindCombine) return w;
    // cv V^n + cu w; with cv + cu = 1 FP32 takes it as w + cv (V^n - w): the
    // difference is small, so that one rounding alone counts
    if constexpr (std::is_same<T, double>::value) return fma_rn(R.cu, w, mul_rn(R.cv, old));
    else return fma_rn(R.cv, add_rn(old, -w), w);
}
// Where w + cv (V^n - w) is not finite (an infinite value on either side, or two
// of opposite sign near the largest), the sum as it stands keeps what is infinite
// infinite and the rest finite. A thread's values are tested together and the rest
// branched over (a select for each cost the batch of 24 solves 2 %), but in 4-D,
// where the selects are the cheaper (81^4 step: 1899 and 1856 us).
template <typename T, int D, int KIND, int N>
__device__ __forceinline__ void finish_values(const StageRun<T>& R, T (&res)[N], const T (&w)[N], const T (&old)[N]) {
    if constexpr (KIND == kKindCombine) {
        if constexpr (std::is_same<T, float>::value) {
            bool odd = true;
            if constexpr (D < 4) {
                float size = fabsf(res[0]);
                if constexpr (N == 2) size = __fadd_rn(size, fabsf(res[1]));
                odd = !(size < INFINITY);
            }
            if (__builtin_expect(odd, 0)) {
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (!(fabsf(res[k]) < INFINITY)) res[k] = fma_rn(R.cu, w[k], mul_rn(R.cv, old[k]));
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) res[k] = R.minv ? fmin(res[k], old[k]) : res[k];
    }
}

// Asynchronous copy of one element from global to shared memory (cp.async:
// no register is involved). The issuing thread waits for its own copies with
// cp_async_wait_all; a barrier after that publishes them to the block.
template <typename T> __device__ __forceinline__ void cp_async_elem(T* dst, const T* src);
template <> __device__ __forceinline__ void cp_async_elem<float>(float* dst, const float* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    const size_t gsrc = __cvta_generic_to_global(src);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gsrc) : "memory");
}
template <> __device__ __forceinline__ void cp_async_elem<double>(double* dst, const double* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    const size_t gsrc = __cvta_generic_to_global(src);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }


__device__ __forceinline__ void block_barrier(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

// Where a tile lies and who works on it (the same for all threads of a block).
struct Tile {
    int x0, sx;     // first node of the segment along dimension 0, nodes in it
    int y0, rv;     // first row, rows in the grid
    int i2;         // dimension-2 index (4-D)
    int zbeg, zend; // planes along the streamed dimension
    int stride;     // SX: node thread t works on column t mod SX, row pair t div SX
    int nn, nt;     // threads of the node warps, all threads
};

// Shared memory: two buffers (plane p in buffer (p - zbeg) mod 2), each a column
// of kPitch values per node of the segment and three more on each side:
//   [0, 16)   rows -4 .. 11 of the plane (row r at 4 + r; -4 and 11 unused)
//   [16, 24)  p+ of the node to the left along dimension 0, per row
//   [24, 29)  p+ of row 2k - 1 along dimension 1
// so that both neighbour directions are constant offsets from one address, and
// a thread's two rows are one aligned access. A pitch of 30 spreads a warp's
// pairs over all banks.
constexpr int kColX = 16, kColY = 24;

// One tile. Planes are software-pipelined with one barrier per plane:
//   phase A(z): interfaces of plane z along dimensions 0 and 1 (node and edge
//               warps); edge warps wait for their copies into plane z+1
//   barrier
//   phase B(z): node updates of plane z; staging of plane z+2 (node values from
//               the column queues, halos by the edge warps' asynchronous copies)
// The p- half of an interface stays in a register, the p+ half goes through
// shared memory where another thread owns the node. Derivatives stay raw
// (undivided differences) until the node combines them, scaled by 1/(2 dx),
// into the means and half differences the Hamiltonian takes. Flat indices are
// 32-bit (the grid has fewer than 2^31 nodes). Threads of the node warps
// without a node work on a clamped one and store nothing.
template <typename T, int D, int SCHEME, bool WAIT>
__device__ __forceinline__ void edge_warps(const StageParams& P, const T* __restrict__ u, const Tile& C, const int t,
                                           T* const smem, const int buf) {
    constexpr int kP = kRowsPitch;
    constexpr int SD = (D >= 3) ? D - 1 : 0;
    const GridDev& g = P.g;
    const int nx = g.n[0], ny = g.n[1];
    const bool per0 = g.periodic_mask & 1u, per1 = (g.periodic_mask >> 1) & 1u;
    const int extrap = g.extrap;
    const int et = t - C.nn, en = C.nt - C.nn;
    const int sS = (D >= 3) ? (int)g.stride[SD] : 0;
    const int plane0 = (D == 4) ? C.i2 * (int)g.stride[2] : 0;
    const T fl0 = SP<T>::floor(P, 0), fl1 = SP<T>::floor(P, 1);

    // A thread's share of a plane's halo: the rows -3, -2, -1 and rv, rv+1, rv+2 of
    // kCols columns (et, et + en, ...), and for the last sixteen threads the columns
    // -3, -2, -1 or sx, sx+1, sx+2 of a row. Sources do not change from plane to
    // plane. Ghost cells (extrapolated edges) need the two outermost values at
    // their end of the line, which are loaded one plane before they are made. In a
    // launch of one wave the blocks that make them take the longest, and this path
    // is kept short: without any edge work a 161x113x79 FP32 stage takes 15.7 us of
    // 19.0, and whole lines in place of sides (eight row threads with twelve cells
    // more than the others) cost 0.8 us.
    constexpr int kCols = rows_edge_cols(sizeof(T) == 8);
    struct Side {
        int src[3];  // flat index, or -1: a ghost cell
        bool ghost;  // the side has ghost cells
        T m;         // distance of its first cell from the grid
        T e, i;      // outermost values in the next plane
    };
    auto make_side = [&](Side& q, int first, int n, bool periodic, int base, int step, bool high) {
        q.ghost = false;
        q.e = q.i = T(0);
        q.m = T(high ? first - (n - 1) : -first);
#pragma unroll
        for (int h = 0; h < 3; ++h) {
            int i = first + h;  // -3 .. n + 2
            const bool out = i < 0 || i >= n;
            if (periodic) i += i < 0 ? n : i >= n ? -n : 0;
            else if (out) q.ghost = true;
            q.src[h] = !periodic && out ? -1 : base + i * step;
        }
    };
    auto fetch = [&](Side& q, const T* __restrict__ line, int n, int step, bool high) {
        if (q.ghost) {
            q.e = ld(line + (high ? (n - 1) * step : 0));
            q.i = ld(line + (high ? (n - 2) * step : step));
        }
    };
    auto copy = [&](const Side& q, const T* __restrict__ plane, T* dst, int step) {
#pragma unroll
        for (int h = 0; h < 3; ++h)
            if (q.src[h] >= 0) cp_async_elem(dst + h * step, plane + q.src[h]);
    };
    auto ghosts = [&](const Side& q, T* dst, int step, T dir) {  // dir: 1 above the grid, -1 below
        if (!q.ghost) return;
        const T slope = outward_slope(q.e, q.i, extrap);
#pragma unroll
        for (int h = 0; h < 3; ++h)
            if (q.src[h] < 0) dst[h * step] = add_rn(q.e, mul_rn(fma_rn(dir, T(h), q.m), slope));
    };
    const int rt = et - (en - 2 * kRowsMaxTy), r = rt & (kRowsMaxTy - 1);
    const bool row_high = rt >= kRowsMaxTy, row_job = rt >= 0 && r < C.rv;
    const int col_base = plane0 + C.x0 + et, row_base = plane0 + (C.y0 + r) * nx;
    Side low[kCols], high[kCols], row;
#pragma unroll
    for (int k = 0; k < kCols; ++k)
        if (et + k * en < C.sx) {
            make_side(low[k], C.y0 - 3, ny, per1, col_base + k * en, nx, false);
            make_side(high[k], C.y0 + C.rv, ny, per1, col_base + k * en, nx, true);
        }
    if (row_job) make_side(row, row_high ? C.x0 + C.sx : C.x0 - 3, nx, per0, row_base, 1, row_high);
    T* const col_low = smem + (et + 3) * kP + 1;
    T* const col_high = smem + (et + 3) * kP + 4 + C.rv;
    T* const row_to = smem + (row_high ? (C.sx + 3) * kP : 0) + 4 + r;
    auto fetch_all = [&](int p) {
        const T* __restrict__ plane = u + p * sS;
#pragma unroll
        for (int k = 0; k < kCols; ++k)
            if (et + k * en < C.sx) {
                fetch(low[k], plane + col_base + k * en, ny, nx, false);
                fetch(high[k], plane + col_base + k * en, ny, nx, true);
            }
        if (row_job) fetch(row, plane + row_base, nx, 1, row_high);
    };
    auto keep = [&](Side* to) {  // the values fetched last
#pragma unroll
        for (int k = 0; k < kCols; ++k) { to[2 * k] = low[k]; to[2 * k + 1] = high[k]; }
        to[2 * kCols] = row;
    };
    auto use = [&](const Side* from) {
#pragma unroll
        for (int k = 0; k < kCols; ++k) { low[k] = from[2 * k]; high[k] = from[2 * k + 1]; }
        row = from[2 * kCols];
    };
    auto copy_all = [&](int p, int o) {
        const T* __restrict__ plane = u + p * sS;
#pragma unroll
        for (int k = 0; k < kCols; ++k)
            if (et + k * en < C.sx) {
                copy(low[k], plane, col_low + o + k * en * kP, 1);
                copy(high[k], plane, col_high + o + k * en * kP, 1);
            }
        if (row_job) copy(row, plane, row_to + o, kP);
    };
    auto ghost_all = [&](int o) {
#pragma unroll
        for (int k = 0; k < kCols; ++k)
            if (et + k * en < C.sx) {
                ghosts(low[k], col_low + o + k * en * kP, 1, T(-1));
                ghosts(high[k], col_high + o + k * en * kP, 1, T(1));
            }
        if (row_job) ghosts(row, row_to + o, kP, row_high ? T(1) : T(-1));
    };

    // first two planes: all copies and all sources are under way before the first
    // ghost cell waits for its own (the stages of 161x113x79 and 101^3 in FP32 took
    // 19.0 and 15.0 us with one plane's sources after the other, 18.5 and 14.4 so)
    if constexpr (WAIT) grid_wait_only();
    const bool second = C.zbeg + 1 < C.zend;
    Side first[2 * kCols + 1], next[2 * kCols + 1];
    copy_all(C.zbeg, 0);
    if (second) copy_all(C.zbeg + 1, buf);
    fetch_all(C.zbeg);
    keep(first);
    if (second) {
        fetch_all(C.zbeg + 1);
        keep(next);
        if (C.zbeg + 2 < C.zend) fetch_all(C.zbeg + 2);
        Side third[2 * kCols + 1];
        keep(third);
        use(next);
        ghost_all(buf);
        use(first);
        ghost_all(0);
        use(third);
    } else {
        ghost_all(0);
    }
    cp_async_wait_all();
    block_barrier(C.nt);

    // left-over interfaces, two an item: the gap above the last row of two
    // columns where no node thread has it (an even number of rows), then the last
    // interface of both rows of a pair
    const int n_gap = (C.rv & 1) ? 0 : (C.sx + 1) >> 1;
    const int n_item = n_gap + ((C.rv + 1) >> 1);
#pragma unroll 1
    for (int z = C.zbeg; z < C.zend; ++z) {
        const int o = ((z - C.zbeg) & 1) * buf;
        T* const bz = smem + o;
        if (et < n_item) {  // en >= (sx + 1) / 2 + 4
            const bool gap = et < n_gap;
            const int pr = et - n_gap;
            const T* w0 = gap ? bz + (2 * et + 3) * kP + 1 + C.rv : bz + C.sx * kP + 4 + 2 * pr;
            const int step = gap ? 1 : kP, second_lane = gap ? kP : 1;  // (an odd last column: a halo column)
            Lanes<T> w[6], pp, pm;
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = lanes(w0[k * step], w0[k * step + second_lane]);
            iface_lanes<SCHEME>(w, gap ? fl1 : fl0, pp, pm);
            if (gap) {
                T* const g0 = bz + (2 * et + 3) * kP + kColY + (C.rv >> 1);
                g0[0] = lane_a(pp);
                g0[kP] = lane_b(pp);
            } else {
                put_lanes(bz + (C.sx + 3) * kP + kColX + 2 * pr, pp);
            }
        }
        cp_async_wait_all();  // this thread's copies into plane z+1
        block_barrier(C.nt);
        if (z + 2 < C.zend) {
            copy_all(z + 2, o);
            ghost_all(o);
            if (z + 3 < C.zend) fetch_all(z + 3);
        }
    }
}

template <typename T, int D, int DYN, int SCHEME, int KIND, bool WAIT>
__device__ __forceinline__ void node_warps(const StageParams& P, const StageRun<T>& R, const Tile& C, const int t,
                                           T* const smem, const int buf) {
    using L = Lanes<T>;
    constexpr int kP = kRowsPitch;
    constexpr int SD = (D >= 3) ? D - 1 : 0;  // streamed dimension
    const GridDev& g = P.g;
    const int nx = g.n[0], ny = g.n[1];
    const T* __restrict__ u = R.u;
    const T* __restrict__ vn = R.vn;
    T* __restrict__ out = R.out;
    T* __restrict__ also_out = R.also_out;

    int pr = t / C.stride, x = t - pr * C.stride;
    const bool node = x < C.sx && 2 * pr < C.rv;      // this thread's first row
    const bool node1 = node && 2 * pr + 1 < C.rv;      // its second
    x = min(x, C.sx - 1);
    pr = min(pr, (C.rv - 1) >> 1);
    const int y = C.y0 + 2 * pr;
    const int y1 = min(y + 1, ny - 1);

    const int ns = (D >= 3) ? g.n[SD] : 1;
    const int sS = (D >= 3) ? (int)g.stride[SD] : 0;
    const bool perS = (D >= 3) ? ((g.periodic_mask >> SD) & 1u) : false;
    const int extrap = g.extrap;
    const int plane0 = (D == 4) ? C.i2 * (int)g.stride[2] : 0;
    const int col0 = plane0 + C.x0 + x + y * nx;   // flat index of the first row's node at streamed index 0
    const int col1 = plane0 + C.x0 + x + y1 * nx;
    const T fl0 = SP<T>::floor(P, 0), fl1 = SP<T>::floor(P, 1), flS = SP<T>::floor(P, SD);

    // values of both columns at plane z (z within three of the grid; ns >= 4)
    auto column = [&](int z) -> L {
        if (z >= 0 && z < ns) return lanes(ld(u + col0 + z * sS), ld(u + col1 + z * sS));
        if (perS) {
            const int w = z + (z < 0 ? ns : -ns);
            return lanes(ld(u + col0 + w * sS), ld(u + col1 + w * sS));
        }
        const int e = z < 0 ? 0 : ns - 1, i = z < 0 ? 1 : ns - 2, m = z < 0 ? -z : z - (ns - 1);
        return lanes(ghost_value(ld(u + col0 + e * sS), ld(u + col0 + i * sS), m, extrap),
                     ghost_value(ld(u + col1 + e * sS), ld(u + col1 + i * sS), m, extrap));
    };

    // 1/(2 dx), or 1/(12 dx) where the interface evaluation returns six times the derivatives
    const auto half_inv = [&P](int d) -> T {
        if constexpr (iface_times6<T, SCHEME>()) return SP<T>::half_inv_dx6(P, d);
        else return SP<T>::half_inv_dx(P, d);
    };
    T hh[D];
#pragma unroll
    for (int d = 0; d < D; ++d) hh[d] = half_inv(d);
    // read before the loop: a batch's descriptors lie in global memory, which its stores may alias
    T par[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) par[k] = SP<T>::param(P, k);
    const bool alpha_global = P.alpha_global;
    // node coordinates that do not change along the streamed dimension
    T xa[D], xb[D];
#pragma unroll
    for (int d = 0; d < D; ++d) xa[d] = xb[d] = T(0);
    if constexpr (uses_coord<D, DYN>(0)) xa[0] = xb[0] = coord(SP<T>::lo(P, 0), C.x0 + x, SP<T>::dx(P, 0));
    if constexpr (uses_coord<D, DYN>(1)) {
        xa[1] = coord(SP<T>::lo(P, 1), y, SP<T>::dx(P, 1));
        xb[1] = coord(SP<T>::lo(P, 1), y1, SP<T>::dx(P, 1));
    }
    if constexpr (D == 4 && uses_coord<D, DYN>(2)) xa[2] = xb[2] = coord(SP<T>::lo(P, 2), C.i2, SP<T>::dx(P, 2));
    if constexpr (WAIT) grid_wait_only();
    const T* __restrict__ trig = Trig<T>::get(P);       // cos of the dimension-2 coordinate
    const T* __restrict__ trig_s = uses_angle<D, DYN>() ? trig + g.n[2] : trig;  // sin
    T cos2 = T(0), sin2 = T(0);  // angle of dimension 2 (fixed for the block in 4-D, the next plane's in 3-D)
    if constexpr (D == 4 && uses_angle<D, DYN>()) {
        cos2 = trig[C.i2];
        sin2 = trig_s[C.i2];
    }
    if constexpr (D == 3 && uses_angle<D, DYN>()) {
        cos2 = trig[C.zbeg];
        sin2 = trig_s[C.zbeg];
    }

    // Streamed-dimension queue: q[k] = V at plane z-2+k (k = 0..5); carry = raw p- at z.
    // A warm-up step evaluates the interface below the first plane, so that
    // every interface goes through the same code and results do not depend
    // on where chunks start. FP64 WENO5 and ENO2 keep the differences instead
    // (Weno5Line, Eno2Line; bit for bit the same results).
    constexpr bool kSlide = std::is_same<T, double>::value && SCHEME == HJ_WENO5 && D >= 3;
    L q[6], q6{}, carry{};
    constexpr bool kSlide2 = std::is_same<T, double>::value && SCHEME == HJ_ENO2 && D >= 3;
    [[maybe_unused]] Weno5Line za, zb;
    [[maybe_unused]] Eno2Line ea, eb;
    if constexpr (D >= 3) {
#pragma unroll
        for (int k = 0; k < 6; ++k) q[k] = column(C.zbeg - 3 + k);
        L unused;
        if constexpr (kSlide) {
            za.start(q[0].a, q[1].a, q[2].a, q[3].a, q[4].a, q[5].a);
            za.eval(flS, unused.a, carry.a);
            zb.start(q[0].b, q[1].b, q[2].b, q[3].b, q[4].b, q[5].b);
            zb.eval(flS, unused.b, carry.b);
        } else if constexpr (kSlide2) {
            ea.start(q[1].a, q[2].a, q[3].a, q[4].a);
            ea.eval(unused.a, carry.a);
            eb.start(q[1].b, q[2].b, q[3].b, q[4].b);
            eb.eval(unused.b, carry.b);
        } else {
            iface_lanes<SCHEME>(q, flS, unused, carry);
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) q[k] = q[k + 1];
        q6 = column(C.zbeg + 3);
    } else {
        q[2] = column(0);
    }

    // The queue's next value, the next angle and V^n of the next plane (2-D and
    // 3-D grids) are loaded one plane ahead of their use, so that a whole plane
    // of work covers their latency. Where out aliases V^n, the value read is
    // this thread's own node, which it writes one plane later.
    constexpr bool kVnAhead = KIND == kKindCombine && D <= 3;
    int f0 = col0 + C.zbeg * sS, f1 = col1 + C.zbeg * sS;  // the two nodes of plane z
    const T* __restrict__ u4 = u + 4 * (long long)sS;
    const T* __restrict__ vn_next = vn + sS;
    T vn0 = T(0), vn1 = T(0);
    if constexpr (kVnAhead) {
        vn0 = ld(vn + f0);
        vn1 = ld(vn + f1);
    }

    const int s_own = (x + 3) * kP + 4 + 2 * pr;            // this thread's pair
    const int s_gap = (x + 3) * kP + kColY + pr;             // p+ of the row below it
    // the row above an odd last row is the edge warps' (a halo row)
    auto put_own = [&](T* b, L v) {
        if (node1) put_lanes(b + s_own, v);
        else if (node) b[s_own] = lane_a(v);
    };
    put_own(smem, q[2]);
    if (D >= 3 && C.zbeg + 1 < C.zend) put_own(smem + buf, q[3]);
    block_barrier(C.nt);
    grid_next();

#pragma unroll 1
    for (int z = C.zbeg; z < C.zend; ++z) {
        T* const bz = smem + ((z - C.zbeg) & 1) * buf;
        const T cosz = cos2, sinz = sin2;
        T va = vn0, vb = vn1;
        if constexpr (D >= 3) q[5] = q6;
        // the next plane's values, a whole plane of work ahead of their use
        if (D >= 3 && z + 1 < C.zend) {
            if (z + 4 < ns) q6 = lanes(ld(u4 + f0), ld(u4 + f1));
            else q6 = column(z + 4);
            if constexpr (D == 3 && uses_angle<D, DYN>()) {
                cos2 = trig[z + 1];
                sin2 = trig_s[z + 1];
            }
            if constexpr (kVnAhead) {
                vn0 = ld(vn_next + f0);
                vn1 = ld(vn_next + f1);
            }
        }

        // the dimension-2 lines of plane z, loaded before phase A covers their latency
        T v0[D == 4 ? 7 : 1], v1[D == 4 ? 7 : 1];
        if constexpr (D == 4) {
            const bool per2 = (g.periodic_mask >> 2) & 1u;
            gather7<T>(u, (long long)f0, C.i2, g.n[2], g.stride[2], per2, extrap, v0);
            gather7<T>(u, (long long)f1, C.i2, g.n[2], g.stride[2], per2, extrap, v1);
            if constexpr (KIND == kKindCombine) {
                va = ld(vn + f0);
                vb = ld(vn + f1);
            }
        }

        // phase A: interfaces of plane z along dimensions 0 and 1
        L pmx, pmy, pp;
        const T* own = bz + s_own;
        L w[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = lanes_at(own + (k - 3) * kP);
        iface_lanes<SCHEME>(w, fl0, pp, pmx);
        if (node) put_lanes(bz + s_own + (kColX - 4), pp);
        const L b2 = lanes_at(own - 4), b1 = lanes_at(own - 2), up = lanes_at(own + 2);
        const T v[7] = {lane_b(b2), lane_a(b1), lane_b(b1), lane_a(w[3]), lane_b(w[3]), lane_a(up), lane_b(up)};
        iface_line<SCHEME>(v, fl1, pp, pmy);
        if (node) bz[s_gap] = lane_a(pp);
        const T ppy_a = lane_b(pp);
        block_barrier(C.nt);

        // phase B: staging of plane z+2, then the node updates of plane z
        const L ppx = lanes_at(bz + s_own + (kColX - 4) + kP);
        const L ppy = lanes(ppy_a, bz[s_gap + 1]);
        if (D >= 3 && z + 2 < C.zend) put_own(bz, q[4]);
        // raw sums and differences of the one-sided derivatives
        L sm[D], df[D];
        sm[0] = pmx + ppx;
        df[0] = ppx - pmx;
        sm[1] = pmy + ppy;
        df[1] = ppy - pmy;
        if constexpr (D >= 3) {
            L pps, next;
            if constexpr (kSlide) {
                za.slide(q[4].a, q[5].a);
                za.eval(flS, pps.a, next.a);
                zb.slide(q[4].b, q[5].b);
                zb.eval(flS, pps.b, next.b);
            } else if constexpr (kSlide2) {
                ea.slide(q[3].a, q[4].a);
                ea.eval(pps.a, next.a);
                eb.slide(q[3].b, q[4].b);
                eb.eval(pps.b, next.b);
            } else {
                iface_lanes<SCHEME>(q, flS, pps, next);
            }
            sm[SD] = carry + pps;
            df[SD] = pps - carry;
            carry = next;
        }
        if constexpr (D == 4) {
            // dimension 2: both interfaces of each node from a 7-point line
            L l[7], pm2, pp2, unused0, unused1;
#pragma unroll
            for (int k = 0; k < 7; ++k) l[k] = lanes(v0[k], v1[k]);
            const T fl2 = SP<T>::floor(P, 2);
            iface_lanes<SCHEME>(l, fl2, unused0, pm2);
            iface_lanes<SCHEME>(l + 1, fl2, pp2, unused1);
            sm[2] = pm2 + pp2;
            df[2] = pp2 - pm2;
            if constexpr (uses_coord<D, DYN>(3)) xa[3] = xb[3] = coord(SP<T>::lo(P, 3), z, SP<T>::dx(P, 3));
        }
        if constexpr (D == 3 && uses_coord<D, DYN>(2)) xa[2] = xb[2] = coord(SP<T>::lo(P, 2), z, SP<T>::dx(P, 2));
        T S[D], Q[D];
#pragma unroll
        for (int d = 0; d < D; ++d) { S[d] = lane_a(sm[d]); Q[d] = lane_a(df[d]); }
        const T vs[2] = {va, vb};
        T res[2], w2[2];
        res[0] = stage_value<T, D, DYN, KIND>(P, R, par, xa, cosz, sinz, S, Q, hh, alpha_global, lane_a(q[2]), va, w2[0]);
#pragma unroll
        for (int d = 0; d < D; ++d) { S[d] = lane_b(sm[d]); Q[d] = lane_b(df[d]); }
        res[1] = stage_value<T, D, DYN, KIND>(P, R, par, xb, cosz, sinz, S, Q, hh, alpha_global, lane_b(q[2]), vb, w2[1]);
        finish_values<T, D, KIND>(R, res, w2, vs);
        if (node) out[f0] = res[0];
        if (node1) out[f1] = res[1];
        if (also_out) {
            if (node) also_out[f0] = res[0];
            if (node1) also_out[f1] = res[1];
        }
        f0 += sS;
        f1 += sS;
        if constexpr (D >= 3) {
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = q[k + 1];
        }
    }
}

template <typename T, int D, int DYN, int SCHEME, int KIND, bool WAIT = false>
__device__ __forceinline__ void rows_tile(const StageParams& P, const StageRun<T>& R, const int SX, const int TY,
                                          const int NT, const int tz, const int tile, const int i2, const int chunk,
                                          const int t, T* const smem) {
    const GridDev& g = P.g;
    const int nseg = (g.n[0] + SX - 1) / SX;
    const int row_tile = tile / nseg, seg = tile - row_tile * nseg;
    constexpr int SD = (D >= 3) ? D - 1 : 0;
    Tile C;
    C.x0 = seg * SX;
    C.sx = min(SX, g.n[0] - C.x0);
    C.y0 = row_tile * TY;
    C.rv = min(TY, g.n[1] - C.y0);
    C.i2 = (D == 4) ? i2 : 0;
    C.zbeg = (D >= 3) ? chunk * tz : 0;
    C.zend = (D >= 3) ? min(g.n[SD], C.zbeg + tz) : 1;
    C.stride = SX;
    C.nn = rows_node_threads(SX, TY);
    C.nt = NT;
    const int buf = rows_buf_elems(SX);
    if (t < C.nn) node_warps<T, D, DYN, SCHEME, KIND, WAIT>(P, R, C, t, smem, buf);
    else edge_warps<T, D, SCHEME, WAIT>(P, R.u, C, t, smem, buf);
}

template <typename T, int D, int DYN, int SCHEME, int KIND>
__global__ void __launch_bounds__(RowsBounds<T, D>::kThreads, 1) rows_kernel(const StageParams P, const RowsCfg C) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const StageRun<T> R = stage_run<T>(P);
    const int i2 = (D == 4) ? (int)blockIdx.y : 0;
    const int chunk = (D == 3) ? (int)blockIdx.y : ((D == 4) ? (int)blockIdx.z : 0);
    rows_tile<T, D, DYN, SCHEME, KIND, true>(P, R, C.sx, C.ty, C.nt, C.tz, blockIdx.x, i2, chunk, threadIdx.x,
                                       reinterpret_cast<T*>(smem_raw));
}

template <int D>
inline void rows_shape(const StageParams& p, const RowsCfg& c, dim3& grid, dim3& block) {
    block = dim3((unsigned)c.nt, 1, 1);
    grid = dim3((unsigned)c.tiles, 1, 1);
    if (D == 3) grid.y = (unsigned)c.nchunks;
    if (D == 4) { grid.y = (unsigned)p.g.n[2]; grid.z = (unsigned)c.nchunks; }
}

// Opts a kernel into 200 KiB of dynamic shared memory, once per device (the
// attribute belongs to the current device's copy of the kernel); `done` holds
// one bit per device already set (devices 0..63; others are set every call).
template <typename K>
inline cudaError_t smem_optin(K* kernel, std::atomic<unsigned long long>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = (dev >= 0 && dev < 64) ? (1ull << dev) : 0ull;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    done.fetch_or(bit, std::memory_order_relaxed);  // setting the attribute twice (a race) is harmless
    return cudaSuccess;
}

template <typename T, int D, int DYN, int SCHEME, int KIND>
inline cudaError_t rows_prepare() {
    static std::atomic<unsigned long long> done{0};
    return smem_optin(rows_kernel<T, D, DYN, SCHEME, KIND>, done);
}

// (plane_kernel.cuh)
template <typename T, int DYN, int SCHEME, int KIND>
cudaError_t launch_plane(const StageParams& p, const RowsCfg& c, cudaStream_t s);

template <typename T, int D, int DYN, int SCHEME, int KIND>
cudaError_t launch_rows_kind(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    if constexpr (D == 2) {
        if (c.plane) return launch_plane<T, DYN, SCHEME, KIND>(p, c, s);
    }
    dim3 grid, block;
    rows_shape<D>(p, c, grid, block);
    cudaError_t e = rows_prepare<T, D, DYN, SCHEME, KIND>();
    if (e != cudaSuccess) return e;
    return launch_dependent(rows_kernel<T, D, DYN, SCHEME, KIND>, grid, block, rows_smem(c.sx, sizeof(T)), s, p, c);
}

template <typename T, int D, int DYN, int SCHEME>
cudaError_t launch_rows_scheme(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    switch (stage_kind(p)) {
    case kKindTerm: return launch_rows_kind<T, D, DYN, SCHEME, kKindTerm>(p, c, s);
    case kKindFirst: return launch_rows_kind<T, D, DYN, SCHEME, kKindFirst>(p, c, s);
    default: return launch_rows_kind<T, D, DYN, SCHEME, kKindCombine>(p, c, s);
    }
}
template <typename T, int D, int DYN>
cudaError_t launch_rows_weno5(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    return launch_rows_scheme<T, D, DYN, HJ_WENO5>(p, c, s);
}
template <typename T, int D, int DYN>
cudaError_t launch_rows_eno2(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    return launch_rows_scheme<T, D, DYN, HJ_ENO2>(p, c, s);
}
template <typename T, int D, int DYN>
cudaError_t launch_rows_eno1(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    return launch_rows_scheme<T, D, DYN, HJ_ENO1>(p, c, s);
}
template <typename T, int D, int DYN>
cudaError_t launch_rows_eno3(const StageParams& p, const RowsCfg& c, cudaStream_t s) {
    return launch_rows_scheme<T, D, DYN, HJ_ENO3>(p, c, s);
}

// Resident blocks per SM of the stage kernels of a configuration (the
// combining stages, the largest of the three kinds); 0 if it cannot launch.
template <typename T, int D, int DYN, int SCHEME>
int rows_bps_scheme(const StageParams& p, const RowsCfg& c) {
    if (c.plane) return D == 2 && c.nt <= kPlaneThreads && plane_smem(c.sx, c.ty, sizeof(T)) <= 200 * 1024 ? 1 : 0;
    if (c.nt > RowsBounds<T, D>::kThreads) return 0;
    if (rows_prepare<T, D, DYN, SCHEME, kKindCombine>() != cudaSuccess) return 0;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, rows_kernel<T, D, DYN, SCHEME, kKindCombine>, c.nt,
                                                      rows_smem(c.sx, sizeof(T))) != cudaSuccess)
        return 0;
    return bps;
}
template <typename T, int D, int DYN>
int rows_bps_weno5(const StageParams& p, const RowsCfg& c) {
    return rows_bps_scheme<T, D, DYN, HJ_WENO5>(p, c);
}
template <typename T, int D, int DYN>
int rows_bps_eno2(const StageParams& p, const RowsCfg& c) {
    return rows_bps_scheme<T, D, DYN, HJ_ENO2>(p, c);
}
template <typename T, int D, int DYN>
int rows_bps_eno1(const StageParams& p, const RowsCfg& c) {
    return rows_bps_scheme<T, D, DYN, HJ_ENO1>(p, c);
}
template <typename T, int D, int DYN>
int rows_bps_eno3(const StageParams& p, const RowsCfg& c) {
    return rows_bps_scheme<T, D, DYN, HJ_ENO3>(p, c);
}

// Dispatch over the (dimension, dynamics) pairs the row kernel is built for.
#define HJ_ROWS_DISPATCH(FN, T, ...)                                                   \
    switch (p.g.ndim * 16 + p.dynamics) {                                              \
    case 2 * 16 + HJ_DYN_DOUBLE_INTEGRATOR: return FN<T, 2, HJ_DYN_DOUBLE_INTEGRATOR>(__VA_ARGS__); \
    case 2 * 16 + HJ_DYN_NORM: return FN<T, 2, HJ_DYN_NORM>(__VA_ARGS__);             \
    case 2 * 16 + HJ_DYN_ADVECT: return FN<T, 2, HJ_DYN_ADVECT>(__VA_ARGS__);         \
    case 2 * 16 + HJ_DYN_ROTATE: return FN<T, 2, HJ_DYN_ROTATE>(__VA_ARGS__);         \
    case 3 * 16 + HJ_DYN_AIR3D: return FN<T, 3, HJ_DYN_AIR3D>(__VA_ARGS__);           \
    case 3 * 16 + HJ_DYN_ROCKETS: return FN<T, 3, HJ_DYN_ROCKETS>(__VA_ARGS__);       \
    case 3 * 16 + HJ_DYN_NORM: return FN<T, 3, HJ_DYN_NORM>(__VA_ARGS__);             \
    case 3 * 16 + HJ_DYN_ADVECT: return FN<T, 3, HJ_DYN_ADVECT>(__VA_ARGS__);         \
    case 3 * 16 + HJ_DYN_ROTATE: return FN<T, 3, HJ_DYN_ROTATE>(__VA_ARGS__);         \
    case 4 * 16 + HJ_DYN_DUBINS4D: return FN<T, 4, HJ_DYN_DUBINS4D>(__VA_ARGS__);     \
    default: break;                                                                    \
    }

// The variants with dissipation local in p (HJ_ALPHA_BOX) of the dynamics
// whose slopes depend on p; instantiated in translation units of their own.
#define HJ_ROWS_BOX_DISPATCH(FN, T, ...)                                                                  \
    switch (p.g.ndim * 16 + p.dynamics) {                                                                  \
    case 2 * 16 + HJ_DYN_NORM: return FN<T, 2, HJ_DYN_NORM + kDynBox>(__VA_ARGS__);                        \
    case 3 * 16 + HJ_DYN_NORM: return FN<T, 3, HJ_DYN_NORM + kDynBox>(__VA_ARGS__);                        \
    case 3 * 16 + HJ_DYN_AIR3D: return FN<T, 3, HJ_DYN_AIR3D + kDynBox>(__VA_ARGS__);                      \
    case 3 * 16 + HJ_DYN_ROCKETS: return FN<T, 3, HJ_DYN_ROCKETS + kDynBox>(__VA_ARGS__);                  \
    default: break;                                                                                        \
    }


}  // namespace hj

#include "plane_kernel.cuh"
