// stage_kernels.cuh -- the fused RK stage kernel (Sec. 3-5): for every node,
// ghost-aware 7-point gathers along each dimension, upwind p-/p+ (ENO or
// WENO5), Lax-Friedrichs Hamiltonian, BRT clamp and the TVD-RK3 stage
// combination, in one pass. Included by one translation unit per element type.
#pragma once

#include "stencil.cuh"

namespace hj {

constexpr int kBX = 32, kBY = 8;

// One thread per node. Threads span (i0, i1); blockIdx.z strides over the
// combined index of dimensions 2 and 3.
template <typename T, int D, int SCHEME>
__global__ void __launch_bounds__(kBX * kBY) stage_kernel(const StageParams P) {
    const GridDev& g = P.g;
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
    const int i1 = (D > 1) ? (int)(blockIdx.y * blockDim.y + threadIdx.y) : 0;
    if (i0 >= g.n[0] || (D > 1 && i1 >= g.n[1])) return;
    const int nz = (D > 2 ? g.n[2] : 1) * (D > 3 ? g.n[3] : 1);
    const T* __restrict__ u = static_cast<const T*>(P.u);
    const T* __restrict__ vn = static_cast<const T*>(P.vn);
    T* __restrict__ out = static_cast<T*>(P.out);
    for (int z = blockIdx.z; z < nz; z += gridDim.z) {
        int idx[4] = {i0, i1, 0, 0};
        if (D > 2) { idx[2] = z % g.n[2]; }
        if (D > 3) { idx[3] = z / g.n[2]; }
        long long flat = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) flat += (long long)idx[d] * g.stride[d];
        T pm[D], pp[D];
#pragma unroll
        for (int d = 0; d < D; ++d) {
            T v[7];
            gather7<T>(u, flat, idx[d], g.n[d], g.stride[d], (g.periodic_mask >> d) & 1u, g.extrap, v);
            upwind_pair<T, SCHEME>(v, g.dx[d], 2.0 * P.half_inv_dx6[d], SP<T>::floor(P, d), pm[d], pp[d]);
        }
        T y = lf_term<T, D>(P, idx, pm, pp);
        if (P.brt_min0) y = fmin(y, T(0));
        T r;
        if (P.mode == kTerm) {
            r = y;
        } else {
            const T w = ld(u + flat) + SP<T>::dt(P) * y;
            r = w;
            if (P.has_vn) {
                const T vv = ld(vn + flat);
                if (P.cv != 0.0) r = SP<T>::cv(P) * vv + SP<T>::cu(P) * w;
                if (P.minv_after) r = fmin(r, vv);
            }
        }
        out[flat] = r;
    }
}

// p- and p+ along one dimension, from one interface evaluation for the two nodes
// it separates: interface j (0 .. n of a line of n nodes) gives p- of node j and
// p+ of node j-1, so that no thread needs another's result. A thread walks over
// a run of interfaces of one line (FP32: of two lines, one per lane), which in
// FP64 WENO5 reuse their differences (Weno5Line: 15 FP64 instructions an
// interface, where two one-sided evaluations per node took 50). 101^3 FP64, all
// three dimensions: 318 -> 153 us, 136 with the sums u in integers. The ENO schemes
// work on divided differences, as their definition does (EnoLine).

// FP32 WENO5 of two lines' interfaces (values v) over the whole range of FP32: a
// line whose largest difference is 2 or more has all five scaled by the power of
// two that brings it to [1, 2), and `unit` is what its results then count in.
// Unscaled, the squared smoothness sums leave FP32 from differences of about 3e8
// on. Where they do not the results are the same bits (the epsilon's floor is far
// below the last place of the rest from differences of 1 on).
__device__ __forceinline__ void weno5_lines(const float (&v)[2][6], float* pp, float* pm, float* unit) {
    float e[2][5], by[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        float top = 0.0f;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            e[l][k] = __fadd_rn(v[l][k + 1], -v[l][k]);
            top = fmaxf(top, fabsf(e[l][k]));
        }
        const unsigned x = min(max(__float_as_uint(top) >> 23, 127u), 253u);  // 2^(x - 127) <= top, both powers normal
        unit[l] = __uint_as_float(x << 23);
        by[l] = __uint_as_float((254u - x) << 23);
    }
    F2 d[5], p, m;
#pragma unroll
    for (int k = 0; k < 5; ++k) d[k] = lanes(__fmul_rn(e[0][k], by[0]), __fmul_rn(e[1][k], by[1]));
    weno_iface2(d[0], d[1], d[2], d[3], d[4], p, m);
    pp[0] = lane_a(p);
    pp[1] = lane_b(p);
    pm[0] = lane_a(m);
    pm[1] = lane_b(m);
}

// Node j of a grid line (node 0 at u, stride s), ghost cells included.
template <typename T>
__device__ __forceinline__ T line_node(const T* u, int j, int n, long long s, bool periodic, int extrap) {
    if (j >= 0 && j < n) return ld(u + j * s);
    if (periodic) {
        int w = j % n;
        if (w < 0) w += n;
        return ld(u + w * s);
    }
    const T e = ld(u + (j < 0 ? 0 : n - 1) * s), i = ld(u + (j < 0 ? 1 : n - 2) * s);
    const T slope = (extrap == HJ_EXTRAP_LINEAR) ? (e - i) : fabs(e - i) * sgn(e);
    return add_rn(e, mul_rn(T(j < 0 ? -j : j - (n - 1)), slope));
}

// The derivatives from what an interface evaluation returns (WENO5: six times the
// raw ones, in FP32 in units of weno5_lines; ENO: the derivatives).
template <int SCHEME>
__device__ __forceinline__ float derivative(float r, float unit, const UpwindParams& P) {
    if constexpr (SCHEME == HJ_WENO5) return r * (float)P.inv_6dx * unit;
    else return r;
}
template <int SCHEME>
__device__ __forceinline__ double derivative(double r, double, const UpwindParams& P) {
    if constexpr (SCHEME == HJ_WENO5) return r * P.inv_6dx;
    else return r;
}

constexpr int kUpwindThreads = 128;
constexpr int kUpwindRun = 8;

// FP32 along a dimension of stride 1. The arithmetic is short here and memory is
// the bound: neighbouring threads take neighbouring interfaces, so that a warp
// reads and writes whole lines of memory (with a run of eight interfaces a
// thread, as along the other dimensions, each store of a warp touched 32 sectors).
// All interfaces are numbered one grid line after the other; a thread takes i and
// i + half of them, one per lane, whatever the number of lines (two lines a
// thread did everything twice where there is one). 300^3 along dimension 0: ENO1
// 225 -> 110 us, WENO5 208 -> 168; one line of 20 M nodes: 298 -> 81 and 294 -> 102.
template <int SCHEME>
__global__ void __launch_bounds__(kUpwindThreads) upwind_row_kernel(const UpwindParams P, const long long half,
                                                                    const long long half_line, const int half_j) {
    const int n = P.g.n[P.dim];
    const bool periodic = (P.g.periodic_mask >> P.dim) & 1u;
    const float* __restrict__ u = static_cast<const float*>(P.u);
    float* __restrict__ pm = static_cast<float*>(P.pm);
    float* __restrict__ pp = static_cast<float*>(P.pp);
    grid_wait();
    const long long i = (long long)blockIdx.x * kUpwindThreads + threadIdx.x;
    if (i >= half) return;
    // line and interface of i, and of i + half from them (half = half_line lines and half_j)
    long long line[2];
    int j[2];
    if (half < (1LL << 31)) {
        line[0] = (unsigned)i / (unsigned)(n + 1);
        j[0] = (int)((unsigned)i - (unsigned)line[0] * (unsigned)(n + 1));
    } else {
        line[0] = i / (n + 1);
        j[0] = (int)(i - line[0] * (n + 1));
    }
    line[1] = line[0] + half_line;
    j[1] = j[0] + half_j;
    if (j[1] > n) {
        j[1] -= n + 1;
        ++line[1];
    }
    const long long lines = P.g.total / n;
    const bool two = line[1] < lines;  // an odd number of interfaces: the last thread's first one twice
    if (!two) {
        line[1] = line[0];
        j[1] = j[0];
    }
    constexpr int kFrom = SCHEME == HJ_ENO1 ? 2 : SCHEME == HJ_ENO2 ? 1 : 0;  // the values it reads: kFrom .. 5 - kFrom
    float v[2][6] = {}, left[2], right[2], unit[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const float* row = u + line[l] * n;
        if (j[l] >= 3 && j[l] + 3 <= n) {
#pragma unroll
            for (int k = kFrom; k < 6 - kFrom; ++k) v[l][k] = ld(row + (j[l] - 3 + k));
        } else {
#pragma unroll
            for (int k = kFrom; k < 6 - kFrom; ++k) v[l][k] = line_node(row, j[l] - 3 + k, n, 1LL, periodic, P.g.extrap);
        }
    }
    if constexpr (SCHEME == HJ_WENO5) {
        weno5_lines(v, right, left, unit);
    } else {
        const EnoSpacing<float> h((float)P.dx);
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            EnoLine<float, SCHEME> e;
            e.start(v[l], h);
            e.eval(h, right[l], left[l]);
        }
    }
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        if (l == 1 && !two) break;
        const long long at = line[l] * n + j[l];
        if (j[l] < n) pm[at] = derivative<SCHEME>(left[l], unit[l], P);
        if (j[l] > 0) pp[at - 1] = derivative<SCHEME>(right[l], unit[l], P);
    }
}

template <typename T, int SCHEME>
__global__ void __launch_bounds__(kUpwindThreads) upwind_kernel(const UpwindParams P) {
    constexpr int kLines = sizeof(T) == 4 ? 2 : 1;
    const int d = P.dim, n = P.g.n[d];
    const long long s = P.g.stride[d], lines = P.g.total / n, group = (lines + kLines - 1) / kLines;
    const int runs = (n + 1 + kUpwindRun - 1) / kUpwindRun;
    const bool periodic = (P.g.periodic_mask >> d) & 1u;
    const T* __restrict__ u = static_cast<const T*>(P.u);
    T* __restrict__ pm = static_cast<T*>(P.pm);
    T* __restrict__ pp = static_cast<T*>(P.pp);
    [[maybe_unused]] const T floor = T(P.weno_floor);
    [[maybe_unused]] const EnoSpacing<T> h(T(P.dx));
    grid_wait();
    const long long item = (long long)blockIdx.x * kUpwindThreads + threadIdx.x;
    if (item >= group * runs) return;
    // neighbouring threads: neighbouring runs of a row along dimension 0, else neighbouring lines
    const long long line = d == 0 ? item / runs : item % group;
    const int j0 = kUpwindRun * (int)(d == 0 ? item % runs : item / group);
    const int j1 = min(j0 + kUpwindRun, n + 1);
    long long base[kLines];
#pragma unroll
    for (int l = 0; l < kLines; ++l) {
        const long long k = min(line + l * group, lines - 1);  // a last odd line is done twice
        base[l] = k / s * (s * n) + k % s;
    }
    const auto at = [&](long long b, int j) -> T { return line_node(u + b, j, n, s, periodic, P.g.extrap); };
    [[maybe_unused]] T unit[kLines];  // FP32 WENO5: of the last results (weno5_lines)
    auto store = [&](int j, const T* left, const T* right) {  // interface j: right = p+ of node j-1, left = p- of node j
#pragma unroll
        for (int l = 0; l < kLines; ++l) {
            if (j < n) pm[base[l] + j * s] = derivative<SCHEME>(left[l], unit[l], P);
            if (j > 0) pp[base[l] + (j - 1) * s] = derivative<SCHEME>(right[l], unit[l], P);
        }
    };
    T v[kLines][6];  // nodes j-3 .. j+2
#pragma unroll
    for (int l = 0; l < kLines; ++l)
#pragma unroll
        for (int k = 0; k < 6; ++k) v[l][k] = at(base[l], j0 - 3 + k);
    constexpr bool kWeno64 = SCHEME == HJ_WENO5 && sizeof(T) == 8;
    [[maybe_unused]] Weno5Line walk;
    [[maybe_unused]] EnoLine<T, SCHEME> eno[kLines];
    if constexpr (kWeno64) {
        walk.start(v[0][0], v[0][1], v[0][2], v[0][3], v[0][4], v[0][5]);
    } else if constexpr (SCHEME != HJ_WENO5) {
#pragma unroll
        for (int l = 0; l < kLines; ++l) eno[l].start(v[l], h);
    }
#pragma unroll 1
    for (int j = j0;; ++j) {
        T left[kLines], right[kLines], next[kLines];
        const bool more = j + 1 < j1;
        if (more) {
#pragma unroll
            for (int l = 0; l < kLines; ++l) next[l] = at(base[l], j + 3);
        }
        if constexpr (kWeno64) {
            walk.eval(floor, right[0], left[0]);
        } else if constexpr (SCHEME == HJ_WENO5) {
            weno5_lines(v, right, left, unit);
        } else {
#pragma unroll
            for (int l = 0; l < kLines; ++l) eno[l].eval(h, right[l], left[l]);
        }
        store(j, left, right);
        if (!more) break;
        if constexpr (kWeno64) {
            walk.slide(v[0][5], next[0]);
            v[0][5] = next[0];
        } else if constexpr (SCHEME == HJ_WENO5) {
#pragma unroll
            for (int l = 0; l < kLines; ++l) {
#pragma unroll
                for (int k = 0; k < 5; ++k) v[l][k] = v[l][k + 1];
                v[l][5] = next[l];
            }
        } else {
#pragma unroll
            for (int l = 0; l < kLines; ++l) eno[l].slide(next[l], h);
        }
    }
}

inline void launch_shape(const GridDev& g, dim3& grid, dim3& block) {
    if (g.ndim == 1) {
        block = dim3(kBX * kBY, 1, 1);
        grid = dim3((unsigned)((g.n[0] + kBX * kBY - 1) / (kBX * kBY)), 1, 1);
        return;
    }
    block = dim3(kBX, kBY, 1);
    long long nz = 1;
    for (int d = 2; d < g.ndim; ++d) nz *= g.n[d];
    grid = dim3((unsigned)((g.n[0] + kBX - 1) / kBX), (unsigned)((g.n[1] + kBY - 1) / kBY),
                (unsigned)(nz < 65535 ? nz : 65535));
}

template <typename T, int SCHEME>
cudaError_t launch_stage_scheme(const StageParams& p, cudaStream_t s) {
    dim3 grid, block;
    launch_shape(p.g, grid, block);
    switch (p.g.ndim) {
    case 1: stage_kernel<T, 1, SCHEME><<<grid, block, 0, s>>>(p); break;
    case 2: stage_kernel<T, 2, SCHEME><<<grid, block, 0, s>>>(p); break;
    case 3: stage_kernel<T, 3, SCHEME><<<grid, block, 0, s>>>(p); break;
    case 4: stage_kernel<T, 4, SCHEME><<<grid, block, 0, s>>>(p); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_stage_t(const StageParams& p, int scheme, cudaStream_t s) {
    switch (scheme) {
    case HJ_ENO1: return launch_stage_scheme<T, HJ_ENO1>(p, s);
    case HJ_ENO2: return launch_stage_scheme<T, HJ_ENO2>(p, s);
    case HJ_ENO3: return launch_stage_scheme<T, HJ_ENO3>(p, s);
    case HJ_WENO5: return launch_stage_scheme<T, HJ_WENO5>(p, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T, int SCHEME>
cudaError_t launch_upwind_scheme(const UpwindParams& p, cudaStream_t s) {
    const long long n = p.g.n[p.dim], lines = p.g.total / n, group = sizeof(T) == 4 ? (lines + 1) / 2 : lines;
    if constexpr (sizeof(T) == 4) {
        if (p.g.stride[p.dim] == 1) {
            const long long half = (lines * (n + 1) + 1) / 2;
            return launch_dependent(upwind_row_kernel<SCHEME>,
                                    dim3((unsigned)((half + kUpwindThreads - 1) / kUpwindThreads)), dim3(kUpwindThreads), 0,
                                    s, p, half, half / (n + 1), (int)(half % (n + 1)));
        }
    }
    const long long items = group * ((n + 1 + kUpwindRun - 1) / kUpwindRun);
    return launch_dependent(upwind_kernel<T, SCHEME>, dim3((unsigned)((items + kUpwindThreads - 1) / kUpwindThreads)),
                            dim3(kUpwindThreads), 0, s, p);
}

template <typename T>
cudaError_t launch_upwind_t(const UpwindParams& p, int scheme, cudaStream_t s) {
    switch (scheme) {
    case HJ_ENO1: return launch_upwind_scheme<T, HJ_ENO1>(p, s);
    case HJ_ENO2: return launch_upwind_scheme<T, HJ_ENO2>(p, s);
    case HJ_ENO3: return launch_upwind_scheme<T, HJ_ENO3>(p, s);
    case HJ_WENO5: return launch_upwind_scheme<T, HJ_WENO5>(p, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hj
