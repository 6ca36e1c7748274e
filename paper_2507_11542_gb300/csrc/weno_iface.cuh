// weno_iface.cuh -- WENO5 (Sec. 3.3; Jiang & Peng 2000) evaluated per grid
// interface. The right derivative p+ at node j and the left derivative p- at
// node j+1 use the same five differences
//   e1..e5 = v_{j-1}-v_{j-2}, v_j-v_{j-1}, v_{j+1}-v_j, v_{j+2}-v_{j+1}, v_{j+3}-v_{j+2}
// (mirrored), hence the same three smoothness indicators and epsilon; only
// the candidate stencils and the order of the ideal weights differ:
//
//   windows A = (e1,e2,e3), B = (e2,e3,e4), C = (e3,e4,e5)
//   SA = 13/12 (e1-2e2+e3)^2 + 1/4 (e1-4e2+3e3)^2
//   SB = 13/12 (e2-2e3+e4)^2 + 1/4 (e2-e4)^2
//   SC = 13/12 (e3-2e4+e5)^2 + 1/4 (3e3-4e4+e5)^2
//   eps = 1e-6 max(e_k^2) + floor
//   p-_{j+1} = sum_k w_k phi_k, phi = (2e1-7e2+11e3, -e2+5e3+2e4, 2e3+5e4-e5)/6,
//              w ~ (0.1, 0.6, 0.3) / (S+eps)^2 over (SA, SB, SC)
//   p+_j     = sum_k w_k psi_k, psi = (2e5-7e4+11e3, -e4+5e3+2e2, 2e3+5e2-e1)/6,
//              w ~ (0.1, 0.6, 0.3) / (S+eps)^2 over (SC, SB, SA)
//
// Evaluated here in an equivalent form (the weights sum to one):
//   p- = phi2 + (w1 T1/3 + w3 T2/6),   p+ = psi2 - (w1' T2/3 + w3' T1/6)
// with the third differences T1 = e1-3e2+3e3-e4 = tA-tB and T2 = e2-3e3+3e4-e5
// = tB-tC shared by both sides. The smoothness indicators are scaled by 4
// (S' = 13/3 t^2 + u^2), eps alike, and the ideal weights by 10, which leaves
// every weight unchanged; both results come out times 6. All differences and
// both results are raw (not divided by dx): the caller scales them once per
// node and dimension, by 1/(12 dx) (iface_times6).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "../../include/hj.h"
#include "hj_internal.h"
#include "lanes.cuh"
#include "weno_weights64.cuh"

namespace hj {

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// FP32, two interfaces at a time (one per lane), rescaled in ways that leave
// every weight unchanged: smoothness values and epsilon times 4 (S' = 13/3 t^2
// + u^2), ideal weights times 10; results times 6 (the caller divides the 6 out
// with 1/(2 dx)), written around the interface's own difference as in FP64
// below. One reciprocal per weight and per side: (S' + eps')^2 >= (4e-18)^2
// stays a normal number, so the approximate reciprocals neither overflow nor
// divide by zero.
//
// The FP32 kernels are bound by instruction issue: 42 packed instructions, 10
// reciprocals and 12 scalar ones for both interfaces, where one alone took 57
// and 5 reciprocals with scalar instructions. A packed constant is a register
// pair, so the formulas get by with three (2, 6, 13/3), and use sums where they
// can: with m = e2 - e4 = -(d23 + d34), 2 d34 + d23 = d34 - m and -(2 d23 + d34)
// = m - d23; squares take either sign. No product's only use is a sum: packed
// products and sums are contracted too, and each inlined copy has to round
// alike.
__device__ __forceinline__ float eps_of(float e1, float e2, float e3, float e4, float e5) {
    const float a = fmaxf(fmaxf(fabsf(e1), fabsf(e2)), fabsf(e3));
    const float amax = fmaxf(fmaxf(a, fabsf(e4)), fabsf(e5));
    return __fmaf_rn(__fmul_rn(4e-6f, amax), amax, 4.0f * kWenoFloorF32);
}
__device__ __forceinline__ F2 rcp2(F2 x) { return lanes(rcp_approx(lane_a(x)), rcp_approx(lane_b(x))); }

__device__ __forceinline__ void weno_iface2(F2 e1, F2 e2, F2 e3, F2 e4, F2 e5, F2& pp_j, F2& pm_j1) {
    const F2 two = both(2.0f), six = both(6.0f), c133 = both(13.0f / 3.0f);
    const F2 d12 = e2 - e1, d23 = e3 - e2, d34 = e4 - e3, d45 = e5 - e4;
    const F2 tA = d23 - d12, tB = d34 - d23, nC = d34 - d45;  // nC = -tC
    const F2 uA = fma2(two, d23, tA);  // e1 - 4e2 + 3e3
    const F2 m = e2 - e4;
    const F2 uC = fma2(two, d34, nC);  // -(3e3 - 4e4 + e5)
    const F2 eps = lanes(eps_of(lane_a(e1), lane_a(e2), lane_a(e3), lane_a(e4), lane_a(e5)),
                         eps_of(lane_b(e1), lane_b(e2), lane_b(e3), lane_b(e4), lane_b(e5)));
    const F2 sA = fma2(uA, uA, fma2(c133 * tA, tA, eps));
    const F2 sB = fma2(m, m, fma2(c133 * tB, tB, eps));
    const F2 sC = fma2(uC, uC, fma2(c133 * nC, nC, eps));
    const F2 rA = rcp2(sA * sA), rB = rcp2(sB * sB), rC = rcp2(sC * sC);
    const F2 T1 = tA - tB, T2 = tB + nC;
    const F2 X = rA * T1, Y = rC * T2;
    const F2 XY = fma2(rA, T1, Y);
    const F2 numL = fma2(two, XY, Y);  // 2X + 3Y
    const F2 numR = fma2(two, XY, X);  // 3X + 2Y
    const F2 all = fma2(six, rB, rA + rC);
    const F2 DL = fma2(two, rC, all), DR = fma2(two, rA, all);
    const F2 sL = fma2(numL, rcp2(DL), d34 - m);
    const F2 sR = fma2(numR, neg2(rcp2(DR)), m - d23);
    pm_j1 = fma2(six, e3, sL);
    pp_j = fma2(six, e3, sR);
}

// 1/x for a positive normal double: the hardware estimate refined by two
// Newton-Raphson steps r <- r + r (1 - x r) (each squares the relative error).
// Nothing in the library calls it since the interface's reciprocals are integer;
// its test (test_gpu_rcp.py) does.
__device__ __forceinline__ double rcp_newton(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = fma(-x, r, 1.0);
    r = fma(r, e, r);
    e = fma(-x, r, 1.0);
    return fma(r, e, r);
}

// FP64. The first, second and third differences and the two results are FP64,
// the weights 64-bit integer arithmetic (weno_weights64.cuh, which takes the
// smoothness sums times 12 and the ideal weights times 10: both leave every
// weight unchanged). Both results are times 6, written around the interface's
// own difference so that one rounding alone happens at their magnitude:
//   6 p- = 6 e3 + (2 d34 + d23 + l1 T1 + l3 T2)
//   6 p+ = 6 e3 - (2 d23 + d34 + r1 T1 + r3 T2)
// with d23 = e3 - e2, d34 = e4 - e3 and the weights l1 = 2 w1, l3 = w3 (left),
// r1 = w3', r3 = 2 w1' (right). The caller divides the 6 out with its
// 1/(2 dx) (iface_times6). A non-finite difference reaches both results
// through T1 or T2, since the weights are finite whatever their input.
//
// The FP64 pipe bounds this (16-20 cycles a warp instruction and SM): 22 FP64
// instructions from five first differences, 12 along a line (Weno5Line), where
// the weights in FP64 took 64 and 50 (measured cycles per warp and SM in
// weno_weights64.cuh).
// The core takes what consecutive interfaces along a line share: tA, tB, tC
// (the second differences of the windows' first differences), d23, d34 and the
// third differences T1 = tA - tB, T2 = tB - tC. floor12: 12 times the epsilon
// floor. No a*b + c is left for the compiler to contract, so every inlined
// copy rounds alike and results do not depend on which thread role evaluates
// an interface.
__device__ __forceinline__ void weno_core(double e1, double e2, double e3, double e4, double e5, double tA, double tB,
                                          double tC, double d23, double d34, double T1, double T2, double floor12,
                                          double& pp_j, double& pm_j1) {
    const w64::u64 amax = w64::umax(w64::umax(w64::umax(w64::abs_bits(e1), w64::abs_bits(e2)),
                                              w64::umax(w64::abs_bits(e3), w64::abs_bits(e4))), w64::abs_bits(e5));
    const w64::Sum eps = w64::eps_sum(amax, w64::floor_term(floor12));
    double l1, l3, r1, r3;
    // u: tA + 2 d23 = e1 - 4e2 + 3e3, d23 + d34 = e4 - e2, tC - 2 d34 = 3e3 - 4e4 + e5
    const w64::Parts pA = w64::parts(tA), pB = w64::parts(tB), pC = w64::parts(tC), p23 = w64::parts(d23),
                     p34 = w64::parts(d34);
    w64::weights(w64::smooth_sum(pA, pA, p23, 1, 0u, eps), w64::smooth_sum(pB, p23, p34, 0, 0u, eps),
                 w64::smooth_sum(pC, pC, p34, 1, ~0u, eps), l1, l3, r1, r3);
    const double sL = fma(l3, T2, fma(l1, T1, fma(2.0, d34, d23)));
    const double sR = fma(r3, T2, fma(r1, T1, fma(2.0, d23, d34)));
    pm_j1 = fma(6.0, e3, sL);
    pp_j = fma(6.0, e3, -sR);
}

// Six times the FP64 one-sided derivatives (weno_core), from the five first
// differences: t as differences of the d = e_{k+1} - e_k.
__device__ __forceinline__ void weno_iface(double e1, double e2, double e3, double e4, double e5, double floor12,
                                           double& pp_j, double& pm_j1) {
    const double d12 = e2 - e1, d23 = e3 - e2, d34 = e4 - e3, d45 = e5 - e4;
    const double tA = d23 - d12, tB = d34 - d23, tC = d45 - d34;
    weno_core(e1, e2, e3, e4, e5, tA, tB, tC, d23, d34, tA - tB, tB - tC, floor12, pp_j, pm_j1);
}

// Whether an interface evaluation returns six times the derivatives (WENO5,
// both precisions; the caller scales by 1/(12 dx) instead of 1/(2 dx)) or the
// derivatives themselves (the ENO schemes).
template <typename T, int SCHEME>
__host__ __device__ constexpr bool iface_times6() {
    return SCHEME == HJ_WENO5;
}

// FP64 WENO5 along a grid line, one interface after the other: the interface
// between nodes j and j+1 reuses four of the five first differences, two of
// the three differences d, two of the three values tA, tB, tC and one of the
// two third differences of the interface before it, so each step computes one
// of each. The results are those of weno_iface, bit for bit (the same
// operations on the same operands).
struct Weno5Line {
    double e[5];   // first differences of the current window
    double d[3];   // d23, d34, d45: differences of consecutive e
    double t[3];   // tA, tB, tC
    double T[2];   // T1, T2
    // the window of the values v0..v5 at nodes j-2 .. j+3
    __device__ __forceinline__ void start(double v0, double v1, double v2, double v3, double v4, double v5) {
        e[0] = v1 - v0; e[1] = v2 - v1; e[2] = v3 - v2; e[3] = v4 - v3; e[4] = v5 - v4;
        const double d12 = e[1] - e[0];
        d[0] = e[2] - e[1]; d[1] = e[3] - e[2]; d[2] = e[4] - e[3];
        t[0] = d[0] - d12; t[1] = d[1] - d[0]; t[2] = d[2] - d[1];
        T[0] = t[0] - t[1]; T[1] = t[1] - t[2];
    }
    // slide by one node: v4, v5 are the values at the new window's last two nodes
    __device__ __forceinline__ void slide(double v4, double v5) {
        e[0] = e[1]; e[1] = e[2]; e[2] = e[3]; e[3] = e[4]; e[4] = v5 - v4;
        d[0] = d[1]; d[1] = d[2]; d[2] = e[4] - e[3];
        t[0] = t[1]; t[1] = t[2]; t[2] = d[2] - d[1];
        T[0] = T[1]; T[1] = t[1] - t[2];
    }
    __device__ __forceinline__ void eval(double floor12, double& pp_j, double& pm_j1) const {
        weno_core(e[0], e[1], e[2], e[3], e[4], t[0], t[1], t[2], d[0], d[1], T[0], T[1], floor12, pp_j, pm_j1);
    }
};

// Second-order ENO (Sec. 3.2; Osher & Fedkiw 2003 Sec. 3.3) per interface.
// Both one-sided derivatives at the interface between nodes j and j+1 (p+ of
// j and p- of j+1) take the stencil that starts at j: the first difference
// across the interface plus or minus half the smaller (in magnitude; ties to
// the left) of the second differences centred at j and j+1. In raw
// (undivided) units, from the values v0..v3 at nodes j-1 .. j+2:
//   e = v2 - v1, dL = e - (v1 - v0), dR = (v3 - v2) - e,
//   c = |dL| <= |dR| ? dL : dR,  p+_j = e - c/2,  p-_{j+1} = e + c/2.
// |a| <= |b|: for FP64 on the bit patterns (an integer comparison, exact for
// finite values; the sign is masked in the high word, see w64::abs_bits).
__device__ __forceinline__ bool abs_le(double a, double b) {
    return w64::abs_bits(a) <= w64::abs_bits(b);
}
__device__ __forceinline__ bool abs_le(float a, float b) { return fabsf(a) <= fabsf(b); }

template <typename T>
__device__ __forceinline__ void eno2_iface(T v0, T v1, T v2, T v3, T& pp_j, T& pm_j1) {
    const T e = v2 - v1;
    const T dL = e - (v1 - v0);
    const T dR = (v3 - v2) - e;
    const T c = abs_le(dL, dR) ? dL : dR;
    pp_j = e - T(0.5) * c;
    pm_j1 = e + T(0.5) * c;
}

// FP64 ENO2 along a grid line: each interface takes two of its three first and
// one of its two second differences from the one below it (4 FP64 instructions
// instead of 7), the results of eno2_iface bit for bit.
struct Eno2Line {
    double e, r, dR;  // v2 - v1, v3 - v2, and the second difference between them
    double dL;
    // the window of the values v0..v3 at nodes j-1 .. j+2
    __device__ __forceinline__ void start(double v0, double v1, double v2, double v3) {
        e = v2 - v1;
        r = v3 - v2;
        dL = e - (v1 - v0);
        dR = r - e;
    }
    // slide by one node: v3, v4 are the values at the new window's last two nodes
    __device__ __forceinline__ void slide(double v3, double v4) {
        e = r;
        dL = dR;
        r = v4 - v3;
        dR = r - e;
    }
    __device__ __forceinline__ void eval(double& pp_j, double& pm_j1) const {
        const double c = abs_le(dL, dR) ? dL : dR;
        pp_j = fma(-0.5, c, e);
        pm_j1 = fma(0.5, c, e);
    }
};

// Third-order ENO (Sec. 3.2; Osher & Fedkiw 2003 Sec. 3.3) per interface.
// p+ of node j and p- of node j+1 both start from k = j, so they take the
// same second-difference choice (c; k* = j-1 on the left, else j) and the
// same third-difference choice (c*, the smaller of the two differences next
// to k*; ties to the left); only the polynomial coefficients differ. In raw
// units, from e_m = v_{m+1} - v_m, second differences d2_m = e_m - e_{m-1}
// and third differences d3 = d2_{m+1} - d2_m (the divided differences are
// e/dx, d2/(2 dx^2), d3/(6 dx^3)):
//   p+_j     = e_j - c/2 + c* (left ? -1 : 2)/6
//   p-_{j+1} = e_j + c/2 + c* (left ? 2 : -1)/6
// from the values v0..v5 at nodes j-2 .. j+3.
template <typename T>
__device__ __forceinline__ void eno3_iface(T v0, T v1, T v2, T v3, T v4, T v5, T& pp_j, T& pm_j1) {
    const T e0 = v1 - v0, e1 = v2 - v1, e2 = v3 - v2, e3 = v4 - v3, e4 = v5 - v4;
    const T dm = e1 - e0, d0 = e2 - e1, d1 = e3 - e2, d2 = e4 - e3;  // second differences at j-1, j, j+1, j+2
    const bool left = abs_le(d0, d1);
    const T c = left ? d0 : d1;
    const T a = left ? d0 - dm : d1 - d0;  // third differences next to k*
    const T b = left ? d1 - d0 : d2 - d1;
    const T cs = abs_le(a, b) ? a : b;
    const T third = cs * T(1.0 / 6.0);
    pp_j = e2 - T(0.5) * c + (left ? -third : T(2) * third);
    pm_j1 = e2 + T(0.5) * c + (left ? T(2) * third : -third);
}

// Two interfaces at a time, one per lane: w0..w5 hold the values at the nodes
// j-2 .. j+3 of each (WENO5 and ENO3 read all six, ENO2 the middle four, ENO1
// the middle two: first order takes the difference across the interface for
// both sides).
template <int SCHEME>
__device__ __forceinline__ void iface_lanes(const F2 w[6], float, F2& pp, F2& pm) {
    if constexpr (SCHEME == HJ_WENO5) {
        weno_iface2(w[1] - w[0], w[2] - w[1], w[3] - w[2], w[4] - w[3], w[5] - w[4], pp, pm);
    } else if constexpr (SCHEME == HJ_ENO1) {
        pp = pm = w[3] - w[2];
    } else {
        float pa, pb, ma, mb;
        if constexpr (SCHEME == HJ_ENO2) {
            eno2_iface(lane_a(w[1]), lane_a(w[2]), lane_a(w[3]), lane_a(w[4]), pa, ma);
            eno2_iface(lane_b(w[1]), lane_b(w[2]), lane_b(w[3]), lane_b(w[4]), pb, mb);
        } else {
            eno3_iface(lane_a(w[0]), lane_a(w[1]), lane_a(w[2]), lane_a(w[3]), lane_a(w[4]), lane_a(w[5]), pa, ma);
            eno3_iface(lane_b(w[0]), lane_b(w[1]), lane_b(w[2]), lane_b(w[3]), lane_b(w[4]), lane_b(w[5]), pb, mb);
        }
        pp = lanes(pa, pb);
        pm = lanes(ma, mb);
    }
}
template <int SCHEME>
__device__ __forceinline__ void iface_lanes(const D2 w[6], double floor12, D2& pp, D2& pm) {
    if constexpr (SCHEME == HJ_WENO5) {
        weno_iface(w[1].a - w[0].a, w[2].a - w[1].a, w[3].a - w[2].a, w[4].a - w[3].a, w[5].a - w[4].a, floor12, pp.a,
                   pm.a);
        weno_iface(w[1].b - w[0].b, w[2].b - w[1].b, w[3].b - w[2].b, w[4].b - w[3].b, w[5].b - w[4].b, floor12, pp.b,
                   pm.b);
    } else if constexpr (SCHEME == HJ_ENO1) {
        pp = pm = w[3] - w[2];
    } else if constexpr (SCHEME == HJ_ENO2) {
        eno2_iface(w[1].a, w[2].a, w[3].a, w[4].a, pp.a, pm.a);
        eno2_iface(w[1].b, w[2].b, w[3].b, w[4].b, pp.b, pm.b);
    } else {
        eno3_iface(w[0].a, w[1].a, w[2].a, w[3].a, w[4].a, w[5].a, pp.a, pm.a);
        eno3_iface(w[0].b, w[1].b, w[2].b, w[3].b, w[4].b, w[5].b, pp.b, pm.b);
    }
}

// Two consecutive interfaces along a line from its seven values v0..v6 (lane a:
// the interface v0..v5, lane b: v1..v6); FP64 WENO5 shares their differences
// (9 of 14 each), with the same results bit for bit.
template <int SCHEME>
__device__ __forceinline__ void iface_line(const float v[7], float floor, F2& pp, F2& pm) {
    F2 w[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = lanes(v[k], v[k + 1]);
    iface_lanes<SCHEME>(w, floor, pp, pm);
}
template <int SCHEME>
__device__ __forceinline__ void iface_line(const double v[7], double floor12, D2& pp, D2& pm) {
    if constexpr (SCHEME == HJ_WENO5) {
        Weno5Line line;
        line.start(v[0], v[1], v[2], v[3], v[4], v[5]);
        line.eval(floor12, pp.a, pm.a);
        line.slide(v[5], v[6]);
        line.eval(floor12, pp.b, pm.b);
    } else {
        D2 w[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = lanes(v[k], v[k + 1]);
        iface_lanes<SCHEME>(w, floor12, pp, pm);
    }
}

// One interface (FP64) or two (FP32, one per lane) from the values at six nodes.
template <int SCHEME>
__device__ __forceinline__ void iface_item(const double (&v)[1][6], double floor12, double* pp, double* pm) {
    const double* w = v[0];
    if constexpr (SCHEME == HJ_WENO5)
        weno_iface(w[1] - w[0], w[2] - w[1], w[3] - w[2], w[4] - w[3], w[5] - w[4], floor12, *pp, *pm);
    else if constexpr (SCHEME == HJ_ENO1) *pp = *pm = __dsub_rn(w[3], w[2]);
    else if constexpr (SCHEME == HJ_ENO2) eno2_iface(w[1], w[2], w[3], w[4], *pp, *pm);
    else eno3_iface(w[0], w[1], w[2], w[3], w[4], w[5], *pp, *pm);
}
template <int SCHEME>
__device__ __forceinline__ void iface_item(const float (&v)[2][6], float floor, float* pp, float* pm) {
    F2 w[6], p, m;
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = lanes(v[0][k], v[1][k]);
    iface_lanes<SCHEME>(w, floor, p, m);
    pp[0] = lane_a(p);
    pp[1] = lane_b(p);
    pm[0] = lane_a(m);
    pm[1] = lane_b(m);
}

}  // namespace hj
