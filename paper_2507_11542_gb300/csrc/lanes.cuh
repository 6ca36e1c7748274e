// lanes.cuh -- two values side by side, one for each of the two grid rows a
// thread of the row kernel works on. FP32 pairs live in one 64-bit register
// pair and use the packed instructions of this GPU (add, mul and fma on two
// floats at once: the same rate per operation as the scalar ones, half the
// instructions to issue); FP64 pairs are two doubles. FP64 operations round once
// each; of the packed ones only fma2 is a single rounding for certain: a product
// whose only use is a sum may be fused with it, so that code which has to round
// alike in every inlined copy leaves none (weno_iface2).
#pragma once

#include <cuda_runtime.h>

namespace hj {

struct F2 {
    unsigned long long v;
};
struct D2 {
    double a, b;
};
template <typename T> struct LanesOf;
template <> struct LanesOf<float> { using type = F2; };
template <> struct LanesOf<double> { using type = D2; };
template <typename T> using Lanes = typename LanesOf<T>::type;

__device__ __forceinline__ F2 lanes(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lane_a(F2 x) { return __uint_as_float((unsigned)x.v); }
__device__ __forceinline__ float lane_b(F2 x) { return __uint_as_float((unsigned)(x.v >> 32)); }
__device__ __forceinline__ F2 operator+(F2 x, F2 y) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 x, F2 y) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 x, F2 y) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(x.v), "l"(y.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 x, F2 y, F2 z) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(x.v), "l"(y.v), "l"(z.v));
    return r;
}
__device__ __forceinline__ F2 both(float a) { return lanes(a, a); }
__device__ __forceinline__ F2 neg2(F2 x) { return lanes(-lane_a(x), -lane_b(x)); }

__device__ __forceinline__ D2 lanes(double a, double b) { return {a, b}; }
__device__ __forceinline__ double lane_a(D2 x) { return x.a; }
__device__ __forceinline__ double lane_b(D2 x) { return x.b; }
__device__ __forceinline__ D2 operator+(D2 x, D2 y) { return {__dadd_rn(x.a, y.a), __dadd_rn(x.b, y.b)}; }
__device__ __forceinline__ D2 operator-(D2 x, D2 y) { return {__dsub_rn(x.a, y.a), __dsub_rn(x.b, y.b)}; }


// A pair in shared memory (8 or 16 bytes, aligned).
__device__ __forceinline__ F2 lanes_at(const float* p) { return {*reinterpret_cast<const unsigned long long*>(p)}; }
__device__ __forceinline__ D2 lanes_at(const double* p) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ void put_lanes(float* p, F2 x) { *reinterpret_cast<unsigned long long*>(p) = x.v; }
__device__ __forceinline__ void put_lanes(double* p, D2 x) { *reinterpret_cast<double2*>(p) = make_double2(x.a, x.b); }

}  // namespace hj
