// weno_weights64.cuh -- the nonlinear WENO5 weights of FP64 data in 64-bit
// integer arithmetic (Sec. 3.3; formulas at the top of weno_iface.cuh).
//
// Why: this GPU issues one FP64 warp instruction per SM every 16 to 20 cycles,
// in which the four schedulers issue 64 to 80 others. An interface's weights
// are the bulk of its arithmetic, and they are products, sums of positive
// numbers and two reciprocals: with 63-bit integer mantissas and integer
// exponents they need no FP64 instruction. Products are good to 2^-58, smoothness
// sums to 2^-54 and the weights to a few units of 2^-53 (2.3 at most against exact
// rationals; 2^-51 is what the sums' error allows). Measured on a sweep over columns in L2, SM
// cycles per warp interface: from six values 1272 with FP64 weights and 460 with
// these, along a line (Weno5Line) 1009 and 298.
//
// A number is a mantissa m < 2^63 and an exponent x; products drop the low
// partial product (an error below two units of a result of at least 2^58).
// Every function runs on the host as well (for the test against exact weights).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define HJ_W64 __host__ __device__ __forceinline__
#else
#define HJ_W64 inline
#endif

namespace hj {
namespace w64 {

typedef uint32_t u32;
typedef uint64_t u64;

HJ_W64 u32 hi(u64 a) { return (u32)(a >> 32); }
HJ_W64 u32 lo(u64 a) { return (u32)a; }
HJ_W64 u64 wide(u32 a, u32 b) { return (u64)a * b; }
HJ_W64 int imin(int a, int b) { return a < b ? a : b; }
HJ_W64 int imax(int a, int b) { return a > b ? a : b; }

HJ_W64 u64 bits(double d) {
#ifdef __CUDA_ARCH__
    return (u64)(u32)__double2loint(d) | (u64)(u32)__double2hiint(d) << 32;
#else
    u64 b;
    std::memcpy(&b, &d, 8);
    return b;
#endif
}
HJ_W64 double value(u64 b) {
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi(b), (int)lo(b));
#else
    double d;
    std::memcpy(&d, &b, 8);
    return d;
#endif
}
// leading zeros of a nonzero word
HJ_W64 int clz(u32 a) {
#ifdef __CUDA_ARCH__
    return __clz((int)a);
#else
    return __builtin_clz(a);
#endif
}
// |d| as bits. On the high word: the compiler turns a 64-bit mask into |x|,
// which it computes with an FP64 addition.
HJ_W64 u64 abs_bits(double d) {
#ifdef __CUDA_ARCH__
    return (u64)(u32)__double2loint(d) | (u64)(u32)(__double2hiint(d) & 0x7fffffff) << 32;
#else
    return bits(d) & 0x7fffffffffffffffull;
#endif
}
HJ_W64 u64 umax(u64 a, u64 b) { return a > b ? a : b; }

// mantissa of a double in [2^62, 2^63) and its biased exponent (the sign is
// ignored; zero and denormal values count as some number below 2^-1021, far
// below the epsilon floor wherever they are used)
HJ_W64 u64 mant(u64 b) { return ((b << 10) & 0x3fffffffffffffffull) | 0x4000000000000000ull; }
HJ_W64 int expo(u64 b) { return (int)((hi(b) >> 20) & 0x7ff); }

// a b / 2^64 for a, b < 2^63 (error below two units)
HJ_W64 u64 mulhi(u64 a, u64 b) {
    const u64 c = wide(hi(a), lo(b)) + wide(lo(a), hi(b));
    return wide(hi(a), hi(b)) + hi(c);
}
HJ_W64 u64 sqrhi(u64 a) {
    const u64 c = wide(hi(a) + hi(a), lo(a));
    return wide(hi(a), hi(a)) + hi(c);
}

// bits of about 1/f (f in (1, 2]), within a few units of 2^-24
HJ_W64 u32 rcp_seed(u32 f) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
    return __float_as_uint(r);
#else
    float x;
    std::memcpy(&x, &f, 4);
    x = 1.0f / x;
    std::memcpy(&f, &x, 4);
    return f;
#endif
}

// 2^125 / D for D in [2^62, 2^63), in (2^62, 2^63], relative error about
// 2^-60: an estimate r0 from below (four units of the FP32 estimate taken
// off), then r0 (1 + e + e^2) with e = 1 - d r0 in (0, 2^-20).
HJ_W64 u64 recip(u64 D) {
    const u32 f = (hi(D) >> 7) + 0x3f000000u;                   // the float with D's leading 24 bits, in [1, 2)
    const u32 r0 = (rcp_seed(f | 1u) << 8 | 0x80000000u) - 0x400u;  // times 2^-32
    const u64 h = wide(hi(D), r0) + hi(wide(lo(D), r0));        // d r0 2^62
    const u64 e = (1ull << 62) - h;                             // below 2^42
    const u32 es = (u32)(e >> 10);
    const u64 f2 = (e + (hi(wide(es, es)) >> 10)) << 22;        // (e + e^2) 2^84
    const u64 g = wide(r0, hi(f2)) + hi(wide(r0, lo(f2)));
    return ((u64)r0 << 31) + (g >> 21);
}

// m 2^x as a double, rounded to nearest, for m in [2^53, 2^64)
HJ_W64 double pack(u64 m, int x) {
    const int lz = clz(hi(m));
    const u64 q = ((m >> (10 - lz)) + 1) >> 1;  // 53 bits (2^53 after a carry: the exponent takes it)
    return value(q + ((u64)(u32)(x - lz + 1085) << 52));
}

// A smoothness sum: m in [2^61, 2^63), value m 2^x in the unit of eps_sum.
struct Sum {
    u64 m;
    int x;
};

// The additive floor of the epsilon, times 12: m 2^x. (t^2 of a double with
// exponent field E and mantissa mant is sqrhi(mant) 2^(2E) in the same unit.)
HJ_W64 Sum floor_term(double floor12) {
    const u64 b = bits(floor12);
    return {mant(b), expo(b) + 1021};
}

// 12 eps = 12e-6 amax^2 + 12 floor, from the bits of amax; m in [2^60, 2^64)
HJ_W64 Sum eps_sum(u64 amax, Sum fl) {
    const u64 ka = mulhi(sqrhi(mant(amax)) << 1, 0x64a9cdc443914f48ull) << 1;  // times 12e-6 = k 2^-79
    const int xa = 2 * expo(amax) - 17;
    const int x = imax(xa, fl.x);
    return {(ka >> imin(x - xa, 63)) + (fl.m >> imin(x - fl.x, 63)), x};
}

// A double as a 62-bit mantissa in [2^61, 2^62) and a biased exponent, and its sign.
struct Parts {
    u64 m;
    int x;
    u32 sign;  // 0 or all ones
};
HJ_W64 Parts parts(double d) {
    const u64 b = bits(d);
    return {((b << 9) & 0x1fffffffffffffffull) | 0x2000000000000000ull, expo(b), (u32)((int32_t)hi(b) >> 31)};
}

// 12 (S + eps) = 13 t^2 + 3 u^2 + 12 eps with u = a + 2^k b (flip: a - 2^k b), added
// up as sixteenths (13/16 = 1 - 3/16) so that each term is cut off once. u is not
// normalised after a cancellation: a (or t = a) is then as large as 2^k b, so that
// t^2 or, for the middle window, whose t is the difference of what u adds, the
// other square carries the sum. Relative error below 2^-54.
HJ_W64 Sum smooth_sum(Parts t, Parts a, Parts b, int k, u32 flip, Sum eps) {
    const int xb = b.x + k;
    const int xu = imax(a.x, xb);
    const u64 am = a.m >> imin(xu - a.x, 63), bm = b.m >> imin(xu - xb, 63);
    const u32 sub = a.sign ^ b.sign ^ flip;         // all ones: the magnitudes are subtracted
    const u64 subw = (u64)sub << 32 | sub;
    const u64 sum = am + (bm ^ subw) + (sub & 1u);   // below 2^63, or negative
    const u32 neg = (u32)((int32_t)hi(sum) >> 31);
    const u64 negw = (u64)neg << 32 | neg;
    const u64 tt = sqrhi(t.m), uu = sqrhi((sum ^ negw) + (neg & 1u));
    const int xt2 = 2 * t.x + 2, xu2 = 2 * xu + 2;
    const int x = imax(imax(xt2, xu2), eps.x);
    const u64 s = ((tt - ((3 * tt) >> 4)) >> imin(x - xt2, 63)) + ((3 * uu) >> imin(x - xu2 + 4, 63)) +
                  (eps.m >> imin(x - eps.x + 4, 63));
    const int n = clz(hi(s)) - 1;
    return {s << n, x - n + 4};
}

// With d_k = (S_k + eps)^2 and P_A = d_B d_C, P_B = d_A d_C, P_C = d_A d_B:
//   l1 = 2 P_A / DL, l3 = 3 P_C / DL, DL = P_A + 6 P_B + 3 P_C
//   r1 = 3 P_A / DR, r3 = 2 P_C / DR, DR = 3 P_A + 6 P_B + P_C
// The P enter the sums aligned to the largest, the products unshifted: each
// weight keeps its relative precision however small it is.
HJ_W64 void weights(Sum A, Sum B, Sum C, double& l1, double& l3, double& r1, double& r3) {
    const u64 pA = sqrhi(mulhi(B.m, C.m) << 1), pB = sqrhi(mulhi(A.m, C.m) << 1), pC = sqrhi(mulhi(A.m, B.m) << 1);
    const int xm = imin(imin(A.x, B.x), C.x);
    const int dA = 2 * (A.x - xm), dB = 2 * (B.x - xm), dC = 2 * (C.x - xm);
    const u64 qA = pA >> imin(dA + 3, 63), qB = pB >> imin(dB + 3, 63), qC = pC >> imin(dC + 3, 63);
    const u64 sum = qA + qC + 6 * qB;
    const u64 DL = sum + 2 * qC, DR = sum + 2 * qA;  // [2^55, 2^62.4)
    const int nL = clz(hi(DL)) - 1, nR = clz(hi(DR)) - 1;
    const u64 iL = recip(DL << nL), iR = recip(DR << nR);
    const int kL = nL - 64, kR = nR - 64;  // p / DL = mulhi(p, iL) 2^(64 - 125 + nL - 3 - d)
    l1 = pack(mulhi(pA, iL), kL - dA + 1);
    l3 = pack(3 * mulhi(pC, iL), kL - dC);
    r1 = pack(3 * mulhi(pA, iR), kR - dA);
    r3 = pack(mulhi(pC, iR), kR - dC + 1);
}

}  // namespace w64
}  // namespace hj
