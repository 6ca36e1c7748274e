// Test probe: the integer WENO5 weights (weno_weights64.cuh) compiled for the
// host. in: n rows of {tA, tB, tC, d23, d34, amax, 12 floor}; out: n rows of
// {l1, l3, r1, r3}.
#include "weno_weights64.cuh"

extern "C" void weights64_probe(const double* in, double* out, long long n) {
    using namespace hj::w64;
    for (long long i = 0; i < n; ++i) {
        const double* p = in + 7 * i;
        const Sum eps = eps_sum(abs_bits(p[5]), floor_term(p[6]));
        const Parts a = parts(p[0]), b = parts(p[1]), c = parts(p[2]), d23 = parts(p[3]), d34 = parts(p[4]);
        weights(smooth_sum(a, a, d23, 1, 0u, eps), smooth_sum(b, d23, d34, 0, 0u, eps),
                smooth_sum(c, c, d34, 1, ~0u, eps), out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
    }
}
