// Test probe: the integer WENO5 weights (weno_weights64.cuh) compiled for the
// host. in: n rows of {tA, tB, tC, uA, uB, uC, amax, 12 floor}; out: n rows of
// {l1, l3, r1, r3}.
#include "weno_weights64.cuh"

extern "C" void weights64_probe(const double* in, double* out, long long n) {
    using namespace hj::w64;
    for (long long i = 0; i < n; ++i) {
        const double* p = in + 8 * i;
        const Sum eps = eps_sum(abs_bits(p[6]), floor_term(p[7]));
        weights(smooth_sum(p[0], p[3], eps), smooth_sum(p[1], p[4], eps), smooth_sum(p[2], p[5], eps), out[4 * i],
                out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
    }
}
