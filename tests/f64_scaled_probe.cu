// Host build of the exact float-to-double widening (csrc/tf32_split.cuh).
#include "../paper_1911_00242_gb300/csrc/tf32_split.cuh"

extern "C" void probe_f64_scaled(const float* x, long long n, int e, int neg, double* out) {
    for (long long i = 0; i < n; ++i) out[i] = ccsdk::f64_scaled(x[i], e, neg != 0);
}
extern "C" int probe_pow2(double p, int* e) { return ccsdk::pow2_exponent(p, *e) ? 1 : 0; }
