// The 64-bit fixed-point arithmetic of the FP64 transforms on the host, for tests/test_fixed_point.py.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

static inline int __double2hiint(double d) {
    long long b;
    std::memcpy(&b, &d, 8);
    return (int)(b >> 32);
}
static inline long long __double_as_longlong(double d) {
    long long b;
    std::memcpy(&b, &d, 8);
    return b;
}
static inline double __longlong_as_double(long long b) {
    double d;
    std::memcpy(&d, &b, 8);
    return d;
}
static inline float __int_as_float(int b) {
    float f;
    std::memcpy(&f, &b, 4);
    return f;
}
static inline unsigned __float_as_uint(float f) {
    unsigned b;
    std::memcpy(&b, &f, 4);
    return b;
}
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }

#include "../paper_2508_07424_gb300/csrc/pff_fixed.cuh"

extern "C" {

void to_fixed(int n, const double *d, int k, long long *out) {
    for (int i = 0; i < n; ++i) out[i] = pff::fx_in(d[i], k);
}

}  // extern "C"
