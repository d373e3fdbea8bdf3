// Device check of the FP64 root of wave speeds (common.cuh): "name worst bound" per property.
#include <cmath>
#include <cstdio>
#include "../paper_1006_2146_gb300/csrc/common.cuh"
using namespace ader;

__device__ unsigned long long mix(unsigned long long s) {
    s ^= s >> 31; s *= 0x9E3779B97F4A7C15ull; s ^= s >> 29; s *= 0xBF58476D1CE4E5B9ull;
    return s ^ (s >> 32);
}

__global__ void k(double* out) {
    double e_r = 0, e_s = 0;
    for (int i = 0; i < 4096; ++i) {
        const unsigned long long s = mix((blockIdx.x * 256ull + threadIdx.x) * 4096ull + i + 1);
        unsigned long long m = s & 0xfffffffffffffull;
        if (i % 8 == 0) m = s & 0xfff;                          // just above a power of two
        if (i % 8 == 1) m = 0xfffffffffffffull - (s & 0xfff);   // just below
        if (i % 8 == 2) m = 0;                                  // on it
        // both parities of the exponent, from 2^-900 (below, the remainder itself would be subnormal) to the largest
        const double x = __longlong_as_double((long long)(m | (unsigned long long)(123 + (s >> 52) % 1924) << 52));
        const double r = speed_root(x);
        // (x - r^2) / 2 x, the relative error; scaled first, so that nothing in it is subnormal
        const int ex = ((__double2hiint(x) >> 20) & 0x7ff) - 1023, half = ex >> 1;
        const double xs = scalbn(x, -2 * half), rs = scalbn(r, -half);
        e_r = fmax(e_r, fabs(fma(-rs, rs, xs)) / (2 * xs));
        // an exponent two higher moves the result by one
        if (speed_root(xs) != rs) e_s += 1;
    }
    atomicMax((unsigned long long*)out, (unsigned long long)__double_as_longlong(e_r));
    atomicMax((unsigned long long*)(out + 1), (unsigned long long)__double_as_longlong(e_s));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double inf = __longlong_as_double(0x7ff0000000000000ll), nan = __longlong_as_double(0x7ff8000000000000ll);
        out[2] = (speed_root(0.0) != 0.0) + (speed_root(4.9e-324) != 0.0) + (speed_root(inf) != inf) +
                 !isnan(speed_root(nan)) + !isnan(speed_root(-inf)) + !isnan(speed_root(-1.0)) + (speed_root(4.0) != 2.0);
    }
}

int main() {
    double *d, h[3];
    cudaMalloc(&d, sizeof h);
    cudaMemset(d, 0, sizeof h);
    k<<<64, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    // a rounding of the last place and the dropped fourth term, 5 / 16 of the third power of e = 2^-18.9
    std::printf("root %.17g %.17g\nscaled %.17g 0\nspecial %.17g 0\n", h[0], std::ldexp(1.0, -53) + std::ldexp(1.0, -58), h[1], h[2]);
    return 0;
}
