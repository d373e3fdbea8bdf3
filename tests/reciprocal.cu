// Device check of the FP64 reciprocal, quotient and halving (common.cuh): "name worst bound" per property.
#include <cmath>
#include <cstdio>
#include "../paper_1006_2146_gb300/csrc/common.cuh"
using namespace ader;

__device__ unsigned long long mix(unsigned long long s) {
    s ^= s >> 31; s *= 0x9E3779B97F4A7C15ull; s ^= s >> 29; s *= 0xBF58476D1CE4E5B9ull;
    return s ^ (s >> 32);
}
__device__ double value(unsigned long long s, int i, unsigned lo_ex, unsigned n_ex) {
    unsigned long long m = s & 0xfffffffffffffull;
    if (i % 8 == 0) m = s & 0xfff;                          // just above a power of two
    if (i % 8 == 1) m = 0xfffffffffffffull - (s & 0xfff);   // just below
    if (i % 8 == 2) m = 0;                                  // on it
    if (i % 8 == 3) m &= ~0xffffffffull;                    // what the seed sees exactly
    return __longlong_as_double((long long)(m | ((unsigned long long)(lo_ex + (unsigned)((s >> 52) % n_ex)) << 52) |
                                            ((s & 0x10ull) << 59)));
}
__device__ void worst(double* out, double e) { atomicMax((unsigned long long*)out, (unsigned long long)__double_as_longlong(e)); }

__global__ void k(double* out) {
    double e_r = 0, e_q = 0, e_h = 0, e_s = 0;
    for (int i = 0; i < 4096; ++i) {
        const unsigned long long a = mix((blockIdx.x * 256ull + threadIdx.x) * 4096ull + i + 1), b = mix(a + 77);
        const double x = value(a, i, 1, 2044), m = value(a, i, 1023, 1), y = value(b, i >> 3, 800, 400);
        e_r = fmax(e_r, fabs(fma(-m, rcp(m), 1.0)));
        // the exponent only moves the result (a subnormal one counts as zero)
        const int ex = (__double2hiint(x) >> 20) & 0x7ff;
        const double want = scalbn(rcp(m), 1023 - ex);
        if (rcp(x) != want) e_s += 1;
        const double n = value(b, i, 900, 200), q = quot(n, y);
        e_q = fmax(e_q, fabs(fma(-q, y, n) / n));
        if (halved(x) != (ex > 1 ? 0.5 * x : x)) e_h += 1;
    }
    worst(out, e_r);
    worst(out + 1, e_q);
    worst(out + 2, e_h);
    worst(out + 3, e_s);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double inf = __longlong_as_double(0x7ff0000000000000ll), nan = __longlong_as_double(0x7ff8000000000000ll);
        out[4] = !isnan(rcp(0.0)) + !isnan(rcp(-0.0)) + !isnan(rcp(inf)) + !isnan(rcp(nan)) + (rcp(1e308) != 0.0) +
                 !isnan(halved(nan)) + (halved(0.0) != 0.0) + (speed_root(0.0) != 0.0) + !isinf(speed_root(inf)) +
                 !isnan(speed_root(nan));
    }
}

int main() {
    double *d, h[5];
    cudaMalloc(&d, sizeof h);
    cudaMemset(d, 0, sizeof h);
    k<<<64, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    // a half unit of the last place, the dropped third power of the seed's 2^-19.9 and the cut products (2^-59, 2^-60)
    const double bound = std::ldexp(1.0, -53) + std::ldexp(1.0, -58);
    std::printf("reciprocal %.17g %.17g\nquotient %.17g %.17g\nhalved %.17g 0\nscaled %.17g 0\nspecial %.17g 0\n", h[0], bound, h[1],
                bound, h[2], h[3], h[4]);
    return 0;
}
