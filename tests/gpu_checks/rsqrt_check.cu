// Errors of the FP64 sweep's reciprocal square root and division
// (drsqrt_newton, ddiv_newton, drcp_third in w5ct_physics.cuh) against the correctly
// rounded 1 / sqrt(x) (from a quotient and one correction in twice the
// working precision) and IEEE a / b, and of the exact scaling dscale2 and the
// integer comparisons.  Prints the largest errors in units in the last place,
// the number of mismatches of the exact helpers and the values checked.
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>

#include "../../paper_1812_04278_gb300/csrc/w5ct_physics.cuh"

__device__ __forceinline__ uint64_t mix(uint64_t x) {      // splitmix64 finaliser
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

__device__ double value(uint64_t r, int range) {   // random mantissa, exponent in [-range, range]
    const int e = (int)((r >> 53) % (2 * range + 1)) - range;
    return __longlong_as_double((long long)(((uint64_t)(e + 1023) << 52) | (r & 0xfffffffffffffULL)));
}

__device__ unsigned long long ulps(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return (unsigned long long)(x > y ? x - y : y - x);
}

__global__ void check(long long n, unsigned long long *worst) {
    unsigned long long ws = 0, wd = 0, bad = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const uint64_t r = mix((uint64_t)i), r2 = mix(r);
        const double x = value(r, 900), a = value(r2, 300), b = value(r, 300);
        // 1/sqrt(x): y, corrected by y (1 - x y^2) / 2 with x y^2 formed exactly enough by two FMAs
        double y = 1.0 / sqrt(x);
        const double h = x * y, hl = fma(x, y, -h), e = fma(-h, y, 1.0) - hl * y;
        y = fma(0.5 * y, e, y);
        ws = max(ws, ulps(w5ct::drsqrt_newton(x), y));
        wd = max(wd, max(ulps(w5ct::ddiv_newton(a, b), a / b), ulps(w5ct::drcp_third(x), 1.0 / x)));
        const double s = (r & 64) ? -a : a, t = (r2 & 64) ? -b : b;
        using m = w5ct::M<double>;
        bad += w5ct::dscale2<2>(s) != 4.0 * s;
        bad += w5ct::dscale2<-1>(t) != 0.5 * t;
        bad += m::max_nonneg(a, b) != fmax(a, b);
        bad += m::ge_pos(s, b) != (s >= b) || m::gt_pos(s, b) != (s > b);
        bad += m::finite_pos(s) != (s > 0.0 && s < 1.0e308);
    }
    const double inf = __longlong_as_double(0x7ff0000000000000LL), nan = __longlong_as_double(0x7ff8000000000000LL);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        bad += w5ct::dscale2<2>(0.0) != 0.0 || w5ct::dscale2<-1>(-0.0) != 0.0 || w5ct::dscale2<-1>(inf) != inf;
        bad += w5ct::dscale2<2>(nan) == w5ct::dscale2<2>(nan) || w5ct::M<double>::finite_pos(nan);
        bad += w5ct::M<double>::finite_pos(0.0) || w5ct::M<double>::finite_pos(inf) || w5ct::M<double>::finite_pos(-1.0);
    }
    atomicMax(worst, ws);
    atomicMax(worst + 1, wd);
    atomicAdd(worst + 2, bad);
}

int main() {
    unsigned long long *w = nullptr, h[3] = {0, 0, 0};
    const long long n = 1LL << 24;
    if (cudaMalloc(&w, sizeof(h)) != cudaSuccess) return 2;
    cudaMemset(w, 0, sizeof(h));
    check<<<1024, 256>>>(n, w);
    if (cudaMemcpy(h, w, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    cudaFree(w);
    printf("rsqrt_ulp %llu div_ulp %llu mismatches %llu checked %lld\n", h[0], h[1], h[2], n);
    return 0;
}
