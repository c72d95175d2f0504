// The FP64 sweep's integer-pipe products (w5ct_physics.cuh: dmul_any, pmul3,
// pmul2, weno_weights) against the FP64 multiplier, bit for bit: random factors
// of every exponent, significands with long runs of zeros and ones (ties and
// carries of the rounding), exponents at the edges of each range check, zeros,
// subnormals, infinities and NaN.  Prints the number of mismatches and of
// values checked.
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>

#include "../../paper_1812_04278_gb300/csrc/w5ct_physics.cuh"

using namespace w5ct;

__device__ __forceinline__ uint64_t mix(uint64_t x) {      // splitmix64 finaliser
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

// significand pattern by `kind`, biased exponent e, sign from bit 52 of r
__device__ double value(uint64_t r, int kind, int e) {
    const uint64_t all = (1ULL << 52) - 1;
    uint64_t f = r & all;
    const int k = (int)((r >> 54) % 53);
    if (kind == 1) f &= ~((1ULL << k) - 1);            // trailing zeros
    if (kind == 2) f |= (1ULL << k) - 1;               // trailing ones
    if (kind == 3) f = all - (f >> k);                 // leading ones
    if (kind == 4) f &= ~((1ULL << 26) - 1);           // 26 bits: exact products and ties
    if (kind == 5) f = k < 52 ? 1ULL << k : 0;         // one bit or none
    return __longlong_as_double((long long)((r << 11 & 0x8000000000000000ULL) | (uint64_t)e << 52 | f));
}

__device__ bool differ(double a, double b) {
    return a == a || b == b ? __double_as_longlong(a) != __double_as_longlong(b) : false;   // any NaN equals any NaN
}

__device__ const int kEdges[] = {0,    1,    2,    3,    512,  513,  514,  766,  767,  768,  862,  863, 864, 1022, 1023,
                                 1118, 1119, 1120, 1278, 1279, 1280, 1531, 1532, 1533, 2044, 2045, 2046, 2047};

__global__ void check(long long n, unsigned long long *out) {
    unsigned long long bad = 0, cnt = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        uint64_t r[7];
        r[0] = mix((uint64_t)i);
        for (int k = 1; k < 7; ++k) r[k] = mix(r[k - 1]);
        double v[7];
        for (int k = 0; k < 7; ++k) {
            const uint64_t t = mix(r[k] ^ 0x5555);
            const int sel = (int)(t & 3), kind = (int)(t >> 8) % 6;
            int e = 1023 - 40 + (int)((t >> 20) % 80);                    // ordinary
            if (sel == 1 && (i & 3) == 0) e = (int)((t >> 20) % 2048);    // any
            if (sel == 2 && (i & 3) == 1) e = kEdges[(t >> 20) % (sizeof(kEdges) / sizeof(int))];
            v[k] = value(r[k], kind, e);
        }
        bad += differ(dmul_any(v[0], v[1]), v[0] * v[1]);
        bad += differ(dmul_call(v[2], v[3]), v[2] * v[3]);
        Pair<double> x, y, z, p;
        const Pair<double> a = {v[1], v[2]}, b = {v[3], v[4]}, c = {v[5], v[6]};
        pmul3(v[0], a, b, c, x, y, z);
        p = pmul(v[0], a);
        bad += differ(x.x, p.x) + differ(x.y, p.y);
        p = pmul(v[0], b);
        bad += differ(y.x, p.x) + differ(y.y, p.y);
        p = pmul(-v[0], c);
        bad += differ(z.x, p.x) + differ(z.y, p.y);
        pmul2(v[0], v[1], b, x, y);
        p = pmul(v[0], b);
        bad += differ(x.x, p.x) + differ(x.y, p.y);
        p = pmul(v[1], b);
        bad += differ(y.x, p.x) + differ(y.y, p.y);
        // weights of indicators: positive; equal s_0 and s_2, or a last-place
        // difference, at times
        const double s0 = fabs(v[0]), s1 = fabs(v[1]);
        double s2 = fabs(v[2]);
        if ((i & 15) == 2) s2 = s0;
        if ((i & 15) == 3) s2 = __longlong_as_double(__double_as_longlong(s0) ^ 1);
        double W0, V1, V2;
        double3 w = weights_mul<0>(s0, s1, s2);
        weno_weights<0>(s0, s1, s2, W0, V1, V2);
        bad += differ(W0, w.x) + differ(V1, w.y) + differ(V2, w.z);
        w = weights_mul<1>(s0, s1, s2);
        weno_weights<1>(s0, s1, s2, W0, V1, V2);
        bad += differ(W0, w.x) + differ(V1, w.y) + differ(V2, w.z);
        cnt += 18;
    }
    atomicAdd(out, bad);
    atomicAdd(out + 1, cnt);
}

int main() {
    unsigned long long *w = nullptr, h[2] = {0, 0};
    if (cudaMalloc(&w, sizeof(h)) != cudaSuccess) return 2;
    cudaMemset(w, 0, sizeof(h));
    check<<<1024, 128>>>(1LL << 23, w);
    if (cudaMemcpy(h, w, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    cudaFree(w);
    printf("mismatches %llu checked %llu\n", h[0], h[1]);
    return 0;
}
