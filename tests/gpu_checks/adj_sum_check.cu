// The sums over faces of adj_cell_kernel: face adjoints that cancel to nothing
// in float and exactly in double.  State at rest (rho = 1, E = 1, B = 0), all face
// planes zero but those of the energy's state difference at positions 0 .. 4:
// the difference d then sums five faces, and the energy's adjoint of cell i is
// D(i-1) - D(i).  Big terms are 2^30 (exact in float, 2^30 + 1 is not), small
// ones integers below 2^10.  Prints the largest error against integer sums.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_1812_04278_gb300/csrc/w5ct_adjoint.cuh"

using namespace w5ct;

template <int AX, typename R>
static double run(int nx, int ny, int nz) {
    const size_t n = (size_t)nx * ny * nz, runs = adj_run_cells(n);
    std::vector<R> fa(runs * kAdjFluxPlanes, R(0)), fb(runs * (kAdjFacePlanes - kAdjFluxPlanes), R(0)), q(5 * n, R(0)), b(3 * n, R(0));
    for (size_t p = 0; p < n; ++p) q[p] = q[4 * n + p] = R(1);
    const int c = 6;                                        // energy
    std::vector<long long> w(5 * n);
    unsigned long long h = 12345;
    for (size_t p = 0; p < n; ++p)
        for (int j = 0; j < 5; ++j) {
            h = h * 6364136223846793005ULL + 1442695040888963407ULL;
            const long long sign = (j & 1) ? -1 : 1;        // small at 0, -2^30 at 1 and 3, 2^30 at 2 and 4
            w[5 * p + j] = j > 0 ? sign * (1LL << 30) : (long long)(h >> 54);
            const int k = kAdjDiff + (c * 5 + j) * 2 + 1;
            const size_t run = p / kAdjRun, at = p % kAdjRun;
            (k < kAdjFluxPlanes ? fa[run * (kAdjFluxPlanes * kAdjRun) + k * kAdjRun + at]
                                : fb[run * ((kAdjFacePlanes - kAdjFluxPlanes) * kAdjRun) + (k - kAdjFluxPlanes) * kAdjRun + at]) = (R)w[5 * p + j];
        }
    auto up = [&](const void *src, size_t bytes) {
        void *d = nullptr;
        if (cudaMalloc(&d, bytes) != cudaSuccess) exit(2);
        if (src) cudaMemcpy(d, src, bytes, cudaMemcpyHostToDevice); else cudaMemset(d, 0, bytes);
        return d;
    };
    AdjSweepArgs<R> a;
    a.nx = nx, a.ny = ny, a.nz = nz, a.rd = 1.0, a.first = true;
    R *dq = (R *)up(q.data(), q.size() * sizeof(R)), *db = (R *)up(b.data(), b.size() * sizeof(R));
    for (int f = 0; f < 5; ++f) a.q[f] = dq + f * n;
    for (int f = 0; f < 3; ++f) a.bc[f] = db + f * n;
    double *lam = (double *)up(nullptr, 8 * n * 8);
    a.lamD = lam, a.lamO = lam + 5 * n;
    a.fa = (R *)up(fa.data(), fa.size() * sizeof(R)), a.fb = (R *)up(fb.data(), fb.size() * sizeof(R));
    a.outq = (double *)up(nullptr, 5 * n * 8), a.outb = (double *)up(nullptr, 3 * n * 8);
    a.K = Phys<R>{};
    a.K.gamma = R(5.0 / 3.0), a.K.gm1 = R(2.0 / 3.0);
    const AdjTile &t = a.cell_tile = adj_cell_tile(AX, nx, ny, nz);
    adj_cell_kernel<AX, R><<<(t.units + t.per - 1) / t.per, 256>>>(a);
    if (cudaDeviceSynchronize() != cudaSuccess) exit(3);
    std::vector<double> out(n);
    cudaMemcpy(out.data(), a.outq + 4 * n, n * 8, cudaMemcpyDeviceToHost);
    double worst = 0;
    for (int z = 0; z < nz; ++z)
        for (int y = 0; y < ny; ++y)
            for (int x = 0; x < nx; ++x) {
                auto at = [&](int o) {
                    const int m = AX == 0 ? nx : AX == 1 ? ny : nz;
                    const int i = ((AX == 0 ? x : AX == 1 ? y : z) + o + 4 * m) % m;
                    return AX == 0 ? (size_t)i + (size_t)nx * (y + (size_t)ny * z)
                           : AX == 1 ? (size_t)x + (size_t)nx * (i + (size_t)ny * z) : (size_t)x + (size_t)nx * (y + (size_t)ny * i);
                };
                long long D[2] = {0, 0};                    // differences i - 1 and i
                for (int d = 0; d < 2; ++d)
                    for (int j = 0; j < 5; ++j) D[d] += w[5 * at(d - 1 + 2 - j) + j];
                const double e = out[at(0)] - (double)(D[0] - D[1]);
                if (!(e <= worst && -e <= worst)) worst = e < 0 ? -e : e;
            }
    for (void *p : {(void *)dq, (void *)db, (void *)lam, (void *)a.fa, (void *)a.fb, (void *)a.outq, (void *)a.outb}) cudaFree(p);
    return worst;
}

int main() {
    printf("float %g %g %g double %g %g %g\n", run<0, float>(33, 9, 10), run<1, float>(33, 9, 10), run<2, float>(33, 9, 10),
           run<0, double>(33, 9, 10), run<1, double>(33, 9, 10), run<2, double>(33, 9, 10));
    return 0;
}
