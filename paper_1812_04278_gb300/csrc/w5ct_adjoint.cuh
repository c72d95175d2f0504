// w5ct_adjoint.cuh -- adjoint (vector-Jacobian product) of one RK4 + CT step
// of fixed dt, and of the initial-condition map from primitive fields and an
// edge vector potential.
//
// One step is linear in its stage results: with D_s the flux divergence and
// Omega_s the corner EMFs of stage s (Sec. 2.1, Eq. num, Eqs. ox1-ox3),
//   q_{s+1} = q^n + c_s dt D_s,   b_{s+1} = b^n + c_s dt curl Omega_s  (s < 3),
//   q^{n+1} = q^n + dt sum_s w_s D_s,   b^{n+1} = b^n + dt curl sum_s w_s Omega_s,
// c = (1/2, 1/2, 1), w = (1, 2, 2, 1)/6.  (D_s, Omega_s) depend on the stage
// state through the sweeps (nonlinear, per face) and the divergence, EMF
// average and cell-field interpolation (linear).  The adjoint runs the
// stages backwards: the linear maps by their transposes (the kernels below),
// the sweeps by adj_face_kernel, the reverse mode of each face's function
// (48 inputs -> 7 outputs) contracted with the incoming flux adjoints.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "w5ct_kernels.cuh"

namespace w5ct {

// ---------------------------------------------------------------- sweep adjoint
//
// Two kernels per axis and stage.  adj_face_kernel runs the face function's
// reverse mode, one thread per face over the same shared-memory cell box as
// the forward sweep, and writes the adjoints of what the face reads of its
// cells: the five stencil differences of the flux and of the conserved vector
// (70), the central flux (7), the interface primitives (8) and the wave
// speeds of its two cells (2 x 4).  adj_cell_kernel sums them over the faces
// of each cell in a fixed order and reverses the cell recovery once per cell.
constexpr int kAdjDiff = 0;                    // plane (c * 5 + j) * 2 + (0: dF_c, 1: du_c) at position j
constexpr int kAdjCentral = 70;                // central flux, component c
constexpr int kAdjPrim = 77;                   // interface primitives (C_RHO .. C_P)
constexpr int kAdjSide = 85;                   // (v_n, c_f, c_A, c_slow) of the lower cell, then of the upper
constexpr int kAdjFacePlanes = 93;
constexpr int kAdjFluxPlanes = 21;             // the first planes lie in the context's flux buffers
// The planes are stored in runs of kAdjRun faces, plane after plane within a
// run: a thread forms one address per face and part, and every plane is a
// constant offset from it (with whole planes the 64-bit address arithmetic of
// 93 stores and of about 120 loads is not free: 64^3 FP32 gradient, 3 steps, 6.89
// -> 6.70 ms).
constexpr int kAdjRun = 128;
constexpr size_t adj_run_cells(size_t n) { return (n + kAdjRun - 1) / kAdjRun * kAdjRun; }

template <typename Real>
struct AdjFaceRef {
    Real *a, *b;
    __device__ __forceinline__ Real &operator[](int k) const {
        return k < kAdjFluxPlanes ? a[k * kAdjRun] : b[(k - kAdjFluxPlanes) * kAdjRun];
    }
};

// Division of 0 <= n < 2^31 by d > 0: with 2^(s - 1) < d <= 2^s and mul =
// ceil(2^(31 + s) / d) <= 2^32 - 1 (d = 1: s = 0, mul = 2^31) the quotient is the
// top of n mul, whose excess over n 2^(31 + s) / d is below n < 2^31, less than the
// 2^(31 + s) / d >= 2^31 that separates two quotients.
struct IntDiv {
    unsigned mul, shift;
    int d;
    __device__ __forceinline__ int div(int n) const { return (int)(((unsigned long long)(unsigned)n * mul) >> shift); }
};
inline IntDiv int_div(int d) {
    int s = 0;
    while (s < 31 && (1LL << s) < d) ++s;
    return {(unsigned)(((1ULL << (31 + s)) + (unsigned)d - 1) / (unsigned)d), (unsigned)(31 + s), d};
}

// Tiles of the two kernels.  The pencils of a sweep (lines of cells along its
// axis) are numbered flat over the other two directions, and cut into nseg
// segments of len positions.  A block computes `per` units: for the x-sweep a
// unit is a segment of one pencil, for the others the same segment of BX
// consecutive pencils, so that neither a narrow x nor a thin axis leaves lanes
// or rows empty (chosen by adj_tile; tiles cut in x and one other direction
// left most of a block idle there: gradient of 256 x 256 x 1 in float 1.45 -> 0.78 ms, 1 x
// 128 x 128 1.56 -> 0.67, in double 19.7 -> 10.1 and 29.5 -> 4.5; 64^3 1.875 -> 1.895 and
// 23.4 -> 23.2).
struct AdjTile {
    int len, nseg, per;
    int units;                       // of the whole sweep
    IntDiv rows, positions, segments, cross;   // by a segment's rows, by len, nseg, and the pencils' faster direction
};

template <typename Real>
struct AdjSweepArgs {
    int nx, ny, nz;
    double rd;                 // 1 / spacing along the axis
    const Real *q[5];          // stage state (rho, m, E), arithmetic type
    const Real *bc[3];         // the stage's cell-centred field
    const double *lamD;        // 5 planes: adjoint of the flux divergence
    const double *lamO;        // 3 planes: adjoint of the corner EMFs
    Real *fa, *fb;             // face adjoints: planes 0..20 in fa, the others in fb
    double *outq, *outb;       // 5 planes of the state's adjoint, 3 of the cell field's
    bool first;                // the first axis of the stage writes outq, outb, the others add
    Phys<Real> K;
    AdjTile face_tile, cell_tile;   // (adj_tiles)
    __device__ __forceinline__ AdjFaceRef<Real> face(size_t p) const {
        const size_t run = p / kAdjRun, at = p % kAdjRun;
        return {fa + run * (kAdjFluxPlanes * kAdjRun) + at, fb + run * ((kAdjFacePlanes - kAdjFluxPlanes) * kAdjRun) + at};
    }
};

// Reverse of speeds_fast and c_slow^2 = c_s^2 c_A^2 / c_f^2: adds to (lcs2,
// lca2, lbt2) the adjoints of the inputs given those of (fmc, cms, cf2, csl2);
// the same branches and guards as the forward formulas (Eqs. slow/fast).
template <typename R>
__device__ __forceinline__ void speeds_rev(R cs2, R ca2, R bt2, R lfmc, R lcms, R lcf2, R lcsl2, R &lcs2, R &lca2,
                                           R &lbt2) {
    using m = M<R>;
    const R aa = ca2 + bt2 - cs2;
    const R dd = m::fma_(aa, aa, R(4) * (cs2 * bt2));
    R isd, sd;
    if (disc_normal(dd)) {
        isd = m::rsqrt_(dd);
        sd = dd * isd;
    } else {
        const Disc<R> d = disc_small(aa, cs2, bt2);
        isd = d.isd;
        sd = d.sd;
    }
    const R big = m::half_(sd + m::abs_(aa));
    const R ibig = m::normal_pos(big) ? m::rcp3_(big) : R(0);
    // ratios of speeds first: products of two squared speeds, or of their
    // adjoints and a reciprocal, may leave the range
    const R ci = cs2 * ibig, bi = bt2 * ibig, oth = cs2 * bi;
    const bool fast_big = m::nonneg(aa);
    const R cf2 = cs2 + (fast_big ? big : oth);
    const R icf2 = m::normal_pos(cf2) ? m::rcp3_(cf2) : R(0);
    const R cc = cs2 * icf2, ac = ca2 * icf2;
    lcs2 += lcsl2 * ac;
    lca2 += lcsl2 * cc;
    lcf2 -= lcsl2 * (cc * ac);
    lcs2 += lcf2;
    lfmc += lcf2;
    // big = (sqrt(dd) + |aa|) / 2, oth = c_s^2 b_t^2 / big
    const R loth = fast_big ? lcms : lfmc;
    R lbig = fast_big ? lfmc : lcms;
    lbig -= loth * (ci * bi);
    lcs2 += loth * bi;
    lbt2 += loth * ci;
    const R hb = m::half_(lbig);
    const R laa = fast_big ? hb : -hb;
    // dd = aa^2 + 4 c_s^2 b_t^2, aa = ca2 + bt2 - cs2
    const R la = laa + hb * (aa * isd);
    lca2 += la;
    lbt2 += la + lbig * (cs2 * isd);
    lcs2 += lbig * (bt2 * isd) - la;
}

// One interpolant phi~ = N / D = 12 phi_N(a, b, c, d) (the weights of the
// forward step: JS, or WENO-Z with the ratio clamped at 1e18 in float) and its
// gradient, times the seed l: smoothness indicators -> weights, in the
// normalised form e_k = alpha_k / d_k from one reciprocal per indicator ->
// N / D, run backwards.  A reciprocal r = 1/x is reversed as -r (r l), never
// with r^2, so that a tiny eps + IS times a zero adjoint stays 0 in float.
template <typename R, int VAR>
__device__ __forceinline__ void phi_rev(R a, R b, R c, R d, R eps12, R l, R &f, R (&g)[4]) {
    using m = M<R>;
    R s0, s1, s2, x0, y0, z0;
    smoothness3<R>(a, b, c, d, eps12, s0, s1, s2, x0, y0, z0);
    const R i0 = m::rcp3_(s0), i1 = m::rcp3_(s1), i2 = m::rcp3_(s2);
    R r0, r1, r2, e0, e1, e2, tau = R(0);
    bool k0 = false, k1 = false, k2 = false;      // clamped ratios
    if constexpr (VAR == 0) {
        e0 = i0 * i0;
        e1 = i1 * i1;
        e2 = i2 * i2;
        r0 = r1 = r2 = R(0);
    } else {
        tau = s0 - s2;
        const R ta = m::abs_(tau);
        r0 = ta * i0;
        r1 = ta * i1;
        r2 = ta * i2;
        if constexpr (float_based<R>) {
            const R top = R(1.0e18);
            k0 = r0 > top;
            k1 = r1 > top;
            k2 = r2 > top;
            r0 = k0 ? top : r0;
            r1 = k1 ? top : r1;
            r2 = k2 ? top : r2;
        }
        e0 = m::fma_(r0, r0, R(1));
        e1 = m::fma_(r1, r1, R(1));
        e2 = m::fma_(r2, r2, R(1));
    }
    const R D = m::fma_(R(3), e2, m::fma_(R(6), e1, e0));
    const R iD = m::rcp3_(D);
    const R w0 = m::times4_(e0 * iD), w2 = m::fma_(R(6) * e2, iD, R(-1));
    const R t1 = x0 - y0, t2 = y0 - z0;
    f = m::fma_(w0, t1, w2 * t2);
    // d(l f): weights
    const R u2 = R(2) * l * iD;      // twice the seeds of e_k
    const R le0 = u2 * (m::fma_(R(4), t1, -t2) - f), le1 = R(-6) * u2 * (t2 + f), le2 = R(3) * u2 * (t2 - f);
    const R lt1 = l * w0, lt2 = l * w2;
    R ls0, ls1, ls2;
    if constexpr (VAR == 0) {
        ls0 = -(le0 * e0) * i0;
        ls1 = -(le1 * e1) * i1;
        ls2 = -(le2 * e2) * i2;
    } else {
        // e = 1 + r^2, r = |tau| / s
        const R v0 = k0 ? R(0) : le0 * r0 * i0, v1 = k1 ? R(0) : le1 * r1 * i1, v2 = k2 ? R(0) : le2 * r2 * i2;
        const R lta = v0 + v1 + v2;
        const R lt = m::nonneg(tau) ? lta : -lta;
        ls0 = m::fma_(-v0, r0, lt);
        ls1 = -(v1 * r1);
        ls2 = m::fma_(-v2, r2, -lt);
    }
    const R k = R(8.0 / 3.0);
    const R lx = m::fma_(ls0, m::fma_(k, x0, -b), lt1);
    const R ly = m::fma_(ls1, m::fma_(k, y0, -b), lt2 - lt1);
    const R lz = m::fma_(ls2, m::fma_(k, z0, c), -lt2);
    g[0] = lx;
    g[1] = m::fma_(ls0, m::fma_(R(2), b, -x0), m::fma_(ls1, m::fma_(R(2), b, -y0), ly - lx));
    g[2] = m::fma_(ls2, m::fma_(R(2), c, z0), lz - ly);
    g[3] = -lz;
}

__device__ __forceinline__ double pair_x(Pair<double> a) { return a.x; }
__device__ __forceinline__ double pair_y(Pair<double> a) { return a.y; }
__device__ __forceinline__ float pair_x(Pair<float> a) { return a.v.x; }
__device__ __forceinline__ float pair_y(Pair<float> a) { return a.v.y; }
__device__ __forceinline__ Pair<double> padd(Pair<double> a, Pair<double> b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Pair<float> padd(Pair<float> a, Pair<float> b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ Pair<double> psub(Pair<double> a, Pair<double> b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Pair<float> psub(Pair<float> a, Pair<float> b) {
    return {make_float2(a.v.x - b.v.x, a.v.y - b.v.y)};
}
template <typename R>
__device__ __forceinline__ void pdot(R &acc, Pair<R> a, Pair<R> b) {
    acc = M<R>::fma_(pair_x(a), pair_x(b), acc);
    acc = M<R>::fma_(pair_y(a), pair_y(b), acc);
}
template <typename R>
__device__ __forceinline__ void pdots(R &acc, Pair<R> a, Pair<R> b) {   // acc -= a.b
    acc = M<R>::fma_(-pair_x(a), pair_x(b), acc);
    acc = M<R>::fma_(-pair_y(a), pair_y(b), acc);
}

// weno_field's reverse: value = phi~(q) - phi~(p) (both 12 phi_N, in units of
// 1/24 of the split fluxes' sum), the pairs P replaced by l times the
// gradient, galpha = l d(value)/d(alpha).
template <typename R, int VAR>
__device__ __forceinline__ R field_rev(Pair<R> (&P)[5], R alpha, R eps3, R l, R &galpha) {
    R fp, fq, gp[4], gq[4];
    phi_rev<R, VAR>(psplit(P[0], alpha), psplit(P[1], alpha), psplit(P[2], alpha), psplit(P[3], alpha), eps3, -l, fp, gp);
    phi_rev<R, VAR>(psplit(P[4], -alpha), psplit(P[3], -alpha), psplit(P[2], -alpha), psplit(P[1], -alpha), eps3, l, fq,
                    gq);
    R ga = R(0);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const R up = j < 4 ? gp[j] : R(0), uq = j > 0 ? gq[4 - j] : R(0);
        const R d = up - uq;
        ga = M<R>::fma_(pair_y(P[j]), d, ga);
        P[j] = make_pair2(up + uq, alpha * d);
    }
    galpha = ga;
    return fq - fp;
}

// One pencil of a sweep along AX: position i lies at base + i * stride of a plane.
template <int AX>
struct Pencil {
    size_t base;
    int n;
    size_t stride;
    __device__ __forceinline__ Pencil(int id, int nx, int ny, int nz, const IntDiv &cross) {
        n = AX == 0 ? nx : AX == 1 ? ny : nz;
        stride = AX == 0 ? 1 : AX == 1 ? (size_t)nx : (size_t)nx * ny;
        const int z = AX == 1 ? cross.div(id) : 0;
        base = AX == 0 ? (size_t)id * nx : AX == 1 ? (size_t)(id - z * nx) + (size_t)nx * ny * z : (size_t)id;
    }
    __device__ __forceinline__ size_t at(int i) const { return base + stride * (size_t)i; }
};
// pencils of a sweep
template <int AX>
__device__ __forceinline__ int pencils(int nx, int ny, int nz) {
    return AX == 0 ? ny * nz : AX == 1 ? nx * nz : nx * ny;
}

// Elements between the cells of the face kernel's box (odd multiples of a
// bank's width, so that neighbouring lanes' cells lie in different banks), and
// the most cells of a box.
template <typename R>
__host__ __device__ constexpr int adj_box_pitch() {
    return float_based<R> ? NCQ : NBQ + 1;
}
template <typename R>
__host__ __device__ constexpr int adj_box_cells() {
    return float_based<R> ? 512 : 768;
}

// Reverse mode of the face function (face_flux and face_eigen: same
// quantities, same branches).  Its outputs are the five lab-order face fluxes
// and the two transport fluxes; their adjoints come from lamD and lamO by the
// transposes of Eq. num and of the EMF averages.  First every field's WENO part
// and its gradient, in place of the field's projections; then, per stencil
// position, the projections again from the box and their transposes; last the
// eigen scalars backwards.  The central flux is not projected, so its adjoint
// is the incoming one (except in Appendix A's fallback a_f = a_s = 1).
//
// Bound: FP64 pipe in double; in float the registers (70 projections and
// their gradients live between the two passes).  One reciprocal per smoothness
// indicator and weight sum (an IEEE division costs 9 FP64 instructions, and a
// field has 28 of them), the shared cell box, the frame projections with their
// transposes and one cell recovery per cell took the 64^3 adjoint step from
// 45.1 to 18.7 ms in its face and cell kernels (FP64, WENO-Z) and from 2.6 to
// 1.35 ms (FP32-bulk, WENO5); the whole 2-step rollout gradient 127.8 -> 66.3 ms,
// in float (3 steps) 12.1 -> 7.8 ms, no larger error against 64-bit gradients.
template <int AX, typename R, int VAR, int BX, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) adj_face_kernel(AdjSweepArgs<R> a) {
    using m = M<R>;
    using P2 = Pair<R>;
    constexpr bool DIFF = box_diff<R>();
    constexpr int ST = BX, PQ = adj_box_pitch<R>();      // (BX = 1 for the x-sweep)
    extern __shared__ __align__(16) unsigned char w5ct_smem[];
    R *sm = reinterpret_cast<R *>(w5ct_smem);
    const int nx = a.nx, ny = a.ny, nz = a.nz, tid = threadIdx.x;
    const AdjTile &t = a.face_tile;
    const int len = t.len, rows = len + 5, np = pencils<AX>(nx, ny, nz), first = (int)blockIdx.x * t.per;
    const Phys<R> K = a.K;
    // cell box: per segments of len + 5 cells, BX pencils side by side (y, z),
    // a cell's quantities together.  Pencils and units past the last repeat it.
    const int ncell = BX * t.per * rows;
    bool bad = false, hit = false;
    for (int c = tid; c < ncell; c += NT) {
        const int row = c / BX, u = t.rows.div(row);
        const int unit = min(first + u, t.units - 1), group = t.segments.div(unit), seg = unit - group * t.nseg;
        const Pencil<AX> pen(min(group * BX + c % BX, np - 1), nx, ny, nz, t.cross);
        const size_t g = pen.at(wrapi(seg * len + (row - u * rows) - 2, pen.n));
        cell_fill<R, AX>(sm + c * PQ, 0, 1, a.q[0][g], a.q[1][g], a.q[2][g], a.q[3][g], a.q[4][g], a.bc[0][g], a.bc[1][g],
                         a.bc[2][g], K, bad, hit);
    }
    __syncthreads();
    if constexpr (DIFF) {
        // (a segment's last cell has no successor, and none is read)
        constexpr int NIT = (adj_box_cells<R>() + NT - 1) / NT;
        CellDiff<R> d[NIT];
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
            const int c = tid + it * NT;
            if (c + ST < ncell) box_diff_load<R>(sm + c * PQ, 1, 0, ST * PQ, d[it]);
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
            const int c = tid + it * NT;
            if (c + ST < ncell) box_diff_store<R>(sm + c * PQ, 1, 0, d[it]);
        }
        __syncthreads();
    }
    // this thread's face
    const int trow = tid / BX, u = t.positions.div(trow), unit = first + u;
    const int group = t.segments.div(unit), id = group * BX + tid % BX;
    const int at = (unit - group * t.nseg) * len + (trow - u * len);
    if (u >= t.per || unit >= t.units || id >= np || at >= (AX == 0 ? nx : AX == 1 ? ny : nz)) return;
    const R *box = sm + ((trow + 5 * u) * BX + tid % BX) * PQ;       // stencil cell i-2
    const size_t n = (size_t)nx * ny * nz;
    const size_t p = Pencil<AX>(id, nx, ny, nz, t.cross).at(at);
    const int slow = t.cross.div(id), fast = id - slow * t.cross.d;   // the other two directions
    const int gx = AX == 0 ? at : fast, gy = AX == 0 ? fast : AX == 1 ? at : slow, gz = AX == 2 ? at : slow;
    const AdjFaceRef<R> out_ = a.face(p);

#define SMQ(q, k) box[(k) * (ST * PQ) + (q)]
    // stencil pair (dF_c, du_c) at position j
    auto X = [&](int c, int j) -> P2 {
        const int qU = c == 0 ? C_RHOQ : c == 1 ? C_MN : c == 2 ? C_MT1 : c == 3 ? C_MT2
                       : c == 4 ? (DIFF ? (int)C_DU4 : (int)C_BT1) : c == 5 ? (DIFF ? (int)C_DU5 : (int)C_BT2) : C_E;
        if constexpr (DIFF)
            return make_pair2(SMQ(C_DF0 + c, j), SMQ(qU, j));
        else
            return make_pair2(SMQ(C_F0 + c, j + 1) - SMQ(C_F0 + c, j), SMQ(qU, j + 1) - SMQ(qU, j));
    };
    auto mean = [&](int q) { return m::half_(SMQ(q, 2) + SMQ(q, 3)); };
    const R r = mean(C_RHO), vn = mean(C_VN), vt1 = mean(C_VT1), vt2 = mean(C_VT2);
    const R Bn = mean(C_BN), Bt1 = mean(C_BT1), Bt2 = mean(C_BT2), P = mean(C_P);
    const R v2 = vn * vn + vt1 * vt1 + vt2 * vt2;
    const R hv2 = m::half_(v2);
    const FaceEigen<R> e = face_eigen<R>(r, v2, Bn, Bt1, Bt2, P, K);
    const R b1 = e.b1, b2 = e.b2, sg = e.sg;
    const R pre = m::half_(e.ics2), tau = K.gm1 * e.ics2;
    const R afcf = e.af * e.cf, ascl = e.as * e.csl;
    const R sas = sg * ascl, saf = sg * afcf;
    const R eps3 = R(1.0 / 3.0) * K.eps_w;
    const R cF = pre * (K.gm1 * e.af), cS = pre * (K.gm1 * e.as);
    const R srcs = pre * (e.sr * e.cs);
    const R hF = srcs * e.as, hS = -(srcs * e.af);
    const R nF = -(pre * afcf), nS = -(pre * ascl), kF = pre * sas, kS = -(pre * saf);
    const R ssr = sg * e.sr;
    const R a5 = ssr * b1, a4 = -(ssr * b2);
    const R csisr = e.cs * e.isr;

    // ---- adjoint of the frame flux, in units of the WENO parts
    const R kw = R(1.0 / 24.0);   // field_rev carries 12 phi_N in both types
    R lX0[7], lW[7];
    {
        const size_t hi = AX == 0 ? (size_t)wrapi(gx + 1, nx) + (size_t)nx * ((size_t)gy + (size_t)ny * gz)
                          : AX == 1 ? (size_t)gx + (size_t)nx * ((size_t)wrapi(gy + 1, ny) + (size_t)ny * gz)
                                    : (size_t)gx + (size_t)nx * ((size_t)gy + (size_t)ny * wrapi(gz + 1, nz));
        auto below = [&](int ax) {
            return ax == 0 ? (size_t)wrapi(gx - 1, nx) + (size_t)nx * ((size_t)gy + (size_t)ny * gz)
                   : ax == 1 ? (size_t)gx + (size_t)nx * ((size_t)wrapi(gy - 1, ny) + (size_t)ny * gz)
                             : (size_t)gx + (size_t)nx * ((size_t)gy + (size_t)ny * wrapi(gz - 1, nz));
        };
        constexpr int t1 = (AX + 1) % 3, t2 = (AX + 2) % 3;
        auto lF = [&](int f) {
            const double *L = a.lamD + (size_t)f * n;
            return from_double<R>(a.rd * (L[hi] - L[p]));
        };
        lX0[0] = lF(0);
        lX0[1] = lF(1 + AX);
        lX0[2] = lF(1 + t1);
        lX0[3] = lF(1 + t2);
        const double *On = a.lamO + (size_t)AX * n, *O2 = a.lamO + (size_t)t2 * n;
        lX0[4] = from_double<R>(-0.5 * (On[p] + On[below(t1)]));
        lX0[5] = from_double<R>(0.5 * (O2[p] + O2[below(t2)]));
        lX0[6] = lF(4);
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) lW[c] = kw * lX0[c];
    const R lS1 = lW[0] + vn * lW[1] + vt1 * lW[2] + vt2 * lW[3] + hv2 * lW[6];
    const R lTn = lW[1] + vn * lW[6], lT1 = lW[2] + vt1 * lW[6], lT2 = lW[3] + vt2 * lW[6];
    const R lS2 = b1 * lW[4] + b2 * lW[5], lhda = b1 * lW[5] - b2 * lW[4];
    const R lTk = b1 * lT1 + b2 * lT2, lhsa = b1 * lT2 - b2 * lT1;
    const R lmg = lS1 - K.g2 * e.cs2 * lW[6];
    const R lsf = e.af * lmg + csisr * e.as * lS2 + afcf * e.cf * lW[6];
    const R lss = e.as * lmg - csisr * e.af * lS2 + ascl * e.csl * lW[6];
    const R ldf = sas * lTk - afcf * lTn, lds = -(ascl * lTn + saf * lTk);
    const R lsa = m::half_(lhsa), lda = m::half_(lhda) * (sg * e.isr);

    // ---- field projections (as face_flux; g with the field part -B_t in full)
    struct Proj {
        P2 Yn, Y1, Y2, h, k, g;
    };
    auto project = [&](P2 X0, P2 X1, P2 X2, P2 X3, P2 X4, P2 X5, P2 X6) -> Proj {
        Proj q;
        q.Yn = pfma(-vn, X0, X1);
        q.Y1 = pfma(-vt1, X0, X2);
        q.Y2 = pfma(-vt2, X0, X3);
        q.h = pfma(b1, X4, pmul(b2, X5));
        q.k = pfma(b1, q.Y1, pmul(b2, q.Y2));
        P2 g = pfma(-hv2, X0, X6);
        g = pfma(-vn, q.Yn, g);
        g = pfma(-vt1, q.Y1, g);
        g = pfma(-vt2, q.Y2, g);
        g = pfma(-Bt1, X4, g);
        q.g = pfma(-Bt2, X5, g);
        return q;
    };
    P2 F[7][5];
    // in double the projections are kept (in local memory) for the transposes,
    // in float they are formed again: 13 operations against 12 loads
    [[maybe_unused]] Proj kept[float_based<R> ? 1 : 5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const P2 X0 = X(0, j), X4 = X(4, j), X5 = X(5, j);
        const Proj q = project(X0, X(1, j), X(2, j), X(3, j), X4, X5, X(6, j));
        if constexpr (!float_based<R>) kept[j] = q;
        const P2 x = pfma(b1, q.Y2, pmul(-b2, q.Y1));
        mode_pair(pfma(cF, q.g, pmul(hF, q.h)), nF, q.Yn, kF, q.k, F[0][j], F[1][j]);
        mode_pair(pfma(cS, q.g, pmul(hS, q.h)), nS, q.Yn, kS, q.k, F[2][j], F[3][j]);
        mode_pair(x, a4, X4, a5, X5, F[4][j], F[5][j]);
        F[6][j] = pfma(-tau, q.g, X0);
    }
    // ---- WENO parts and gradients, field by field: fast -+, slow -+, Alfven
    // -+, entropy.  LF speeds: alpha = max over the two cells of |v_n + s c|,
    // with the cell and sign that attain it.  In double one copy of the code
    // in a loop, the projections in local memory (unrolled, the scheduler
    // mixes the fields and spills four times as much); in float unrolled.
    R V[7], gs[7];
    const R lf[7] = {lsf + ldf, lsf - ldf, lss + lds, lss - lds, lsa + lda, lsa - lda, lS1};
    unsigned lower = 0;
    constexpr int kUnroll = float_based<R> ? 7 : 1;
#pragma unroll kUnroll
    for (int mo = 0; mo < 7; ++mo) {
        const int qc = mo < 2 ? C_CF : mo < 4 ? C_CSL : C_CA;
        const R s = mo == 6 ? R(0) : (mo & 1) ? R(1) : R(-1);
        const R xL = m::fma_(s, SMQ(qc, 2), SMQ(C_VN, 2)), xR = m::fma_(s, SMQ(qc, 3), SMQ(C_VN, 3));
        const bool lo = m::abs_(xL) >= m::abs_(xR);
        const R xa = lo ? xL : xR;
        P2 f[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) f[j] = F[mo][j];
        R ga;
        V[mo] = field_rev<R, VAR>(f, m::abs_(xa), mo == 4 || mo == 5 ? R(4) * eps3 : eps3, lf[mo], ga);
        gs[mo] = m::nonneg(xa) ? ga : -ga;
        lower |= lo ? 1u << mo : 0u;
#pragma unroll
        for (int j = 0; j < 5; ++j) F[mo][j] = f[j];
    }
    R side[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int mo = 0; mo < 7; ++mo) {
        const int o = mo < 2 ? 1 : mo < 4 ? 3 : 2;
        const R gL = (lower >> mo) & 1u ? gs[mo] : R(0), gR = (lower >> mo) & 1u ? R(0) : gs[mo];
        side[0] += gL;
        side[4] += gR;
        if (mo < 6) {
            side[o] += (mo & 1) ? gL : -gL;
            side[4 + o] += (mo & 1) ? gR : -gR;
        }
    }
    R sf = V[0] + V[1], df = V[0] - V[1], ss = V[2] + V[3], ds = V[2] - V[3], sa = V[4] + V[5], da = V[4] - V[5], Fe = V[6];

    // ---- transposes of the projections.  The stencil differences are read
    // again: the compiler may not keep the first reads' 70 values across the
    // WENO parts.
    asm volatile("" ::: "memory");
    R lhv2 = 0, lvn = 0, lvt1 = 0, lvt2 = 0, lBt1 = 0, lBt2 = 0, lb1 = 0, lb2 = 0, ltau = 0;
    R lcF = 0, lcS = 0, lhF = 0, lhS = 0, lnF = 0, lnS = 0, lkF = 0, lkS = 0, la4 = 0, la5 = 0;
    // position j: from the pairs X, their projections and the fields' adjoints
    // to the adjoint of X
    auto transpose = [&](P2 X0, P2 X4, P2 X5, const Proj &q, P2 Lfu, P2 Lfl, P2 Lsu, P2 Lsl, P2 Lau, P2 Lal, P2 Len, P2 (&out)[7]) {
        const P2 Yn = q.Yn, Y1 = q.Y1, Y2 = q.Y2, h = q.h, k = q.k, g = q.g;
        const P2 fc = padd(Lfu, Lfl), fs = psub(Lfu, Lfl), sc = padd(Lsu, Lsl), sd = psub(Lsu, Lsl);
        const P2 lx = padd(Lau, Lal), ls = psub(Lau, Lal);
        pdot(lcF, g, fc);
        pdot(lhF, h, fc);
        pdot(lnF, Yn, fs);
        pdot(lkF, k, fs);
        pdot(lcS, g, sc);
        pdot(lhS, h, sc);
        pdot(lnS, Yn, sd);
        pdot(lkS, k, sd);
        pdot(la4, X4, ls);
        pdot(la5, X5, ls);
        pdots(ltau, g, Len);
        const P2 lg = pfma(-tau, Len, pfma(cF, fc, pmul(cS, sc)));
        const P2 lh = pfma(hF, fc, pmul(hS, sc));
        const P2 lk = pfma(kF, fs, pmul(kS, sd));
        P2 lYn = pfma(nF, fs, pmul(nS, sd));
        // k = b1 Y1 + b2 Y2, x = b1 Y2 - b2 Y1, h = b1 X4 + b2 X5
        P2 lY1 = pfma(b1, lk, pmul(-b2, lx)), lY2 = pfma(b2, lk, pmul(b1, lx));
        pdot(lb1, Y1, lk);
        pdot(lb2, Y2, lk);
        pdot(lb1, Y2, lx);
        pdots(lb2, Y1, lx);
        pdot(lb1, X4, lh);
        pdot(lb2, X5, lh);
        // g = X6 - v^2/2 X0 - v.Y - B_t.X_B
        pdots(lhv2, X0, lg);
        pdots(lvn, Yn, lg);
        pdots(lvt1, Y1, lg);
        pdots(lvt2, Y2, lg);
        pdots(lBt1, X4, lg);
        pdots(lBt2, X5, lg);
        lYn = pfma(-vn, lg, lYn);
        lY1 = pfma(-vt1, lg, lY1);
        lY2 = pfma(-vt2, lg, lY2);
        out[6] = lg;
        out[4] = pfma(a4, ls, pfma(b1, lh, pmul(-Bt1, lg)));
        out[5] = pfma(a5, ls, pfma(b2, lh, pmul(-Bt2, lg)));
        // Y = X_m - v X0
        out[1] = lYn;
        out[2] = lY1;
        out[3] = lY2;
        pdots(lvn, X0, lYn);
        pdots(lvt1, X0, lY1);
        pdots(lvt2, X0, lY2);
        out[0] = pfma(-hv2, lg, pfma(-vn, lYn, pfma(-vt1, lY1, pfma(-vt2, lY2, Len))));
    };
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        P2 out[7];
        const P2 X0 = X(0, j), X4 = X(4, j), X5 = X(5, j);
        Proj q;
        if constexpr (float_based<R>)
            q = project(X0, X(1, j), X(2, j), X(3, j), X4, X5, X(6, j));
        else
            q = kept[j];
        transpose(X0, X4, X5, q, F[0][j], F[1][j], F[2][j], F[3][j], F[4][j], F[5][j], F[6][j], out);
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            out_[kAdjDiff + (c * 5 + j) * 2] = pair_x(out[c]);
            out_[kAdjDiff + (c * 5 + j) * 2 + 1] = pair_y(out[c]);
        }
    }
    if (!e.apart) {
        // Appendix A's fallback: the central flux went through L and R, each
        // field's central part added to its WENO part (in units of kw)
        P2 Xc[7], out[7];
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            R x;
            if constexpr (DIFF)
                x = SMQ(C_F0 + c, 2) + (R(6) * SMQ(C_DF0 + c, 2) + SMQ(C_DF0 + c, 1) - SMQ(C_DF0 + c, 3)) * R(1.0 / 12.0);
            else
                x = (R(7) * (SMQ(C_F0 + c, 2) + SMQ(C_F0 + c, 3)) - (SMQ(C_F0 + c, 1) + SMQ(C_F0 + c, 4))) * R(1.0 / 12.0);
            Xc[c] = make_pair2(x, R(0));
        }
        const R u = R(24);
        auto one = [&](R l) { return make_pair2(u * l, R(0)); };
        const Proj q = project(Xc[0], Xc[1], Xc[2], Xc[3], Xc[4], Xc[5], Xc[6]);
        transpose(Xc[0], Xc[4], Xc[5], q, one(lsf + ldf), one(lsf - ldf), one(lss + lds), one(lss - lds), one(lsa + lda),
                  one(lsa - lda), one(lS1), out);
#pragma unroll
        for (int c = 0; c < 7; ++c) lX0[c] = pair_x(out[c]);
        const R Yn = pair_x(q.Yn), Y1 = pair_x(q.Y1), Y2 = pair_x(q.Y2), h = pair_x(q.h), k = pair_x(q.k), g = pair_x(q.g);
        sf += R(2) * u * (cF * g + hF * h);
        df += R(2) * u * (nF * Yn + kF * k);
        ss += R(2) * u * (cS * g + hS * h);
        ds += R(2) * u * (nS * Yn + kS * k);
        sa += R(2) * u * (b1 * Y2 - b2 * Y1);
        da += R(2) * u * (a4 * pair_x(Xc[4]) + a5 * pair_x(Xc[5]));
        Fe += u * (pair_x(Xc[0]) - tau * g);
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) out_[kAdjCentral + c] = lX0[c];
#pragma unroll
    for (int t = 0; t < 8; ++t) out_[kAdjSide + t] = side[t];
#undef SMQ

    // ---- back-projection's scalars
    R lafcf = 0, lascl = 0, laf, las, lcf, lcsl, lcs, lisr, lsr, lcs2, lpre;
    {
        const R mg = e.af * sf + e.as * ss, S1 = mg + Fe, D2 = e.as * sf - e.af * ss, S2 = csisr * D2;
        const R hsa = m::half_(sa), hda = m::half_(da) * (sg * e.isr);
        const R Tn = -(afcf * df + ascl * ds), Tk = sas * df - saf * ds;
        const R Tt1 = Tk * b1 - hsa * b2, Tt2 = Tk * b2 + hsa * b1;
        lvn += lW[1] * S1 + lW[6] * Tn;
        lvt1 += lW[2] * S1 + lW[6] * Tt1;
        lvt2 += lW[3] * S1 + lW[6] * Tt2;
        lhv2 += lW[6] * S1;
        lb1 += lT1 * Tk + lT2 * hsa + lW[4] * S2 + lW[5] * hda;
        lb2 += lT2 * Tk - lT1 * hsa + lW[5] * S2 - lW[4] * hda;
        lisr = lhda * m::half_(da) * sg + lS2 * e.cs * D2;
        lcs = lS2 * e.isr * D2;
        laf = lmg * sf - lS2 * csisr * ss;
        las = lmg * ss + lS2 * csisr * sf;
        const R sT = sg * lTk;
        lafcf = lW[6] * e.cf * sf - lTn * df - sT * ds;
        lascl = lW[6] * e.csl * ss - lTn * ds + sT * df;
        lcf = lW[6] * afcf * sf;
        lcsl = lW[6] * ascl * ss;
        lcs2 = -(K.g2 * lW[6] * mg);
    }
    // ---- projection coefficients
    {
        const R lsrcs = lhF * e.as - lhS * e.af;
        lpre = K.gm1 * (lcF * e.af + lcS * e.as) + lsrcs * (e.sr * e.cs) - lnF * afcf - lnS * ascl + lkF * sas - lkS * saf;
        laf += lcF * (pre * K.gm1) - lhS * srcs;
        las += lcS * (pre * K.gm1) + lhF * srcs;
        lsr = pre * lsrcs * e.cs + sg * (b1 * la5 - b2 * la4);
        lcs += pre * lsrcs * e.sr;
        lafcf -= pre * (lnF + sg * lkS);
        lascl += pre * (sg * lkF - lnS);
        lb1 += ssr * la5;
        lb2 -= ssr * la4;
        laf += lafcf * e.cf;
        lcf += lafcf * e.af;
        las += lascl * e.csl;
        lcsl += lascl * e.as;
        const R lics2 = K.gm1 * ltau + m::half_(lpre);
        lcs2 -= e.ics2 * (e.ics2 * lics2);
    }
    // ---- eigen scalars (face_eigen) backwards
    const R ir = e.isr * e.isr;
    const R ca2 = Bn * Bn * ir, btm = Bt1 * Bt1 + Bt2 * Bt2, bt2 = btm * ir;
    R lir = lisr * e.sr;                       // isr = sr ir
    lsr += lisr * ir;
    R lr = m::half_(lsr * e.isr);              // sr = sqrt(r)
    R lbtm = R(0);
    if (m::gt_pos(btm, K.eps_b)) {
        const R ib = m::rsqrt_(btm);
        lBt1 += lb1 * ib;
        lBt2 += lb2 * ib;
        lbtm = -m::half_(ib * (ib * (ib * (lb1 * Bt1 + lb2 * Bt2))));
    }
    R lfmc = R(0), lcms = R(0);
    if (e.apart) {
        R fmc, cms, cf2;
        speeds_fast<R>(e.cs2, ca2, bt2, fmc, cms, cf2);
        const R idf = m::rcp3_(fmc + cms);
        // a_f = sqrt(cms idf), a_s = sqrt(fmc idf)
        const R lqa = m::normal_pos(e.af) ? m::half_(laf * m::rcp3_(e.af)) : R(0);
        const R lqs = m::normal_pos(e.as) ? m::half_(las * m::rcp3_(e.as)) : R(0);
        const R ldfs = -(idf * (idf * (lqa * cms + lqs * fmc)));
        lcms = lqa * idf + ldfs;
        lfmc = lqs * idf + ldfs;
    }
    const R ics = e.cs * e.ics2;
    lcs2 += m::half_(lcs * ics);
    const R lcsl2 = m::normal_pos(e.csl) ? m::half_(lcsl * m::rcp3_(e.csl)) : R(0);
    const R lcf2 = m::normal_pos(e.cf) ? m::half_(lcf * m::rcp3_(e.cf)) : R(0);
    R lca2 = R(0), lbt2 = R(0), lP = R(0), lv2 = m::half_(lhv2);
    speeds_rev<R>(e.cs2, ca2, bt2, lfmc, lcms, lcf2, lcsl2, lcs2, lca2, lbt2);
    bool bound = false;
    if constexpr (float_based<R>) bound = K.cs2_rel * (v2 + ca2 + bt2) > K.gamma * P * ir;
    if (bound) {
        const R t = K.cs2_rel * lcs2;
        lv2 += t;
        lca2 += t;
        lbt2 += t;
    } else {
        lP = K.gamma * ir * lcs2;
        lir += K.gamma * P * lcs2;
    }
    lvn += R(2) * vn * lv2;
    lvt1 += R(2) * vt1 * lv2;
    lvt2 += R(2) * vt2 * lv2;
    lbtm += ir * lbt2;
    lir += btm * lbt2 + Bn * Bn * lca2;
    lBt1 += R(2) * Bt1 * lbtm;
    lBt2 += R(2) * Bt2 * lbtm;
    lr -= ir * (ir * lir);
    const R lw[8] = {lr, lvn, lvt1, lvt2, R(2) * Bn * ir * lca2, lBt1, lBt2, lP};
#pragma unroll
    for (int t = 0; t < 8; ++t) out_[kAdjPrim + t] = lw[t];
}

// Reverse of cell_fill<R, AX>: given the adjoints lq of a cell's 23
// quantities, the adjoints of its eight inputs (rho, m_x, m_y, m_z, E, B_x,
// B_y, B_z) in out: the primitives and the flux (Eq. P and Eq. fluxes), and
// the three wave speeds through speeds_rev.  The floors, when they apply, cut
// the dependence as in the forward step.
template <typename R, int AX>
__device__ __forceinline__ void cell_fill_adjoint(const R (&in)[8], const R (&lq)[NCQ], const Phys<R> &K, R (&out)[8]) {
    using m = M<R>;
    constexpr int n = AX, t1 = (AX + 1) % 3, t2 = (AX + 2) % 3;
    const R rho = in[0], mn = in[1 + n], m1 = in[1 + t1], m2 = in[1 + t2], E = in[4];
    const R Bn = in[5 + n], B1 = in[5 + t1], B2 = in[5 + t2];
    R r = rho;
    bool rfloor = false, pfloor = false;
    if (K.floors && r < K.rho_min) {
        r = K.rho_min;
        rfloor = true;
    }
    const R isr = m::rsqrt_(r), ir = isr * isr;
    const R vn = mn * ir, v1 = m1 * ir, v2 = m2 * ir;
    const R vv = vn * vn + v1 * v1 + v2 * v2;
    const R Bn2 = Bn * Bn, Bt2 = B1 * B1 + B2 * B2;
    const R BB = Bn2 + Bt2;
    R P = K.gm1 * (E - R(0.5) * (r * vv + BB));
    if (K.floors && P < K.p_min) {
        P = K.p_min;
        pfloor = true;
    }
    const R Pt = P + R(0.5) * BB;
    const R vB = vn * Bn + v1 * B1 + v2 * B2;
    R lr = lq[C_RHO], lvn = lq[C_VN], lv1 = lq[C_VT1], lv2 = lq[C_VT2];
    R lBn = lq[C_BN], lB1 = lq[C_BT1], lB2 = lq[C_BT2], lP = lq[C_P];
    R lE = lq[C_E], lmn = lq[C_MN], lm1 = lq[C_MT1], lm2 = lq[C_MT2], lrho = lq[C_RHOQ];
    // F0 = r vn, F1 = r vn^2 + Pt - Bn^2, F2 = r vn v1 - Bn B1, F3 = r vn v2 - Bn B2,
    // F4 = B1 vn - Bn v1, F5 = B2 vn - Bn v2, F6 = (E + Pt) vn - Bn vB
    const R f0 = lq[C_F0], f1 = lq[C_F1], f2 = lq[C_F2], f3 = lq[C_F3], f4 = lq[C_F4], f5 = lq[C_F5], f6 = lq[C_F6];
    const R fv = f0 + f1 * vn + f2 * v1 + f3 * v2;      // adjoint of r vn times the rest
    lr += fv * vn;
    lvn += r * (fv + f1 * vn) + f4 * B1 + f5 * B2 + f6 * (E + Pt);
    lv1 += r * (f2 * vn) - f4 * Bn;
    lv2 += r * (f3 * vn) - f5 * Bn;
    lBn -= R(2) * f1 * Bn + f2 * B1 + f3 * B2 + f4 * v1 + f5 * v2 + f6 * vB;
    lB1 += f4 * vn - f2 * Bn;
    lB2 += f5 * vn - f3 * Bn;
    lE += f6 * vn;
    const R lPt = f1 + f6 * vn, lvB = -(f6 * Bn);
    // vB = vn Bn + v1 B1 + v2 B2; Pt = P + BB/2
    lvn += lvB * Bn;
    lv1 += lvB * B1;
    lv2 += lvB * B2;
    lBn += lvB * vn + lPt * Bn;
    lB1 += lvB * v1 + lPt * B1;
    lB2 += lvB * v2 + lPt * B2;
    lP += lPt;
    // wave speeds c_f, c_A, c_slow of the cell from (r, P, Bn, B1, B2); |Bn| and
    // sqrt(0) take the sign of Bn and the subgradient 0
    {
        const R lcf = lq[C_CF], lca = lq[C_CA], lcs = lq[C_CSL];
        const R cs2 = K.gamma * P * ir, ca2 = Bn2 * ir, bt2 = Bt2 * ir;
        R fmc, cms, cf2;
        speeds_fast<R>(cs2, ca2, bt2, fmc, cms, cf2);
        const R icf2 = m::normal_pos(cf2) ? m::rcp3_(cf2) : R(0);
        const R csl2 = (cs2 * icf2) * ca2;
        const R lcf2 = m::normal_pos(cf2) ? m::half_(lcf * m::rsqrt_(cf2)) : R(0);
        const R lcsl2 = m::normal_pos(csl2) ? m::half_(lcs * m::rsqrt_(csl2)) : R(0);
        R lcs2 = R(0), lca2 = R(0), lbt2 = R(0);
        speeds_rev<R>(cs2, ca2, bt2, R(0), R(0), lcf2, lcsl2, lcs2, lca2, lbt2);
        // c_A = |Bn| / sqrt(r)
        const R g = Bn >= R(0) ? lca : -lca;
        lBn += g * isr;
        lr -= m::half_(g * Bn) * (isr * ir);
        // cs2 = gamma P / r, ca2 = Bn^2 / r, bt2 = (B1^2 + B2^2) / r
        lP += K.gamma * ir * lcs2;
        lBn += R(2) * Bn * ir * lca2;
        lB1 += R(2) * B1 * ir * lbt2;
        lB2 += R(2) * B2 * ir * lbt2;
        const R lirr = K.gamma * P * lcs2 + Bn2 * lca2 + Bt2 * lbt2;
        lr -= ir * (ir * lirr);
    }
    // P = gm1 (E - r vv / 2 - BB / 2)
    if (!pfloor) {
        const R gl = K.gm1 * lP;
        lE += gl;
        lr -= R(0.5) * vv * gl;
        lvn -= r * vn * gl;
        lv1 -= r * v1 * gl;
        lv2 -= r * v2 * gl;
        lBn -= Bn * gl;
        lB1 -= B1 * gl;
        lB2 -= B2 * gl;
    }
    // v = m / r
    lmn += lvn * ir;
    lm1 += lv1 * ir;
    lm2 += lv2 * ir;
    lr -= (lvn * vn + lv1 * v1 + lv2 * v2) * ir;
    if (!rfloor) lrho += lr;
    out[0] = lrho;
    out[1 + n] = lmn;
    out[1 + t1] = lm1;
    out[1 + t2] = lm2;
    out[4] = lE;
    out[5 + n] = lBn;
    out[5 + t1] = lB1;
    out[5 + t2] = lB2;
}

// A sum over faces.  The face adjoints that meet in a cell cancel (a difference's
// sum against its neighbour's above all), so a float sum would lose what float
// adjoints hold: in double a plain sum; in float the running sum and the sum of
// its rounding errors (TwoSum), which together keep 48 bits until value()
// rounds once.  64^3 FP32 gradient, three steps: 6.67 ms with float sums, 6.92 with
// these pairs, 15.8 with sums in double (conversions and the FP64 pipe), the
// gradient 3.3e-6 from 64 bits in all three.  The rounding errors of an infinite
// sum are not numbers and are left out.
template <typename R> struct FaceSum;
template <> struct FaceSum<double> {
    double s;
    static __device__ __forceinline__ FaceSum of(double x) { return {x}; }
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void add(const FaceSum &x) { s += x.s; }
    __device__ __forceinline__ FaceSum minus(const FaceSum &x) const { return {s - x.s}; }
    __device__ __forceinline__ double value() const { return s; }
    // (7 (a + b) - (c + d)) / 12
    static __device__ __forceinline__ FaceSum central(double a, double b, double c, double d) {
        return {(7.0 * (a + b) - (c + d)) * (1.0 / 12.0)};
    }
};
template <> struct FaceSum<float> {
    float s, e;
    static __device__ __forceinline__ FaceSum of(float x) { return {x, 0.0f}; }
    __device__ __forceinline__ void add(float x) {
        const dw t = ef_twosum(s, x);
        s = t.hi;
        e = __fadd_rn(e, t.lo);
    }
    __device__ __forceinline__ void add(const FaceSum &x) {
        add(x.s);
        e = __fadd_rn(e, x.e);
    }
    __device__ __forceinline__ FaceSum minus(const FaceSum &x) const {
        FaceSum d = *this;
        d.add(FaceSum{-x.s, -x.e});
        return d;
    }
    __device__ __forceinline__ float value() const {
        const float v = __fadd_rn(s, e);
        return v == v ? v : s;
    }
    static __device__ __forceinline__ FaceSum central(float a, float b, float c, float d) {
        const dw p = ef_twoprod(7.0f, a), q = ef_twoprod(7.0f, b);
        FaceSum t = {p.hi, __fadd_rn(p.lo, q.lo)};
        t.add(q.hi);
        t.add(-c);
        t.add(-d);
        const float k = 1.0f / 12.0f;
        const dw r = ef_twoprod(t.s, k);
        return {r.hi, __fmaf_rn(t.e, k, r.lo)};
    }
};

// A cell of a tile of segments (AdjTile): the adjoint of the difference between
// cells d and d + 1 is the sum of the face adjoints at position j over the five
// faces d + 2 - j that read it, formed once per difference (a segment's first
// cell also needs the one below it) and kept in shared memory; a flux or conserved component of cell i then takes D(i-1) -
// D(i), plus, for the flux, the central combinations of four faces.  Fixed
// order throughout; every sum over faces is a FaceSum.
constexpr int kAdjCellEntries = 384;       // differences of a block
template <int AX, typename R>
__global__ void __launch_bounds__(256) adj_cell_kernel(AdjSweepArgs<R> a) {
    using Sum = FaceSum<R>;
    constexpr int BX = AX == 0 ? 1 : 32;
    __shared__ Sum acc[14][kAdjCellEntries];
    const int nx = a.nx, ny = a.ny, nz = a.nz, tid = threadIdx.x;
    const size_t n = (size_t)nx * ny * nz;
    const AdjTile &t = a.cell_tile;
    const int len = t.len, rows = len + 1, np = pencils<AX>(nx, ny, nz), first = (int)blockIdx.x * t.per;
    // entry (unit u, row r, pencil b) at (u rows + r) BX + b: the difference
    // between positions r - 1 and r of the unit's segment
    const int entries = BX * t.per * rows;
    for (int e = tid; e < entries; e += 256) {
        const int row = e / BX, u = t.rows.div(row), unit = first + u, group = t.segments.div(unit);
        const int id = group * BX + e % BX, at = (unit - group * t.nseg) * len + (row - u * rows) - 1;
        if (unit >= t.units || id >= np) continue;
        const Pencil<AX> pen(id, nx, ny, nz, t.cross);
        if (at >= pen.n) continue;
        AdjFaceRef<R> f[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) f[j] = a.face(pen.at(wrapi(at + 2 - j, pen.n)));
#pragma unroll
        for (int c = 0; c < 14; ++c) {
            Sum s = Sum::of(f[0][kAdjDiff + (c % 7) * 10 + c / 7]);
#pragma unroll
            for (int j = 1; j < 5; ++j) s.add(f[j][kAdjDiff + ((c % 7) * 5 + j) * 2 + c / 7]);
            acc[c][e] = s;
        }
    }
    __syncthreads();
    const int trow = tid / BX, u = t.positions.div(trow), unit = first + u, group = t.segments.div(unit);
    const int id = group * BX + tid % BX, at = (unit - group * t.nseg) * len + (trow - u * len);
    if (u >= t.per || unit >= t.units || id >= np) return;
    const Pencil<AX> pen(id, nx, ny, nz, t.cross);
    if (at >= pen.n) return;
    const int below_ = (trow + u) * BX + tid % BX;         // D(i - 1); D(i) one row on
    const size_t p = pen.at(at), pm = pen.at(wrapi(at - 1, pen.n));
    const AdjFaceRef<R> f0 = a.face(p), fm = a.face(pm), fm2 = a.face(pen.at(wrapi(at - 2, pen.n))),
                        fp = a.face(pen.at(wrapi(at + 1, pen.n)));
    const int slow = t.cross.div(id), fast = id - slow * t.cross.d;
    const int gx = AX == 0 ? at : fast, gy = AX == 0 ? fast : AX == 1 ? at : slow, gz = AX == 2 ? at : slow;
    constexpr int t1 = (AX + 1) % 3, t2 = (AX + 2) % 3;
    R cell[8], lq[NCQ];
#pragma unroll
    for (int f = 0; f < 5; ++f) cell[f] = a.q[f][p];
#pragma unroll
    for (int f = 0; f < 3; ++f) cell[5 + f] = a.bc[f][p];
    auto D = [&](int c) { return acc[c][below_].minus(acc[c][below_ + BX]); };
    // a primitive in the interface means, and a speed of the cell: the lower cell
    // of its own face, the upper one of the face before
    auto mean = [&](int t) {
        Sum v = Sum::of(R(0.5) * f0[kAdjPrim + t]);
        v.add(R(0.5) * fm[kAdjPrim + t]);
        return v;
    };
    auto side = [&](int k) {
        Sum v = Sum::of(f0[kAdjSide + k]);
        v.add(fm[kAdjSide + 4 + k]);
        return v;
    };
    // transport fluxes <B_n v_t>: half the sum of the two faces' adjoints
    R tn, tv1, tv2;
    {
        // of the cell `o` along the sweep (0 or -1), the neighbour below along ax
        auto below = [&](int ax, int o) {
            const int x = ax == 0 ? wrapi(gx - 1, nx) : AX == 0 ? wrapi(gx + o, nx) : gx;
            const int y = ax == 1 ? wrapi(gy - 1, ny) : AX == 1 ? wrapi(gy + o, ny) : gy;
            const int z = ax == 2 ? wrapi(gz - 1, nz) : AX == 2 ? wrapi(gz + o, nz) : gz;
            return (size_t)x + (size_t)nx * ((size_t)y + (size_t)ny * (size_t)z);
        };
        const double *On = a.lamO + (size_t)AX * n, *O2 = a.lamO + (size_t)t2 * n;
        const R l1 = from_double<R>(-0.25 * ((On[p] + On[below(t1, 0)]) + (On[pm] + On[below(t1, -1)])));
        const R l2 = from_double<R>(0.25 * ((O2[p] + O2[below(t2, 0)]) + (O2[pm] + O2[below(t2, -1)])));
        const R ir = M<R>::rcp3_(a.K.floors ? M<R>::max_(cell[0], a.K.rho_min) : cell[0]);
        tn = (l1 * cell[1 + t1] + l2 * cell[1 + t2]) * ir;
        tv1 = l1 * cell[5 + AX];
        tv2 = l2 * cell[5 + AX];
    }
    constexpr int qU[7] = {C_RHOQ, C_MN, C_MT1, C_MT2, C_BT1, C_BT2, C_E};
    constexpr int prim[8] = {C_RHO, C_VN, C_VT1, C_VT2, C_BN, C_BT1, C_BT2, C_P};
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        Sum v = mean(t);
        if (prim[t] == C_VN) v.add(side(0));
        if (prim[t] == C_VT1) v.add(tv1);
        if (prim[t] == C_VT2) v.add(tv2);
        if (prim[t] == C_BN) v.add(tn);
        if (prim[t] == C_BT1) v.add(D(7 + 4));
        if (prim[t] == C_BT2) v.add(D(7 + 5));
        lq[prim[t]] = v.value();
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) {
        const int k = kAdjCentral + c;
        Sum v = D(c);
        v.add(Sum::central(f0[k], fm[k], fp[k], fm2[k]));
        lq[C_F0 + c] = v.value();
        if (c != 4 && c != 5) lq[qU[c]] = D(7 + c).value();
    }
    lq[C_CF] = side(1).value();
    lq[C_CA] = side(2).value();
    lq[C_CSL] = side(3).value();
    R g[8];
    cell_fill_adjoint<R, AX>(cell, lq, a.K, g);
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        double *o = v < 5 ? a.outq + (size_t)v * n : a.outb + (size_t)(v - 5) * n;
        o[p] = a.first ? to_double(g[v]) : o[p] + to_double(g[v]);
    }
}

// ---------------------------------------------------------------- linear parts

struct AdjGrid {
    int nx, ny, nz;
    double rdx, rdy, rdz;
    __device__ __forceinline__ size_t at(int i, int j, int k) const {
        return (size_t)wrapi(i, nx) + (size_t)nx * ((size_t)wrapi(j, ny) + (size_t)ny * (size_t)wrapi(k, nz));
    }
};

__device__ __forceinline__ bool adj_cell(const AdjGrid &g, int &i, int &j, int &k, size_t &p) {
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= n) return false;
    if (n <= 0x7fffffffLL) {        // (a 64-bit division costs more than most of these kernels' cells)
        const unsigned r = (unsigned)q / (unsigned)g.nx;
        i = (int)((unsigned)q - r * (unsigned)g.nx);
        k = (int)(r / (unsigned)g.ny);
        j = (int)(r - (unsigned)k * (unsigned)g.ny);
    } else {
        const long long r = q / g.nx;
        i = (int)(q - r * g.nx);
        k = (int)(r / g.ny);
        j = (int)(r - (long long)k * g.ny);
    }
    p = (size_t)q;
    return true;
}

// Stage sources: lamD = cf lamq_fin + cn lamq_next (the adjoint of the flux
// divergence) and lamO = curl^T mu, mu = cf lamb_fin + cn lamb_next, for the
// face update of Sec. 2.3:
//   db_x = -(O_x - O_x(j-1)) rdy + (O_z - O_z(k-1)) rdz
//   db_y = -(O_y - O_y(k-1)) rdz + (O_x - O_x(i-1)) rdx
//   db_z = -(O_z - O_z(i-1)) rdx + (O_y - O_y(j-1)) rdy
// The flux adjoints follow from them face by face (adj_face_kernel):
//   lamF_d = (lamD(+1 along d) - lamD) / dx_d  (transpose of Eq. num),
// and, from the EMF averages of Eqs. ox1-ox3
//   O_x = (g*_x + g*_x(i+1))/2 - (f*_y + f*_y(j+1))/2
//   O_y = (h*_y + h*_y(j+1))/2 - (g*_z + g*_z(k+1))/2
//   O_z = (f*_z + f*_z(k+1))/2 - (h*_x + h*_x(i+1))/2,
// the sweep along d (t1, t2 the next axes, cyclic) has lamS_1 = -(lamO_d +
// lamO_d(-1 along t1))/2 and lamS_2 = (lamO_t2 + lamO_t2(-1 along t2))/2.
static __global__ void __launch_bounds__(256) adj_sources_kernel(AdjGrid g, double cf, double cn,
                                                                 const double *__restrict__ lq_fin,
                                                                 const double *__restrict__ lb_fin,
                                                                 const double *__restrict__ lq_next,
                                                                 const double *__restrict__ lb_next, double *lamD,
                                                                 double *lamO) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        const size_t o = (size_t)f * n + p;
        lamD[o] = cf * lq_fin[o] + (lq_next ? cn * lq_next[o] : 0.0);
    }
    auto mu = [&](int f, size_t q) {
        const size_t o = (size_t)f * n + q;
        return cf * lb_fin[o] + (lb_next ? cn * lb_next[o] : 0.0);
    };
    const size_t px = g.at(i + 1, j, k), py = g.at(i, j + 1, k), pz = g.at(i, j, k + 1);
    const double mx = mu(0, p), my = mu(1, p), mz = mu(2, p);
    lamO[p] = g.rdy * (mu(0, py) - mx) + g.rdx * (my - mu(1, px));
    lamO[n + p] = g.rdz * (mu(1, pz) - my) + g.rdy * (mz - mu(2, py));
    lamO[2 * n + p] = g.rdz * (mx - mu(0, pz)) + g.rdx * (mu(2, px) - mz);
}

// Transpose of the fourth-order face -> centre interpolation of Sec. 2.3,
// B_d(i) = (9 (b_d(i-1) + b_d(i)) - (b_d(i-2) + b_d(i+1))) / 16 along d:
// lamb_d(m) = (9 (lamB(m+1) + lamB(m)) - (lamB(m+2) + lamB(m-1))) / 16.
// Writes lamb (3 planes) and adds lamq, lamb into the step's outputs.
static __global__ void __launch_bounds__(256) adj_interp_kernel(AdjGrid g, const double *__restrict__ lamBc,
                                                                const double *__restrict__ lamq, double *lamb,
                                                                double *out_q, double *out_b) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    const double s = 1.0 / 16.0;
    const double *Lx = lamBc, *Ly = lamBc + n, *Lz = lamBc + 2 * n;
    const double bx = (9.0 * (Lx[g.at(i + 1, j, k)] + Lx[p]) - (Lx[g.at(i + 2, j, k)] + Lx[g.at(i - 1, j, k)])) * s;
    const double by = (9.0 * (Ly[g.at(i, j + 1, k)] + Ly[p]) - (Ly[g.at(i, j + 2, k)] + Ly[g.at(i, j - 1, k)])) * s;
    const double bz = (9.0 * (Lz[g.at(i, j, k + 1)] + Lz[p]) - (Lz[g.at(i, j, k + 2)] + Lz[g.at(i, j, k - 1)])) * s;
    const double bb[3] = {bx, by, bz};
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        lamb[(size_t)f * n + p] = bb[f];
        out_b[(size_t)f * n + p] += bb[f];
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) out_q[(size_t)f * n + p] += lamq[(size_t)f * n + p];
}

// ---------------------------------------------------------------- misfit

// L = 1/2 dV sum over cells of |q - q*|^2 + |b - b*|^2 (five conserved and
// three face fields); lam = dV (q - q*), dV (b - b*).  Per-block partial sums.
static __global__ void __launch_bounds__(kRedThreads) misfit_partial_kernel(long long n, double dV, const double *q,
                                                                            const double *b, const double *tq,
                                                                            const double *tb, double *lq, double *lb,
                                                                            double *part) {
    __shared__ double red[32];
    double v[1] = {0.0};
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            const size_t o = (size_t)f * (size_t)n + (size_t)p;
            const double d = q[o] - tq[o];
            v[0] += d * d;
            lq[o] = dV * d;
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const size_t o = (size_t)f * (size_t)n + (size_t)p;
            const double d = b[o] - tb[o];
            v[0] += d * d;
            lb[o] = dV * d;
        }
    }
    bool ismax[1] = {false};
    block_reduce<double, 1>(v, ismax, red);
    if (threadIdx.x == 0) part[blockIdx.x] = 0.5 * dV * v[0];
}

// ---------------------------------------------------------------- initial state

// Face field b = curl A + B0 of an edge vector potential (A_x at (i, j+1/2,
// k+1/2), A_y at (i+1/2, j, k+1/2), A_z at (i+1/2, j+1/2, k) in cell units
// from the centre of cell (i, j, k)), first-order discrete curl (Sec. 4.1).
static __global__ void __launch_bounds__(256) ic_curl_kernel(AdjGrid g, const double *__restrict__ A, double B0x,
                                                             double B0y, double B0z, double *bface) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    const double *Ax = A, *Ay = A + n, *Az = A + 2 * n;
    bface[p] = (Az[p] - Az[g.at(i, j - 1, k)]) * g.rdy - (Ay[p] - Ay[g.at(i, j, k - 1)]) * g.rdz + B0x;
    bface[n + p] = (Ax[p] - Ax[g.at(i, j, k - 1)]) * g.rdz - (Az[p] - Az[g.at(i - 1, j, k)]) * g.rdx + B0y;
    bface[2 * n + p] = (Ay[p] - Ay[g.at(i - 1, j, k)]) * g.rdx - (Ax[p] - Ax[g.at(i, j - 1, k)]) * g.rdy + B0z;
}

// sixth-order face -> centre weights of the initial conditions (Sec. 4.14),
// faces i-5/2 .. i+5/2 = face indices i-3 .. i+2, divided by 256
__device__ __forceinline__ double ic_w6(int o) {
    return o == 0 || o == 5 ? 3.0 / 256.0 : o == 1 || o == 4 ? -25.0 / 256.0 : 150.0 / 256.0;
}

__device__ __forceinline__ void ic_cell_field(const AdjGrid &g, const double *bface, int i, int j, int k,
                                              double (&Bc)[3]) {
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    Bc[0] = Bc[1] = Bc[2] = 0.0;
#pragma unroll
    for (int o = 0; o < 6; ++o) {
        const double w = ic_w6(o);
        Bc[0] += w * bface[g.at(i - 3 + o, j, k)];
        Bc[1] += w * bface[n + g.at(i, j - 3 + o, k)];
        Bc[2] += w * bface[2 * n + g.at(i, j, k - 3 + o)];
    }
}

// conserved state (rho, rho v, E) with E from Eq. P, the cell field from the
// sixth-order interpolation of the faces
static __global__ void __launch_bounds__(256) ic_cons_kernel(AdjGrid g, double gm1, const double *__restrict__ rho,
                                                             const double *__restrict__ v, const double *__restrict__ P,
                                                             const double *__restrict__ bface, double *cons) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    double Bc[3];
    ic_cell_field(g, bface, i, j, k, Bc);
    const double r = rho[p], vx = v[p], vy = v[n + p], vz = v[2 * n + p];
    cons[p] = r;
    cons[n + p] = r * vx;
    cons[2 * n + p] = r * vy;
    cons[3 * n + p] = r * vz;
    cons[4 * n + p] = P[p] / gm1 + 0.5 * r * (vx * vx + vy * vy + vz * vz) + 0.5 * (Bc[0] * Bc[0] + Bc[1] * Bc[1] + Bc[2] * Bc[2]);
}

// adjoint of ic_cons_kernel in rho and v; lamBc = Bc lamE (3 planes, scratch)
static __global__ void __launch_bounds__(256) ic_cons_adjoint_kernel(AdjGrid g, const double *__restrict__ rho,
                                                                     const double *__restrict__ v,
                                                                     const double *__restrict__ bface,
                                                                     const double *__restrict__ lcons, double *lrho,
                                                                     double *lv, double *lBc) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    double Bc[3];
    ic_cell_field(g, bface, i, j, k, Bc);
    const double r = rho[p], vv[3] = {v[p], v[n + p], v[2 * n + p]};
    const double lE = lcons[4 * n + p];
    double lr = lcons[p] + 0.5 * lE * (vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2]);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double lm = lcons[(size_t)(1 + d) * n + p];
        lr += vv[d] * lm;
        lv[(size_t)d * n + p] = r * lm + r * vv[d] * lE;
        lBc[(size_t)d * n + p] = Bc[d] * lE;
    }
    lrho[p] = lr;
}

// lamb = lam_bface + (sixth-order interpolation)^T lamBc
static __global__ void __launch_bounds__(256) ic_interp_adjoint_kernel(AdjGrid g, const double *__restrict__ lbface,
                                                                       const double *__restrict__ lBc, double *lb) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    double s[3] = {lbface[p], lbface[n + p], lbface[2 * n + p]};
    // face m feeds cell m + 3 - o with weight w_o
#pragma unroll
    for (int o = 0; o < 6; ++o) {
        const double w = ic_w6(o);
        s[0] += w * lBc[g.at(i + 3 - o, j, k)];
        s[1] += w * lBc[n + g.at(i, j + 3 - o, k)];
        s[2] += w * lBc[2 * n + g.at(i, j, k + 3 - o)];
    }
    lb[p] = s[0];
    lb[n + p] = s[1];
    lb[2 * n + p] = s[2];
}

// lamA = curl^T lamb (transpose of ic_curl_kernel)
static __global__ void __launch_bounds__(256) ic_curl_adjoint_kernel(AdjGrid g, const double *__restrict__ lb,
                                                                     double *lA) {
    int i, j, k;
    size_t p;
    if (!adj_cell(g, i, j, k, p)) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    const double *bx = lb, *by = lb + n, *bz = lb + 2 * n;
    // b_y(i,j,k) has +A_x/dz, b_y(i,j,k+1) -A_x/dz; b_z(i,j,k) -A_x/dy, b_z(i,j+1,k) +A_x/dy
    lA[p] = (by[p] - by[g.at(i, j, k + 1)]) * g.rdz - (bz[p] - bz[g.at(i, j + 1, k)]) * g.rdy;
    // b_z: +A_y/dx at (i), -A_y/dx at (i+1); b_x: -A_y/dz at (k), +A_y/dz at (k+1)
    lA[n + p] = (bz[p] - bz[g.at(i + 1, j, k)]) * g.rdx - (bx[p] - bx[g.at(i, j, k + 1)]) * g.rdz;
    // b_x: +A_z/dy at (j), -A_z/dy at (j+1); b_y: -A_z/dx at (i), +A_z/dx at (i+1)
    lA[2 * n + p] = (bx[p] - bx[g.at(i, j + 1, k)]) * g.rdy - (by[p] - by[g.at(i + 1, j, k)]) * g.rdx;
}

// The tile of a kernel whose block has `rows` positions to give (of BX pencils
// each) and room for `room` rows, `extra` of them per segment beside its
// positions: the segment length that takes the fewest blocks, a block's cells
// counting a sixteenth of a face each.  Of blocks that leave some of the `slots`
// (SMs times blocks on each) empty, those with the fewest positions, down to a
// warp's, that still fit in the slots.
inline AdjTile adj_tile(int ax, int nx, int ny, int nz, int BX, int rows, int room, int extra, int slots) {
    const int na = ax == 0 ? nx : ax == 1 ? ny : nz;
    const long long n = (long long)nx * ny * nz, groups = (n / na + BX - 1) / BX;
    AdjTile best = {};
    for (int r = rows; r * BX >= 32; r /= 2) {
        AdjTile tile = {};
        long long fewest = 0;
        double cost = 1e300;
        for (int most = std::min(r, na); most > 0; --most) {
            const int nseg = (na + most - 1) / most, len = (na + nseg - 1) / nseg;      // (nearly equal segments)
            const int per = std::min(r / len, room / (len + extra));
            const long long units = groups * nseg, blocks = (units + per - 1) / per;
            const double c = (double)blocks * (r + per * (len + extra) / 16.0);
            if (c < 0.999 * cost) {
                cost = c;
                fewest = blocks;
                tile.len = len;
                tile.nseg = nseg;
                tile.per = per;
                tile.units = (int)units;
            }
        }
        if (r < rows && fewest > slots) break;
        best = tile;
    }
    best.rows = int_div(best.len + extra);
    best.positions = int_div(best.len);
    best.segments = int_div(best.nseg);
    best.cross = int_div(ax == 0 ? ny : nx);
    return best;
}

// The face kernel: one face per thread at up to 255 registers, eight warps per
// SM: in double 256 threads (16 pencils side by side along y and z), in float two
// blocks of 128 (8 pencils).  64^3 WENO5 rollout in float, three steps: 7.76 ms;
// one block of 256 threads 7.82, three blocks of 128 (168 registers) 7.96, four
// (128 registers) 8.49.
template <int AX, typename R, int VAR>
struct AdjFace {
    static constexpr bool kF = float_based<R>;
    static constexpr int BX = AX == 0 ? 1 : kF ? 8 : 16, NT = kF ? 128 : 256, MINB = kF ? 2 : 1;
    static constexpr size_t cell_bytes = adj_box_pitch<R>() * sizeof(R);
    static cudaError_t prepare() {
        return cudaFuncSetAttribute(adj_face_kernel<AX, R, VAR, BX, NT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(adj_box_cells<R>() * cell_bytes));
    }
    static AdjTile tile(int nx, int ny, int nz) {
        return adj_tile(AX, nx, ny, nz, BX, NT / BX, adj_box_cells<R>() / BX, 5, 152 * MINB);
    }
    static cudaError_t launch(const AdjSweepArgs<R> &a, cudaStream_t s) {
        const AdjTile &f = a.face_tile, &c = a.cell_tile;
        const size_t smem = (size_t)BX * f.per * (f.len + 5) * cell_bytes;
        adj_face_kernel<AX, R, VAR, BX, NT, MINB><<<(f.units + f.per - 1) / f.per, NT, smem, s>>>(a);
        adj_cell_kernel<AX, R><<<(c.units + c.per - 1) / c.per, 256, 0, s>>>(a);
        return cudaGetLastError();
    }
};

inline AdjTile adj_cell_tile(int ax, int nx, int ny, int nz) {
    const int BX = ax == 0 ? 1 : 32;
    return adj_tile(ax, nx, ny, nz, BX, 256 / BX, kAdjCellEntries / BX, 1, 152 * 2);
}

// The tiles of the sweep along each axis over a grid (a few hundred trial
// divisions each: once per grid, not per launch).
template <typename R>
void adj_tiles(int nx, int ny, int nz, AdjTile (&face)[3], AdjTile (&cell)[3]) {
    face[0] = AdjFace<0, R, 0>::tile(nx, ny, nz);
    face[1] = AdjFace<1, R, 0>::tile(nx, ny, nz);
    face[2] = AdjFace<2, R, 0>::tile(nx, ny, nz);
    for (int ax = 0; ax < 3; ++ax) cell[ax] = adj_cell_tile(ax, nx, ny, nz);
}

// Defined in w5ct_adjoint{32,64}{js,z}.cu (one translation unit per
// arithmetic type and WENO variant, compiled in parallel): the face and cell
// kernels along `axis`, and their shared-memory allowance.
template <typename R, int VAR>
cudaError_t launch_adj_sweep(int axis, const AdjSweepArgs<R> &a, cudaStream_t s);
template <typename R, int VAR>
cudaError_t prepare_adj_sweep();

template <typename R, int VAR>
cudaError_t launch_adj_sweep_impl(int axis, const AdjSweepArgs<R> &a, cudaStream_t s) {
    if (axis == 0) return AdjFace<0, R, VAR>::launch(a, s);
    if (axis == 1) return AdjFace<1, R, VAR>::launch(a, s);
    return AdjFace<2, R, VAR>::launch(a, s);
}

template <typename R, int VAR>
cudaError_t prepare_adj_sweep_impl() {
    cudaError_t e = AdjFace<0, R, VAR>::prepare();
    if (e == cudaSuccess) e = AdjFace<1, R, VAR>::prepare();
    if (e == cudaSuccess) e = AdjFace<2, R, VAR>::prepare();
    return e;
}

}  // namespace w5ct
