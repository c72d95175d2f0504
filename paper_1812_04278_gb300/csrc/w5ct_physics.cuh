// w5ct_physics.cuh -- device arithmetic of the WENO5 + CT ideal-MHD scheme
// of Donnert et al. (arXiv:1812.04278), templated on the arithmetic type
// (double for the FP64 path, float for the FP32-bulk path).
//
//   cell_fill  : primitives (Eq. P), flux along the sweep axis (Eq. fluxes),
//                wave speeds (Eqs. slow, fast, ca) of one cell.
//   face_flux  : characteristic WENO5 / WENO5-Z flux at one interface
//                (Sec. 2.2, Eq. FWENO) with the eigenvectors of Appendix A.
//
// Readings of the garbled passages (identical in the CPU oracle):
//   P* = P + B^2/2; fast/slow speeds from the discriminant
//   d = (c_s^2 - c_A^2)^2 + b_t^2 (b_t^2 + 2 c_A^2 + 2 c_s^2) without
//   cancellation, c_slow^2 = c_s^2 c_A^2 / c_f^2; Appendix A's "slow" block is
//   the Alfven pair (m = 2, 6) and its "Alfven" block the slow pair (m = 3, 5);
//   upper signs for m <= 3; beta normalised by |B_t|; sgn(B_n) = +1 iff
//   B_n >= eps_B; fast-mode left eigenvector with the 1/(2 c_s^2) factor on
//   every component, gamma_1 alpha_f v^2 +- Gamma_f, -+ alpha_f c_f and
//   + sqrt(rho) c_s alpha_s beta in the field rows; entropy right eigenvector
//   energy row v^2/2; interface state = mean of the two cells' primitives;
//   alpha(m) = max(|lambda_m(i)|, |lambda_m(i+1)|); WENO-Z weights
//   d_k (1 + (tau_5/(eps_Z + IS_k))^2).
#pragma once
#include <cuda_runtime.h>
#include <type_traits>

namespace w5ct {

// per-cell quantities kept in shared memory during a sweep (frame components)
enum CellQ {
    C_RHO = 0, C_VN, C_VT1, C_VT2, C_BN, C_BT1, C_BT2, C_P,   // primitives w
    C_RHOQ, C_MN, C_MT1, C_MT2, C_E,                          // conserved u (rho, m, E)
    C_F0, C_F1, C_F2, C_F3, C_F4, C_F5, C_F6,                 // flux along n
    C_CF, C_CA, C_CSL,                                        // c_fast, c_Alfven, c_slow
    NCQ
};

// The FP64 sweep's cell box holds, after its difference pass, besides the
// NCQ quantities of cell_fill_frame: the forward differences dF_c(i) =
// F_c(i+1) - F_c(i) of the seven frame fluxes (planes C_DF0..C_DF6) and
// du_c(i) = u_c(i+1) - u_c(i) of the conserved 7-vector -- in place of u_c
// for rho, m and E (planes C_RHOQ, C_MN, C_MT1, C_MT2, C_E), in C_DU4, C_DU5
// for B_t1, B_t2 (whose planes stay the primitives).
enum BoxQ { C_DF0 = NCQ, C_DU4 = NCQ + 7, C_DU5, NBQ };

// The difference pass pays in double, where the sweep is bound by the FP64
// pipe and it removes 77 FP64 operations per interface (the stencil
// differences and the central combination) for 14 per cell; in float its
// extra barriers and shared-memory traffic cost more than the FP32
// operations it saves.  Boxes of the compile-time tiles (sweep_tile_at):
template <typename Real>
__host__ __device__ constexpr bool box_diff() {
    return sizeof(Real) == 8;
}
template <typename Real>
__host__ __device__ constexpr int box_quantities() {
    return box_diff<Real>() ? NBQ : NCQ;
}

// Where quantity q of a cell lies in a box whose planes are `stride` elements
// apart.  Paired (the float sweeps): the flux and conserved component c of a
// cell are neighbours (one 8-byte load, and the packed differences need no
// regrouping), the other nine quantities (rho, v, B_n, P, the speeds) follow in
// planes of their own; B_t1, B_t2 are their conserved components.  Half the
// shared loads of the stencil and half its differences: two 256^3 WENO-Z steps
// 27.36 -> 26.92 ms.
template <bool PAIRED>
__host__ __device__ constexpr int box_at(int q, int stride, int cell) {
    if (!PAIRED) return q * stride + cell;
    const int c = q >= C_F0 && q <= C_F6 ? q - C_F0 : q >= C_RHOQ && q <= C_MT2 ? q - C_RHOQ : q == C_E ? 6
                  : q == C_BT1 ? 4 : q == C_BT2 ? 5 : -1;
    if (c >= 0) return 2 * (c * stride + cell) + (q >= C_F0 && q <= C_F6 ? 0 : 1);
    const int k = q <= C_BN ? q : q == C_P ? 5 : q - C_CF + 6;
    return (14 + k) * stride + cell;
}

template <typename Real>
struct Phys {
    Real gamma, gm1, g1, g2;     // gamma, gamma-1, (gamma-1)/2, (gamma-2)/(gamma-1)
    Real eps_w;                  // WENO epsilon (JS or Z, per the variant)
    Real eps_b;                  // eps_B of Appendix A
    Real eps_b2;                 // threshold on c_f^2 - c_slow^2 (eps_B^2, >= FLT_MIN in float)
    Real rho_min, p_min;
    // lower bound on c_s^2 in the interface eigenvectors, relative to
    // v^2 + c_A^2 + b_t^2 (0 in double; see face_flux)
    Real cs2_rel;
    int floors;
};

// float_based<Real> selects the float-specific guards of the FP32-bulk
// arithmetic.
template <typename R>
constexpr bool float_based = std::is_same<R, float>::value;

// ---------------------------------------------------------------- math helpers
template <typename Real> struct M;
// ---------------------------------------------------------------- products
// Products of doubles on the integer pipes, with the bits of an IEEE product
// rounded to nearest even.  The FP64 sweeps are bound by the FP64 pipe (2 lanes
// per SM and clock: 16 clocks for a warp's instruction) while the issue slots
// are a tenth used, and the 30 integer instructions of a product issue in 8
// clocks of an SM beside it: every product moved here is time off the bound.
// (A fused multiply-add or a sum would take twice as many and stays where it
// is.)  256^3 WENO-Z step, with the looped face function (face_flux): 413 ms
// with all products in the FP64 multiplier, 388 with the products of the
// weights moved, 371 with those of the quotients, 353 with those of the
// projections, 331 with those of the eigenvectors, cells and roots.  Groups with
// a zero factor go to the multiplier, so data with exact zeros gain less: 128^3
// WENO-Z step 66.6 -> 41.4 ms with all fields varying, 68.1 -> 43.7 with v_z = B_z = 0,
// 75.9 -> 59.7 varying along x alone with v and B along x, 77.4 -> 61.1 uniform
// (WENO5 63.0 -> 39.3, 63.2 -> 39.5, 63.3 -> 44.1, 63.3 -> 43.4; with the tiles and the
// face algebra of the same time).
//
// DFactor holds the magnitude of a factor: its 53-bit significand and its
// exponent field less one, in place.  dmul_int multiplies two of them whose
// product is normal: the first significand is shifted left by 11, so that the
// upper half of the 128-bit product is the result's significand or half of it.
struct DFactor {
    unsigned lo, hi, e;
    __device__ __forceinline__ explicit DFactor(double x) {
        const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
        lo = (unsigned)__double2loint(x);
        hi = (h & 0xfffffu) | 0x100000u;
        e = h - hi;
    }
};

__device__ __forceinline__ double dmul_int(const DFactor &a, const DFactor &b) {
    using u64 = unsigned long long;
    const unsigned ah = __funnelshift_l(a.lo, a.hi, 11), al = a.lo << 11;
    const u64 p0 = (u64)al * b.lo;
    const u64 p1 = (u64)ah * b.lo + (p0 >> 32);
    const u64 p2 = (u64)al * b.hi + (unsigned)p1;
    const u64 p3 = (u64)ah * b.hi + (p1 >> 32) + (p2 >> 32);
    const unsigned h = (unsigned)(p3 >> 32), l = (unsigned)p3, f = (unsigned)p2, z = (unsigned)p0;
    const unsigned s = (h >> 20) ^ 1u;   // 1: the upper half lacks its top bit
    unsigned m1 = __funnelshift_l(l, h, s), m0 = __funnelshift_l(f, l, s);
    const unsigned r = f << s;
    // nearest even: add one half less a bit, plus the last place, to the
    // remainder r : z, and its carry to the significand
    const unsigned odd = m0 & 1u;
    const unsigned e = a.e + b.e + ((h & 0x100000u) - (1022u << 20));
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %2, %3;\n\t"
        "addc.cc.u32 t, %4, %5;\n\t"
        "addc.cc.u32 %0, %0, 0;\n\t"
        "addc.u32 %1, %1, %6;\n\t}"
        : "+r"(m0), "+r"(m1)
        : "r"(z), "r"(odd - 1u), "r"(r), "r"(odd + 0x7fffffffu), "r"(e));
    return __hiloint2double((int)m1, (int)m0);
}

// a product in the FP64 multiplier, out of line: inlined beside the integer form
// it would issue there predicated off
static __device__ __noinline__ double dmul_fp64(double a, double b) { return a * b; }

__device__ __forceinline__ unsigned dmag_hi(double a) { return (unsigned)__double2hiint(a) & 0x7fffffffu; }

// a b where the caller knows that both and the product are normal
__device__ __forceinline__ double dmul_normal(double a, double b) {
    const double p = dmul_int(DFactor(a), DFactor(b));
    return __hiloint2double(__double2hiint(p) | ((__double2hiint(a) ^ __double2hiint(b)) & (int)0x80000000),
                            __double2loint(p));
}

// 2^-510 <= |a| < 2^510: products of two such are normal (zero, subnormals,
// infinities and NaN are outside)
__device__ __forceinline__ bool dmid(double a) { return dmag_hi(a) - (513u << 20) < (1020u << 20); }

// the exponent field of |a| less 767: below 2^9 << 20 for 2^-256 <= |a| < 2^256;
// the form for several factors, whose results are joined by |
__device__ __forceinline__ unsigned dwindow(double a) { return dmag_hi(a) - (767u << 20); }
constexpr unsigned kInWindow = 512u << 20;

// a b for any a and b: in the FP64 multiplier unless both are normal and the
// exponents' sum leaves the product normal with a place to spare
__device__ __forceinline__ double dmul_any(double a, double b) {
    const unsigned u = dmag_hi(a), v = dmag_hi(b);
    const bool fits = u - (1u << 20) < (2046u << 20) && v - (1u << 20) < (2046u << 20) &&
                      u + v - (1026u << 20) < (2040u << 20);
    return fits ? dmul_normal(a, b) : dmul_fp64(a, b);
}

// the same out of line, for the many products that appear once (inlined, the 70
// of a face and a cell overrun the instruction cache: 100 x 70 x 50 WENO-JS
// step 8.8 against 8.2 ms)
static __device__ __noinline__ double dmul_call(double a, double b) { return dmul_any(a, b); }

// Reciprocal of a positive finite double by Newton-Raphson iteration on
// f(r) = 1/r - y (r' = r + r (1 - y r), quadratic convergence), started from
// the hardware's approximate reciprocal (PTX rcp.approx.ftz.f64); two
// iterations reach the rounding limit.  The FP64 sweep is bound by the FP64
// pipe, and this takes fewer of its instructions than the IEEE division.
// Only for y > 0 finite and normal (the callers guard zero; a reciprocal below
// the normal range is flushed to zero).
__device__ __forceinline__ double drcp_newton(double y) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(y));
    double e = fma(-y, r, 1.0);
    r = fma(r, e, r);
    e = fma(-y, r, 1.0);
    return fma(r, e, r);
}

// 1 / sqrt(x) of a positive finite double: the hardware's approximation y0
// (PTX rsqrt.approx.ftz.f64) and one third-order step, y = y0 + y0 e (1/2 +
// 3 e / 8) with e = 1 - x y0^2 (the series of (1 - e)^(-1/2); the next term,
// 5 e^3 / 16, is below 2^-60).  5 FP64 instructions.  The callers take
// square roots as x / sqrt(x) and reciprocals as (1 / sqrt(x))^2 from the
// same value: CUDA's sqrt and a Newton reciprocal of the same x take 13.
__device__ __forceinline__ double drsqrt_newton(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-dmul_any(x, y), y, 1.0);
    return fma(fma(0.375, e, 0.5), dmul_any(y, e), y);
}

// a / b, b > 0 finite and normal: the approximate quotient q0 = a r0 (r0
// PTX rcp.approx.ftz.f64, e = 1 - b r0) times 1 + e + e^2 (next term below
// 2^-57): 4 FP64 instructions, one fewer than a drcp_newton(b).
__device__ __forceinline__ double ddiv_newton(double a, double b) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    const double e = fma(-b, r, 1.0);
    const double q = dmul_any(a, r);
    return fma(fma(e, e, e), q, q);
}

// 1 / b, b > 0 finite and normal, the same way: 3 FP64 instructions
__device__ __forceinline__ double drcp_third(double b) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    const double e = fma(-b, r, 1.0);
    return fma(fma(e, e, e), r, r);
}

// 2^n x by an addition to the exponent field (binary64: bits 52-62) on the
// integer pipes, |n| <= 4; exact for 2^-1018 <= |x| < 2^1018, x itself
// otherwise (zero, infinities and NaN keep their value; magnitudes outside
// that range do not occur in a physical state).
template <int N>
__device__ __forceinline__ double dscale2(double x) {
    const int hi = __double2hiint(x);
    const unsigned e = (unsigned)hi & 0x7ff00000u;
    const bool in = e - 0x00500000u < 0x7f400000u;
    return __hiloint2double(in ? hi + N * 0x00100000 : hi, __double2loint(x));
}

// the larger of two non-negative doubles: they order like their bit
// patterns, and an integer comparison leaves the FP64 pipe free (a NaN is
// the larger one and is kept)
__device__ __forceinline__ double dmax_nonneg(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// the same with a NaN b left out (fmax of non-negative doubles)
__device__ __forceinline__ double dmax_number(double a, double b) {
    const long long v = __double_as_longlong(b);
    return v > __double_as_longlong(a) && v <= 0x7ff0000000000000LL ? b : a;
}

template <> struct M<double> {
    static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
    static __device__ __forceinline__ double mul_(double a, double b) { return a * b; }
    static __device__ __forceinline__ double div_(double a, double b) { return ddiv_newton(a, b); }
    static __device__ __forceinline__ double rcp_(double x) { return drcp_newton(x); }
    static __device__ __forceinline__ double rcp3_(double x) { return drcp_third(x); }
    static __device__ __forceinline__ double times4_(double x) { return dscale2<2>(x); }
    static __device__ __forceinline__ double rsqrt_(double x) { return drsqrt_newton(x); }
    static __device__ __forceinline__ double abs_(double x) { return fabs(x); }
    static __device__ __forceinline__ double max_(double a, double b) { return fmax(a, b); }
    static __device__ __forceinline__ double max_nonneg(double a, double b) { return dmax_nonneg(a, b); }
    static __device__ __forceinline__ double min_(double a, double b) { return fmin(a, b); }
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
    static __device__ __forceinline__ double half_(double x) { return dscale2<-1>(x); }
    static __device__ __forceinline__ double sixteenth_(double x) { return dscale2<-4>(x); }
    // comparisons on the bit patterns (order preserving for a positive right
    // side; a comparison of doubles would issue on the FP64 pipe)
    static __device__ __forceinline__ bool ge_pos(double x, double c) { return __double_as_longlong(x) >= __double_as_longlong(c); }
    static __device__ __forceinline__ bool gt_pos(double x, double c) { return __double_as_longlong(x) > __double_as_longlong(c); }
    static __device__ __forceinline__ bool nonneg(double x) { return __double2hiint(x) >= 0; }
    static __device__ __forceinline__ bool normal_pos(double x) { return __double2hiint(x) >= 0x00200000; }
    static __device__ __forceinline__ bool finite_pos(double x) {   // 0 < x < 1e308; false for NaN
        return __double_as_longlong(x) > 0 && __double_as_longlong(x) < __double_as_longlong(1.0e308);
    }
};
template <> struct M<float> {
    static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
    static __device__ __forceinline__ float mul_(float a, float b) { return a * b; }
    static __device__ __forceinline__ float div_(float a, float b) { return __fdividef(a, b); }
    static __device__ __forceinline__ float rcp_(float x) { return __fdividef(1.0f, x); }
    static __device__ __forceinline__ float rcp3_(float x) { return __fdividef(1.0f, x); }
    static __device__ __forceinline__ float times4_(float x) { return 4.0f * x; }
    static __device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
    static __device__ __forceinline__ float abs_(float x) { return fabsf(x); }
    static __device__ __forceinline__ float max_(float a, float b) { return fmaxf(a, b); }
    static __device__ __forceinline__ float max_nonneg(float a, float b) { return fmaxf(a, b); }
    static __device__ __forceinline__ float min_(float a, float b) { return fminf(a, b); }
    static __device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ float half_(float x) { return 0.5f * x; }
    static __device__ __forceinline__ float sixteenth_(float x) { return 0.0625f * x; }
    static __device__ __forceinline__ bool ge_pos(float x, float c) { return x >= c; }
    static __device__ __forceinline__ bool gt_pos(float x, float c) { return x > c; }
    static __device__ __forceinline__ bool nonneg(float x) { return x >= 0.0f; }
    static __device__ __forceinline__ bool normal_pos(float x) { return !(x < 1.17549435e-38f); }
    static __device__ __forceinline__ bool finite_pos(float x) { return x > 0.0f && x < 3.0e38f; }
};

// The sweeps' choice for the products that appear once (MM of cell_fill and
// face_flux): MCalled takes them through dmul_call.  Same bits; faster in the
// three-in-one launch (256^3 WENO-Z step 342.6 -> 330.6 ms), slower where
// another pipe or the tile's tail is the bound (128^3 step with double-word
// weights 32.7 -> 34.2 ms; 48 patches 47.5 -> 48.6; adjoint 58.3 -> 58.8).
struct MCalled : M<double> {
    static __device__ __forceinline__ double mul_(double a, double b) { return dmul_call(a, b); }
};

// ---------------------------------------------------------------- wave speeds
// The discriminant d = aa^2 + 4 c_s^2 b_t^2 (aa = c_A^2 + b_t^2 - c_s^2) of the
// fast and slow speeds is a square of squared speeds: speeds below 3e-10 in
// float (1e-77 in double) take it below the normal range, where its root
// c_f^2 - c_slow^2 still has all its digits.  Below disc_normal, where either
// square may have lost some of them (2^28, 2^61 times the smallest normal
// number: a flushed c_s^2 b_t^2 is then below rounding), it is formed from aa and
// 2 c_s b_t times 2^100 (2^900).  sd = sqrt(d), isd = 1 / sd, small = c_s^2 b_t^2 / big
// with big = (sd + |aa|) / 2; all 0 where sd itself is below the normal range.
__device__ __forceinline__ bool disc_normal(float dd) { return !(dd < 0x1p-98f); }
__device__ __forceinline__ bool disc_normal(double dd) { return __double2hiint(dd) >= 63 << 20; }   // 2^-960
template <typename Real>
struct Disc {
    Real sd, isd, small;
};
template <typename Real>
__device__ __forceinline__ Disc<Real> disc_scaled(Real aa, Real cs2, Real bt2) {
    using m = M<Real>;
    constexpr Real S = std::is_same<Real, float>::value ? Real(0x1p100) : Real(0x1p900);
    constexpr Real iS = std::is_same<Real, float>::value ? Real(0x1p-100) : Real(0x1p-900);
    const Real cs = m::normal_pos(cs2) ? cs2 * m::rsqrt_(cs2) : Real(0);
    const Real bt = m::normal_pos(bt2) ? bt2 * m::rsqrt_(bt2) : Real(0);
    const Real a = aa * S, h = (cs * bt) * S;
    const Real dd = m::fma_(a, a, Real(4) * (h * h));
    if (!m::normal_pos(dd)) return {Real(0), Real(0), Real(0)};
    const Real isd = m::rsqrt_(dd), sd = dd * isd;
    if (!m::normal_pos(sd * iS)) return {Real(0), Real(0), Real(0)};
    return {sd * iS, isd * S, m::div_(h * iS, m::half_(sd + m::abs_(a))) * h};
}
// (double: out of line, so that its rare instructions do not issue, predicated
// off, on the FP64 pipe)
static __device__ __noinline__ double3 disc_scaled_call(double aa, double cs2, double bt2) {
    const Disc<double> d = disc_scaled<double>(aa, cs2, bt2);
    return make_double3(d.sd, d.isd, d.small);
}
__device__ __forceinline__ Disc<float> disc_small(float aa, float cs2, float bt2) { return disc_scaled<float>(aa, cs2, bt2); }
__device__ __forceinline__ Disc<double> disc_small(double aa, double cs2, double bt2) {
    const double3 d = disc_scaled_call(aa, cs2, bt2);
    return {d.x, d.y, d.z};
}

// c_f^2 - c_s^2 (fmc), c_s^2 - c_slow^2 (cms) without cancellation, and c_f^2.
// The larger of the two differences is (sd + |aa|) / 2 (aa = c_A^2 + b_t^2 -
// c_s^2), the other c_s^2 b_t^2 over it; the discriminant is the same one as
// (c_s^2 - c_A^2)^2 + b_t^2 (b_t^2 + 2 c_A^2 + 2 c_s^2), written as
// aa^2 + 4 c_s^2 b_t^2: still a sum of non-negative terms, so nothing cancels.
template <typename Real>
__device__ __forceinline__ void speeds_fast(Real cs2, Real ca2, Real bt2, Real &fmc, Real &cms, Real &cf2) {
    using m = M<Real>;
    const Real q = cs2 * bt2;
    const Real aa = ca2 + bt2 - cs2;
    const Real dd = m::fma_(aa, aa, Real(4) * q);
    if (disc_normal(dd)) {
        const Real sd = dd * m::rsqrt_(dd);
        const Real big = m::half_(sd + m::abs_(aa));
        // a branch, not a select: the callers that use only fmc skip the division
        // where it is the larger one
        if (m::nonneg(aa)) {
            fmc = big;
            cms = m::normal_pos(big) ? m::div_(q, big) : Real(0);
        } else {
            cms = big;
            fmc = m::normal_pos(big) ? m::div_(q, big) : Real(0);
        }
    } else {
        const Disc<Real> d = disc_small(aa, cs2, bt2);
        const Real big = m::half_(d.sd + m::abs_(aa));
        fmc = m::nonneg(aa) ? big : d.small;
        cms = m::nonneg(aa) ? d.small : big;
    }
    cf2 = cs2 + fmc;
}

// ---------------------------------------------------------------- one cell
// Fills the NCQ per-cell quantities of a cell from its state in the sweep
// frame (n, t1, t2): momentum (mn, m1, m2), cell field (Bn, B1, B2), into the
// box (box_at).
template <typename Real, bool PAIRED = false, typename MM = M<Real>>
__device__ __forceinline__ void cell_fill_frame(Real *box, int cell, int stride, Real rho, Real mn, Real m1, Real m2, Real E,
                                                Real Bn, Real B1, Real B2, const Phys<Real> &K, bool &bad, bool &hit) {
    using m = MM;
    Real r = rho;
    if (K.floors && r < K.rho_min) { r = K.rho_min; hit = true; }
    const Real isr = m::rsqrt_(r), ir = m::mul_(isr, isr);
    const Real vn = m::mul_(mn, ir), v1 = m::mul_(m1, ir), v2 = m::mul_(m2, ir);
    const Real vv = m::fma_(v2, v2, m::fma_(v1, v1, m::mul_(vn, vn)));
    const Real Bn2 = m::mul_(Bn, Bn), Bt2 = m::fma_(B2, B2, m::mul_(B1, B1));
    const Real BB = Bn2 + Bt2;
    Real P = K.gm1 * m::fma_(Real(-0.5), m::fma_(r, vv, BB), E);
    if (K.floors && P < K.p_min) { P = K.p_min; hit = true; }
    if (!(r > Real(0)) || !m::finite_pos(P)) bad = true;
    const Real Pt = m::fma_(Real(0.5), BB, P);
    const Real vB = m::fma_(v2, B2, m::fma_(v1, B1, m::mul_(vn, Bn)));
    box[box_at<PAIRED>(C_RHO, stride, cell)] = r;
    box[box_at<PAIRED>(C_VN, stride, cell)] = vn;
    box[box_at<PAIRED>(C_VT1, stride, cell)] = v1;
    box[box_at<PAIRED>(C_VT2, stride, cell)] = v2;
    box[box_at<PAIRED>(C_BN, stride, cell)] = Bn;
    box[box_at<PAIRED>(C_BT1, stride, cell)] = B1;
    box[box_at<PAIRED>(C_BT2, stride, cell)] = B2;
    box[box_at<PAIRED>(C_P, stride, cell)] = P;
    box[box_at<PAIRED>(C_RHOQ, stride, cell)] = rho;
    box[box_at<PAIRED>(C_MN, stride, cell)] = mn;
    box[box_at<PAIRED>(C_MT1, stride, cell)] = m1;
    box[box_at<PAIRED>(C_MT2, stride, cell)] = m2;
    box[box_at<PAIRED>(C_E, stride, cell)] = E;
    // rho v_n = m_n (v = m / rho with the same, possibly floored, rho)
    box[box_at<PAIRED>(C_F0, stride, cell)] = mn;
    box[box_at<PAIRED>(C_F1, stride, cell)] = m::fma_(mn, vn, Pt - Bn2);
    box[box_at<PAIRED>(C_F2, stride, cell)] = m::fma_(mn, v1, -m::mul_(Bn, B1));
    box[box_at<PAIRED>(C_F3, stride, cell)] = m::fma_(mn, v2, -m::mul_(Bn, B2));
    box[box_at<PAIRED>(C_F4, stride, cell)] = m::fma_(B1, vn, -m::mul_(Bn, v1));
    box[box_at<PAIRED>(C_F5, stride, cell)] = m::fma_(B2, vn, -m::mul_(Bn, v2));
    box[box_at<PAIRED>(C_F6, stride, cell)] = m::fma_(E + Pt, vn, -m::mul_(Bn, vB));
    // c_f, c_A and c_slow = c_s c_A / c_f, from reciprocal square roots
    const Real cs2 = m::mul_(m::mul_(K.gamma, P), ir);
    Real fmc, cms, cf2;
    speeds_fast<Real>(cs2, m::mul_(Bn2, ir), m::mul_(Bt2, ir), fmc, cms, cf2);
    const Real icf = m::rsqrt_(cf2);
    const Real ca = m::mul_(m::abs_(Bn), isr);
    box[box_at<PAIRED>(C_CF, stride, cell)] = m::mul_(cf2, icf);
    box[box_at<PAIRED>(C_CA, stride, cell)] = ca;
    box[box_at<PAIRED>(C_CSL, stride, cell)] = m::mul_(m::mul_(cs2, m::rsqrt_(cs2)), m::mul_(ca, icf));
}

// cell_fill_frame for a sweep along axis AX (frame (n, t1, t2) = (AX, AX+1,
// AX+2) mod 3) from the lab components
template <typename Real, int AX, bool PAIRED = false, typename MM = M<Real>>
__device__ __forceinline__ void cell_fill(Real *box, int cell, int stride, Real rho, Real mx, Real my, Real mz, Real E,
                                          Real Bx, Real By, Real Bz, const Phys<Real> &K, bool &bad, bool &hit) {
    constexpr int n = AX, t1 = (AX + 1) % 3, t2 = (AX + 2) % 3;
    const Real mm[3] = {mx, my, mz};
    const Real BB3[3] = {Bx, By, Bz};
    cell_fill_frame<Real, PAIRED, MM>(box, cell, stride, rho, mm[n], mm[t1], mm[t2], E, BB3[n], BB3[t1], BB3[t2], K, bad, hit);
}

// the same with the axis known only at run time (selects, no indexed arrays)
template <typename Real>
__device__ __forceinline__ void cell_fill_axis(Real *sm, int stride, Real rho, Real mx, Real my, Real mz, Real E,
                                               Real Bx, Real By, Real Bz, int ax, const Phys<Real> &K, bool &bad,
                                               bool &hit) {
    const Real mn = ax == 0 ? mx : (ax == 1 ? my : mz);
    const Real m1 = ax == 0 ? my : (ax == 1 ? mz : mx);
    const Real m2 = ax == 0 ? mz : (ax == 1 ? mx : my);
    const Real Bn = ax == 0 ? Bx : (ax == 1 ? By : Bz);
    const Real B1 = ax == 0 ? By : (ax == 1 ? Bz : Bx);
    const Real B2 = ax == 0 ? Bz : (ax == 1 ? Bx : By);
    cell_fill_frame<Real>(sm, 0, stride, rho, mn, m1, m2, E, Bn, B1, B2, K, bad, hit);
}

// The difference pass of a sweep's cell box, in two steps around a barrier
// (du overwrites u in place): box_diff_load reads the flux and conserved
// 7-vectors of cell i and of its successor i + st along the sweep axis and
// forms their differences; box_diff_store writes them.  sm points at the
// box, `stride` elements between quantities.
template <typename Real>
struct CellDiff {
    Real dF[7], dU[7];
};

template <typename Real>
__device__ __forceinline__ void box_diff_load(const Real *sm, int stride, int i, int st, CellDiff<Real> &d) {
    const Real *a = sm + i, *b = sm + i + st;
#pragma unroll
    for (int c = 0; c < 7; ++c) d.dF[c] = b[(C_F0 + c) * stride] - a[(C_F0 + c) * stride];
    constexpr int qU[7] = {C_RHOQ, C_MN, C_MT1, C_MT2, C_BT1, C_BT2, C_E};
#pragma unroll
    for (int c = 0; c < 7; ++c) d.dU[c] = b[qU[c] * stride] - a[qU[c] * stride];
}

template <typename Real>
__device__ __forceinline__ void box_diff_store(Real *sm, int stride, int i, const CellDiff<Real> &d) {
    Real *a = sm + i;
#pragma unroll
    for (int c = 0; c < 7; ++c) a[(C_DF0 + c) * stride] = d.dF[c];
    constexpr int qD[7] = {C_RHOQ, C_MN, C_MT1, C_MT2, C_DU4, C_DU5, C_E};
#pragma unroll
    for (int c = 0; c < 7; ++c) a[qD[c] * stride] = d.dU[c];
}

// ---------------------------------------------------------------- WENO
// phi_N(a, b, c, d) of Sec. 2.2 with JS (VAR = 0) or WENO-Z (VAR = 1)
// weights, in the form the kernels evaluate.
//
// Two rewrites that leave phi_N unchanged up to rounding:
// * the weights depend only on the ratios of eps + IS_k (JS: alpha_k =
//   d_k / (eps + IS_k)^2 normalised; WENO-Z: tau_5 / (eps + IS_k)), so the
//   smoothness indicators are evaluated as IS_k / 12 with eps / 12 (the
//   caller passes it);
// * with w_k = a_k / D (D = a_0 + a_1 + a_2) and the second differences
//   t1 = a - 2b + c = x0 - y0, t2 = b - 2c + d = y0 - z0 of the first ones
//   (x0 = a - b, y0 = b - c, z0 = c - d, also those of the indicators),
//   phi_N = w_0 t1 / 3 + (w_2 - 1/2) t2 / 6
//         = [4 a_0 t1 + (2 a_2 - D) t2] / (12 D);
//   in double each interpolant returns that numerator and D, and weno_field
//   divides once for the two; in float the weights are normalised first
//   (D = 1) and phi_N = Nn / 3.
//
// smoothness3 returns s_k = (eps + IS_k) / 12 and the first differences x0,
// y0, z0.  With a = b + x0, b = c + y0, d = c - z0 the three indicators are
// quadratics in one difference and b or c,
//   IS_0 / 12 = x0 (4 x0 / 3 - b) + b^2,  IS_1 / 12 = y0 (4 y0 / 3 - b) + b^2,
//   IS_2 / 12 = z0 (4 z0 / 3 + c) + c^2,
// positive definite (the minimum over the difference is 13/16 of the square),
// so nothing cancels: 11 operations with the differences, where 13 x^2 / 3 +
// y^2 each takes 15.  eps12 = eps / 12 of the caller's epsilon.
template <typename Real>
__device__ __forceinline__ void smoothness3(Real a, Real b, Real c, Real d, Real eps12, Real &s0, Real &s1, Real &s2,
                                            Real &x0, Real &y0, Real &z0) {
    using m = M<Real>;
    const Real k = Real(4.0 / 3.0);
    x0 = a - b;
    y0 = b - c;
    z0 = c - d;
    const Real bb = m::fma_(b, b, eps12), cc = m::fma_(c, c, eps12);
    s0 = m::fma_(x0, m::fma_(k, x0, -b), bb);
    s1 = m::fma_(y0, m::fma_(k, y0, -b), bb);
    s2 = m::fma_(z0, m::fma_(k, z0, c), cc);
}

// float: phi_N = Nn / 3 with the weights normalised here by one reciprocal
// (the WENO-Z ratio tau_5 / (eps + IS_k) is clamped at 1e18, so nothing
// overflows; unnormalised WENO-Z weights reach 1e36 in float)
template <int VAR>
__device__ __forceinline__ float phi_nf(float a, float b, float c, float d, float eps12) {
    float s0, s1, s2, x0, y0, z0;
    smoothness3<float>(a, b, c, d, eps12, s0, s1, s2, x0, y0, z0);
    float e0, e1, e2;   // alpha_k / d_k
    if constexpr (VAR == 0) {
        e0 = __fdividef(1.0f, s0 * s0);
        e1 = __fdividef(1.0f, s1 * s1);
        e2 = __fdividef(1.0f, s2 * s2);
    } else {
        const float tau = fabsf(s0 - s2);   // |IS_0 - IS_2| / 12
        const float r0 = fminf(tau * __fdividef(1.0f, s0), 1.0e18f);
        const float r1 = fminf(tau * __fdividef(1.0f, s1), 1.0e18f);
        const float r2 = fminf(tau * __fdividef(1.0f, s2), 1.0e18f);
        e0 = __fmaf_rn(r0, r0, 1.0f);
        e1 = __fmaf_rn(r1, r1, 1.0f);
        e2 = __fmaf_rn(r2, r2, 1.0f);
    }
    // D = e0 + 6 e1 + 3 e2; a_2 / 2 = 1.5 e2
    const float inv = __fdividef(1.0f, __fmaf_rn(3.0f, e2, __fmaf_rn(6.0f, e1, e0)));
    return __fmaf_rn(e0 * inv, x0 - y0, __fmaf_rn(e2, 1.5f * inv, -0.25f) * (y0 - z0));
}

// double: the weights times the common factor (s_0 s_1 s_2)^2, so that no
// weight needs a division; phi_N = N / (12 D), and the two interpolants of
// one field share a single division in weno_field.
//
// W0, V1, V2 are the alpha_k / d_k times that factor: weights_mul in the FP64
// multiplier, weno_weights with the products on the integer pipes.  The
// latter's range is checked once for all products: 2^-160 <= s_k < 2^96 by the
// exponent fields, and (WENO-Z) tau != 0, so |tau| >= 2^-213.  The largest and
// smallest are then q^2 in 2^-960 .. 2^576 and tau p_0 >= 2^-533.
template <int VAR>
static __device__ __noinline__ double3 weights_mul(double s0, double s1, double s2) {
    const double p0 = s1 * s2;
    if constexpr (VAR == 0) {
        // alpha_k / d_k = 1 / s_k^2
        const double p1 = s0 * s2, p2 = s0 * s1;
        return make_double3(p0 * p0, p1 * p1, p2 * p2);
    } else {
        // alpha_k / d_k = 1 + tau^2 / s_k^2: (s0 s1 s2)^2 + (tau prod_{j != k} s_j)^2,
        // tau = (IS_0 - IS_2) / 12 (its sign drops out)
        const double tau = s0 - s2;
        const double q = s0 * p0, t0 = tau * s0;
        const double A = tau * p0, B = t0 * s2, C = t0 * s1;
        const double Q = q * q;
        return make_double3(fma(A, A, Q), fma(B, B, Q), fma(C, C, Q));
    }
}

template <int VAR>
__device__ __forceinline__ void weno_weights(double s0, double s1, double s2, double &W0, double &V1, double &V2) {
    const unsigned c = 863u << 20;
    const unsigned out = ((unsigned)__double2hiint(s0) - c) | ((unsigned)__double2hiint(s1) - c) |
                         ((unsigned)__double2hiint(s2) - c);
    if (out < (256u << 20) && (VAR == 0 || __double_as_longlong(s0) != __double_as_longlong(s2))) {
        const DFactor f0(s0), f1(s1), f2(s2);
        const DFactor p0(dmul_int(f1, f2));
        if constexpr (VAR == 0) {
            const DFactor p1(dmul_int(f0, f2)), p2(dmul_int(f0, f1));
            W0 = dmul_int(p0, p0);
            V1 = dmul_int(p1, p1);
            V2 = dmul_int(p2, p2);
        } else {
            const DFactor ft(s0 - s2), q(dmul_int(f0, p0)), t0(dmul_int(ft, f0));
            const double A = dmul_int(ft, p0), B = dmul_int(t0, f2), C = dmul_int(t0, f1);
            const double Q = dmul_int(q, q);
            W0 = fma(A, A, Q);
            V1 = fma(B, B, Q);
            V2 = fma(C, C, Q);
        }
    } else {
        const double3 w = weights_mul<VAR>(s0, s1, s2);
        W0 = w.x;
        V1 = w.y;
        V2 = w.z;
    }
}

// The two interpolants of a field, phi_N(p_0 .. p_3) = Np / (12 Dp) and
// phi_N(q_3 .. q_0) = Nm / (12 Dm), with D = W0 + 6 V1 + 3 V2 and
// N = 4 W0 t1 + (6 V2 - D) t2
template <int VAR>
__device__ __forceinline__ void phi_nd(const double (&p)[4], const double (&q)[4], double eps12, double &Np, double &Dp,
                                       double &Nm, double &Dm) {
    double a0, a1, a2, ax, ay, az, b0, b1, b2, bx, by, bz;
    smoothness3<double>(p[0], p[1], p[2], p[3], eps12, a0, a1, a2, ax, ay, az);
    smoothness3<double>(q[3], q[2], q[1], q[0], eps12, b0, b1, b2, bx, by, bz);
    double A0, A1, A2, B0, B1, B2;
    weno_weights<VAR>(a0, a1, a2, A0, A1, A2);
    weno_weights<VAR>(b0, b1, b2, B0, B1, B2);
    const double YA = fma(6.0, A1, A0), YB = fma(6.0, B1, B0);
    Dp = fma(3.0, A2, YA);
    Dm = fma(3.0, B2, YB);
    const double vA = fma(3.0, A2, -YA), vB = fma(3.0, B2, -YB), tA = ay - az, tB = by - bz;
    double mA, mB;
    if (dmid(vA) && dmid(vB) && dmid(tA) && dmid(tB)) {
        mA = dmul_normal(vA, tA);
        mB = dmul_normal(vB, tB);
    } else {
        mA = dmul_fp64(vA, tA);
        mB = dmul_fp64(vB, tB);
    }
    Np = fma(A0, dscale2<2>(ax - ay), mA);
    Nm = fma(B0, dscale2<2>(bx - by), mB);
}

// N_m / D_m - N_p / D_p where the product of the denominators leaves the
// range of one shared reciprocal (flat data: D ~ eps^6; huge data).  Not
// inlined: rare, and its IEEE divisions would be issued, predicated off, on
// the FP64 pipe of every field.
static __device__ __noinline__ double weno_quotients(double Np, double Dp, double Nm, double Dm) {
    return Nm / Dm - Np / Dp;
}

// ---------------------------------------------------------------- double-word
// A double-word number is the unevaluated sum hi + lo of two floats with
// |lo| <= ulp(hi) / 2: 48 significand bits (unit roundoff u^2, u = 2^-24)
// and float's exponent range.  Each operation is a short sequence of FP32
// operations built on the error-free transforms TwoSum (Knuth), Fast2Sum
// (Dekker; |a| >= |b|) and TwoProd (one FMA), as analysed by Joldes, Muller
// and Popescu, "Tight and rigorous error bounds for basic building blocks of
// double-word arithmetic", ACM TOMS 44(2), 2017.  The intrinsics keep every
// step a separately rounded operation (no contraction into FMAs).
struct dw {
    float hi, lo;
};

__device__ __forceinline__ dw ef_fast2sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ dw ef_twosum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bv = __fsub_rn(s, a);
    const float av = __fsub_rn(s, bv);
    return {s, __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv))};
}
__device__ __forceinline__ dw ef_twoprod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
// x + y: TwoSum of the high parts, the low parts added to its error term,
// Fast2Sum (the "sloppy" sum of Joldes et al.).  The error is about
// 2 u^2 (|x| + |y|): relative to the result for operands of one sign, and
// relative to the operands where they cancel -- the accuracy the WENO
// differences need, whose double inputs enter with relative errors of
// 2^-49 from the conversion anyway.
__device__ __forceinline__ dw dw_add(dw x, dw y) {
    const dw s = ef_twosum(x.hi, y.hi);
    return ef_fast2sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ dw dw_neg(dw x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ dw dw_sub(dw x, dw y) { return dw_add(x, dw_neg(y)); }
// x * y with y a float, and with y a double-word
__device__ __forceinline__ dw dw_mul_f(dw x, float y) {
    const dw c = ef_twoprod(x.hi, y);
    return ef_fast2sum(c.hi, __fmaf_rn(x.lo, y, c.lo));
}
__device__ __forceinline__ dw dw_mul(dw x, dw y) {
    const dw c = ef_twoprod(x.hi, y.hi);
    const float t = __fmaf_rn(x.hi, y.lo, __fmul_rn(x.lo, y.hi));
    return ef_fast2sum(c.hi, __fadd_rn(c.lo, t));
}
// x / y: the float quotient q from a reciprocal refined by one Newton step,
// the residual x - y q in double-word, and its quotient as the correction
__device__ __forceinline__ dw dw_div(dw x, dw y) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y.hi));
    r = __fmaf_rn(r, __fmaf_rn(-y.hi, r, 1.0f), r);
    const float q = __fmul_rn(x.hi, r);
    const dw yq = dw_mul_f(y, q);
    const dw p = ef_twosum(x.hi, -yq.hi);
    const float d = __fadd_rn(p.hi, __fadd_rn(__fsub_rn(p.lo, yq.lo), x.lo));
    return ef_fast2sum(q, __fmul_rn(d, r));
}
__device__ __forceinline__ bool dw_eq(dw x, dw y) { return x.hi == y.hi && x.lo == y.lo; }

// A double as a double-word on the integer pipes (IEEE 754 binary64 layout:
// exponent bias 1023, 52 fraction bits): hi is x truncated to 24 significand
// bits, lo the remaining 29 bits rounded to 24, then renormalised (Fast2Sum).
// |x| below 2^-126 gives 0, |x| at or above 2^128 gives +-inf: neither
// occurs for the WENO inputs of a physical state, whose relative precision
// here is 2^-48.
__device__ __forceinline__ dw dw_from_double(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const unsigned hw = (unsigned)(u >> 32), lw = (unsigned)u;
    const unsigned sgn = hw & 0x80000000u;
    const int e = (int)((hw >> 20) & 0x7ffu);
    const unsigned hb = sgn | ((unsigned)(e - 896) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29);
    const float m = __uint2float_rn(lw & 0x1fffffffu);
    const float lo = __fmul_rn(m, __uint_as_float((unsigned)(e - 948) << 23));   // m 2^(e - 1075)
    float h = __uint_as_float(hb), l = __uint_as_float(__float_as_uint(lo) | sgn);
    if (e <= 948) l = 0.0f;
    if (e <= 896) h = 0.0f;
    if (e >= 1151) {
        h = __uint_as_float(sgn | 0x7f800000u);
        l = 0.0f;
    }
    return ef_fast2sum(h, l);
}

// A float as the double of equal value on the integer pipes (binary32:
// bias 127, 23 fraction bits); zeros and subnormals give 0, infinities and
// NaNs a NaN.
__device__ __forceinline__ double dw_f2d(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned ef = (b >> 23) & 0xffu;
    const unsigned hw = (b & 0x80000000u) | ((ef + 896u) << 20) | ((b & 0x7fffffu) >> 3);
    double d = __hiloint2double((int)hw, (int)(b << 29));
    if (ef == 0u) d = 0.0;
    if (ef == 0xffu) d = __longlong_as_double(0x7ff8000000000000LL);
    return d;
}

// phi_N (Sec. 2.2) of four double-word stencil differences (eps3 as in
// smoothness3), returned as 3 phi_N = (e_0 / D) t1 + (3 e_2 / (2 D) - 1/4) t2
// with e_k = alpha_k / d_k up to a common factor and D = e_0 + 6 e_1 + 3 e_2.
// The weights are formed relative to the smallest s_k (index m), so that no
// intermediate leaves float's range: with rho_k = s_m / s_k (rho_m = 1),
//   JS: alpha_k / d_k = 1 / s_k^2 = rho_k^2 / s_m^2, the common factor dropped;
//   Z:  alpha_k / d_k = 1 + (tau / s_k)^2 = 1 + (R rho_k)^2 with R = tau / s_m,
//       and, where R > 1e18, R^2 rho_k^2 (the 1 is below 1e-36 of the rest).
// Where eps / 3 is below float's range (WENO-Z) an indicator of a stencil
// without variation is 0; then rho_k = 0 for the others (their weights
// vanish against it, as in double), rho_k = 1 between equal indicators, and
// R = 0 where tau = 0.  An indicator below float's normal range (stencil
// differences under about 1e-19) counts as 0 as well: the reciprocal of a
// subnormal is not representable, and in double the weights of such
// stencils are set by rounding noise anyway.
template <int VAR>
__device__ __forceinline__ dw phi_dw(dw a, dw b, dw c, dw d, dw eps3) {
    const dw x0 = dw_sub(a, b), y0 = dw_sub(b, c), z0 = dw_sub(c, d);
    const dw x1 = dw_sub(x0, dw{2.0f * b.hi, 2.0f * b.lo});     // a - 3b
    const dw y1 = dw_add(b, c);
    const dw z1 = dw_add(z0, dw{2.0f * c.hi, 2.0f * c.lo});     // 3c - d
    const dw k = {4.33333349f, -1.58945719e-07f};              // 13/3
    auto normal_or_zero = [](dw s) { return s.hi < 1.17549435e-38f ? dw{0.0f, 0.0f} : s; };
    const dw s0 = normal_or_zero(dw_add(dw_add(dw_mul(k, dw_mul(x0, x0)), dw_mul(x1, x1)), eps3));
    const dw s1 = normal_or_zero(dw_add(dw_add(dw_mul(k, dw_mul(y0, y0)), dw_mul(y1, y1)), eps3));
    const dw s2 = normal_or_zero(dw_add(dw_add(dw_mul(k, dw_mul(z0, z0)), dw_mul(z1, z1)), eps3));
    dw sm = s0;
    if (s1.hi < sm.hi) sm = s1;
    if (s2.hi < sm.hi) sm = s2;
    const dw one = {1.0f, 0.0f};
    const dw r0 = dw_eq(s0, sm) ? one : dw_div(sm, s0);
    const dw r1 = dw_eq(s1, sm) ? one : dw_div(sm, s1);
    const dw r2 = dw_eq(s2, sm) ? one : dw_div(sm, s2);
    dw e0 = dw_mul(r0, r0), e1 = dw_mul(r1, r1), e2 = dw_mul(r2, r2);
    if constexpr (VAR == 1) {
        dw tau = dw_sub(s0, s2);
        if (tau.hi < 0.0f) tau = dw_neg(tau);
        const dw R = tau.hi == 0.0f ? dw{0.0f, 0.0f} : dw_div(tau, sm);
        if (R.hi <= 1.0e18f) {
            const dw R2 = dw_mul(R, R);
            e0 = dw_add(one, dw_mul(R2, e0));
            e1 = dw_add(one, dw_mul(R2, e1));
            e2 = dw_add(one, dw_mul(R2, e2));
        }
    }
    const dw D = dw_add(dw_add(e0, dw_mul_f(e1, 6.0f)), dw_mul_f(e2, 3.0f));
    const dw inv = dw_div(one, D);
    const dw w0 = dw_mul(e0, inv);
    const dw w2 = dw_add(dw_mul_f(dw_mul(e2, inv), 1.5f), dw{-0.25f, 0.0f});
    return dw_add(dw_mul(w0, dw_sub(x0, y0)), dw_mul(w2, dw_sub(y0, z0)));
}

// ---------------------------------------------------------------- pairs
// The stencil's flux difference and state difference at one position, (dF_j,
// du_j), share every projection coefficient, so they are carried as a pair.
// In float one packed two-lane FMA (sm_100 f32x2) acts on both; each lane
// rounds exactly as the scalar FMA would.
template <typename Real> struct Pair;
template <> struct Pair<float> { float2 v; };
template <> struct Pair<double> { double x, y; };

__device__ __forceinline__ Pair<float> make_pair2(float x, float y) { return {make_float2(x, y)}; }
__device__ __forceinline__ Pair<double> make_pair2(double x, double y) { return {x, y}; }
__device__ __forceinline__ Pair<float> pmul(float s, Pair<float> a) { return {__fmul2_rn(make_float2(s, s), a.v)}; }
__device__ __forceinline__ Pair<double> pmul(double s, Pair<double> a) { return {s * a.x, s * a.y}; }
__device__ __forceinline__ Pair<float> pfma(float s, Pair<float> a, Pair<float> c) {
    return {__ffma2_rn(make_float2(s, s), a.v, c.v)};
}
__device__ __forceinline__ Pair<double> pfma(double s, Pair<double> a, Pair<double> c) {
    return {fma(s, a.x, c.x), fma(s, a.y, c.y)};
}
// s a, s b, -s c and s a, t a: in double one range check for all their products
__device__ __forceinline__ void pmul3(float s, Pair<float> a, Pair<float> b, Pair<float> c, Pair<float> &x,
                                      Pair<float> &y, Pair<float> &z) {
    x = pmul(s, a);
    y = pmul(s, b);
    z = pmul(-s, c);
}
__device__ __forceinline__ void pmul2(float s, float t, Pair<float> a, Pair<float> &x, Pair<float> &y) {
    x = pmul(s, a);
    y = pmul(t, a);
}
__device__ __forceinline__ void pmul3(double s, Pair<double> a, Pair<double> b, Pair<double> c, Pair<double> &x,
                                      Pair<double> &y, Pair<double> &z) {
    const unsigned w = dwindow(s) | dwindow(a.x) | dwindow(a.y) | dwindow(b.x) | dwindow(b.y) | dwindow(c.x) | dwindow(c.y);
    if (w < kInWindow) {
        x = {dmul_normal(s, a.x), dmul_normal(s, a.y)};
        y = {dmul_normal(s, b.x), dmul_normal(s, b.y)};
        z = {dmul_normal(-s, c.x), dmul_normal(-s, c.y)};
    } else {
        x = {dmul_fp64(s, a.x), dmul_fp64(s, a.y)};
        y = {dmul_fp64(s, b.x), dmul_fp64(s, b.y)};
        z = {dmul_fp64(-s, c.x), dmul_fp64(-s, c.y)};
    }
}
__device__ __forceinline__ void pmul2(double s, double t, Pair<double> a, Pair<double> &x, Pair<double> &y) {
    if ((dwindow(s) | dwindow(t) | dwindow(a.x) | dwindow(a.y)) < kInWindow) {
        x = {dmul_normal(s, a.x), dmul_normal(s, a.y)};
        y = {dmul_normal(t, a.x), dmul_normal(t, a.y)};
    } else {
        x = {dmul_fp64(s, a.x), dmul_fp64(s, a.y)};
        y = {dmul_fp64(t, a.x), dmul_fp64(t, a.y)};
    }
}
// dF + alpha du and dF - alpha du
__device__ __forceinline__ float psplit(Pair<float> a, float al) { return __fmaf_rn(al, a.v.y, a.v.x); }
__device__ __forceinline__ double psplit(Pair<double> a, double al) { return fma(al, a.y, a.x); }

// The two members u = c + s, l = c - s of a mode pair, c the sign-free part
// of the projection and s = c1 a + c2 b.  In double u is one chain on c and
// l = 2 c - u (one instruction fewer than s, c + s, c - s); in float l is a
// chain of its own (a packed negation of u would cost what it saves).
__device__ __forceinline__ void mode_pair(Pair<double> c, double c1, Pair<double> a, double c2, Pair<double> b,
                                          Pair<double> &u, Pair<double> &l) {
    u = pfma(c1, a, pfma(c2, b, c));
    l = {fma(2.0, c.x, -u.x), fma(2.0, c.y, -u.y)};
}
__device__ __forceinline__ void mode_pair(Pair<float> c, float c1, Pair<float> a, float c2, Pair<float> b,
                                          Pair<float> &u, Pair<float> &l) {
    u = pfma(c1, a, pfma(c2, b, c));
    l = pfma(-c1, a, pfma(-c2, b, c));
}

// The WENO part of Eq. (FWENO) for one characteristic field: its flux is
// L.central + kWenoScale weno_field(...), from the five pairs L.(dF_j, du_j) at
// i-3/2 .. i+5/2.
//
// The split differences are (dF +- alpha dq)/2.  IS_k scales with the square
// of its arguments and phi_N linearly, so phi_N(x/2; eps) = phi_N(x; 4 eps)/2
// for both weight variants: the factor 1/2 is applied once to the result.
// With the IS_k / 12 form above the epsilon passed in is eps3 = 4 eps / 12.
// float: -N_p + N_m with phi_N = N / 3, times 1/6; double: phi_N = N / (12 D),
// times 1/24.
//
// DWW (double only): the split differences, formed in double, go to
// double-word, phi_dw evaluates both interpolants there, and their
// difference returns to double.
template <typename Real>
constexpr Real kWenoScale = std::is_same<Real, double>::value ? Real(1.0 / 24.0) : Real(1.0 / 6.0);

template <typename Real, int VAR, bool DWW = false>
__device__ __forceinline__ Real weno_field(const Pair<Real> (&P)[5], Real alpha, Real eps3) {
    Real p[4], q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        p[j] = psplit(P[j], alpha);
        q[j] = psplit(P[j + 1], -alpha);
    }
    if constexpr (std::is_same<Real, double>::value && DWW) {
        dw pd[4], qd[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            pd[j] = dw_from_double(p[j]);
            qd[j] = dw_from_double(q[j]);
        }
        const dw e3 = dw_from_double(4.0 * eps3);
        const dw Np = phi_dw<VAR>(pd[0], pd[1], pd[2], pd[3], e3);
        const dw Nm = phi_dw<VAR>(qd[3], qd[2], qd[1], qd[0], e3);
        const dw r = dw_sub(Nm, Np);
        return dw_f2d(4.0f * r.hi) + dw_f2d(4.0f * r.lo);
    }
    if constexpr (std::is_same<Real, double>::value) {
        double Np, Dp, Nm, Dm;
        phi_nd<VAR>(p, q, eps3, Np, Dp, Nm, Dm);
        double prod, cross;
        if (dmid(Dp) && dmid(Dm) && dmid(Np)) {
            prod = dmul_normal(Dp, Dm);
            cross = dmul_normal(Np, Dm);
        } else {
            prod = dmul_fp64(Dp, Dm);
            cross = dmul_fp64(Np, Dm);
        }
        // 2^-962 <= prod < 2^962 by its exponent field (positive, or NaN: outside)
        if ((unsigned)__double2hiint(prod) - 0x03d00000u < 0x78400000u)
            // -Np/Dp + Nm/Dm over the common denominator: one division
            return ddiv_newton(fma(Nm, Dp, -cross), prod);
        return weno_quotients(Np, Dp, Nm, Dm);
    } else {
        static_assert(std::is_same<Real, float>::value, "weno_field takes float or double");
        const float Np = phi_nf<VAR>(p[0], p[1], p[2], p[3], eps3);
        const float Nm = phi_nf<VAR>(q[3], q[2], q[1], q[0], eps3);
        return Nm - Np;
    }
}

// ---------------------------------------------------------------- one face

// The scalars of Appendix A's eigenvectors at an interface state (the mean
// of the two cells' primitives), from reciprocal square roots: 1 / sqrt(rho),
// 1 / c_s, 1 / sqrt(d) (d the discriminant of the speeds, whose root is
// c_f^2 - c_slow^2), 1 / |B_t|, 1 / c_f and one for the larger of (a_f, a_s).
// With big = (sqrt(d) + |aa|) / 2 (aa = c_A^2 + b_t^2 - c_s^2) the larger of
// a_f, a_s is sqrt(big / sqrt(d)) in [1/sqrt2, 1], and their product c_s b_t /
// sqrt(d) gives the smaller one without a second root or a division.
template <typename Real>
struct FaceEigen {
    Real sr, isr, cs, cs2, cf, cf2, csl, csl2, ics2, af, as, b1, b2, bt, sg;
    bool apart;   // c_f > c_slow: a_f, a_s as above (else both 1, Appendix A)
};

template <typename Real, typename MM = M<Real>>
__device__ __forceinline__ FaceEigen<Real> face_eigen(Real r, Real v2, Real Bn, Real Bt1, Real Bt2, Real P,
                                                      const Phys<Real> &K) {
    using m = MM;
    FaceEigen<Real> e;
    e.isr = m::rsqrt_(r);
    const Real ir = m::mul_(e.isr, e.isr);
    e.sr = m::mul_(r, e.isr);
    const Real ca2 = m::mul_(m::mul_(Bn, Bn), ir);
    const Real btm = m::fma_(Bt2, Bt2, m::mul_(Bt1, Bt1));
    const Real bt2 = m::mul_(btm, ir);
    // The slow and fast left eigenvectors carry 1/(2 c_s^2): the projection
    // amplifies the rounding of the data by about (v^2 + c_A^2 + b_t^2)/c_s^2.
    // In float, near a pressure floor, that reaches 1e9 and the split fluxes
    // drown in rounding, so the eigenvectors (never the LF speeds) take c_s^2
    // no smaller than cs2_rel times that sum.  L and R stay exact inverses, so
    // the flux stays consistent and conservative; only the basis in which
    // WENO reconstructs changes.  cs2_rel = 0 in double.
    e.cs2 = m::mul_(m::mul_(K.gamma, P), ir);
    if constexpr (float_based<Real>) e.cs2 = m::max_(e.cs2, K.cs2_rel * (v2 + ca2 + bt2));
    const Real ics = m::rsqrt_(e.cs2);
    e.cs = m::mul_(e.cs2, ics);
    e.ics2 = m::mul_(ics, ics);
    const Real q = m::mul_(e.cs2, bt2);
    const Real aa = ca2 + bt2 - e.cs2;
    const Real dd = m::fma_(aa, aa, Real(4) * q);
    Real sd, isd;
    bool some = true;
    if (disc_normal(dd)) {
        isd = m::rsqrt_(dd);
        sd = m::mul_(dd, isd);
    } else {
        const Disc<Real> d = disc_small(aa, e.cs2, bt2);
        sd = d.sd;
        isd = d.isd;
        some = m::normal_pos(sd);
    }
    const Real big = m::half_(sd + m::abs_(aa));
    const Real ibt = m::normal_pos(btm) ? m::rsqrt_(btm) : Real(0);
    const Real bta = m::mul_(btm, ibt);   // |B_t|
    const Real wb = m::mul_(big, isd);
    const Real iwb = m::rsqrt_(wb);
    const Real small_a = some ? m::mul_(m::mul_(e.cs, m::mul_(bta, e.isr)), m::mul_(isd, iwb)) : Real(0);
    e.apart = some && m::ge_pos(sd, K.eps_b2);
    const Real ab = e.apart ? m::mul_(wb, iwb) : Real(1), al = e.apart ? small_a : Real(1);
    const bool fast_big = m::nonneg(aa);
    e.as = fast_big ? ab : al;
    e.af = fast_big ? al : ab;
    // c_f^2 = c_s^2 + (c_f^2 - c_s^2), the difference a_s^2 sqrt(d)
    e.cf2 = e.cs2 + (fast_big ? big : m::mul_(m::mul_(small_a, small_a), sd));
    const Real icf = m::rsqrt_(e.cf2);
    e.cf = m::mul_(e.cf2, icf);
    // c_slow = c_s c_A / c_f (c_slow^2 = c_s^2 c_A^2 / c_f^2), c_A = |B_n| / sqrt(rho)
    e.csl = m::mul_(m::mul_(e.cs, m::mul_(m::abs_(Bn), e.isr)), icf);
    e.csl2 = m::mul_(e.csl, e.csl);
    if (m::gt_pos(btm, K.eps_b)) {   // b = B_t / |B_t|
        e.b1 = Bt1 * ibt;
        e.b2 = Bt2 * ibt;
        e.bt = bta;
    } else {
        e.b1 = Real(0.70710678118654752440);
        e.b2 = Real(0.70710678118654752440);
        e.bt = Real(0);
    }
    e.sg = m::ge_pos(Bn, K.eps_b) ? Real(1) : Real(-1);
    return e;
}

// Characteristic WENO flux at the face between stencil cells 2 and 3 of the
// six cells cell + k*st (k = 0..5) of the box, whose planes are `ncell`
// elements apart (box_at).  Ff receives the frame flux (rho, m_n, m_t1, m_t2, B_t1, B_t2, E) and
// s1, s2 the CT transport fluxes F_{B_t} + <B_n v_t> of Eqs. (fct1)-(fct6).
//
// The left and right eigenvectors of Appendix A are inverses (sum_m R_m L_m =
// identity on the 7-vector), so the central part of Eq. (FWENO) needs no
// projection: sum_m R_m (L_m . central + phi_m) = central + sum_m R_m phi_m.  Only
// the five pairs of stencil differences are projected, and the flux keeps
// the unprojected central combination (whose rounding no longer passes
// through 1 / c_s^2).  The exception is Appendix A's fallback a_f = a_s = 1 at
// c_f = c_slow, where L and R are not inverses: there the central part goes
// through both, as printed.
//
// Bound: the FP64 pipe in double (2 lanes per SM and clock: one instruction
// of a warp takes 16 clocks, in which 64 others can issue, hence the
// comparisons, halvings and maxima on the integer pipes), the issue slots in
// float.  Against the form that projected eleven vectors on Appendix A's rows
// in the lab frame: 535.0 -> 416.7 ms per 256^3 FP64 step (WENO-Z), 15.57 ->
// 14.46 ms in FP32-bulk, 56.6 -> 49.3 ms per 128^3 step with double-word
// weights; no larger error against 64-bit values in any of them.  With the tiles
// of today and the products on the integer pipes: 330 ms, FP64 pipe 88% busy on
// 861 FP64 instructions per interface with its share of the cells (128^3
// WENO-Z), issue slots 25%; FP32-bulk 13.2 ms, issue slots 74-76%.
template <typename Real, int VAR, bool DIFF = false, bool DWW = false, bool PAIRED = false, typename MM = M<Real>>
__device__ __forceinline__ void face_flux(const Real *__restrict__ box, int cell, int ncell, int st, const Phys<Real> &K,
                                          Real (&Ff)[7], Real &s1, Real &s2) {
    using m = MM;
    using P2 = Pair<Real>;
#define SMQ(q, k) box[box_at<PAIRED>(q, ncell, cell + (k) * st)]
    // stencil differences X[c][j] = (dF_c, du_c) at position j, and the
    // central combination (7 (f2 + f3) - (f1 + f4)) / 12 written as
    // f2 + (6 dF(2) + dF(1) - dF(3)) / 12
    [[maybe_unused]] P2 X[7][5];
    Real X0[7];
#pragma unroll
    for (int c = 0; c < 7; ++c) {
        if constexpr (DIFF) {
            // from the box's forward differences (its difference pass)
            const int qD = C_DF0 + c;
            X0[c] = m::fma_(m::fma_(Real(6), SMQ(qD, 2), SMQ(qD, 1)) - SMQ(qD, 3), Real(1.0 / 12.0), SMQ(C_F0 + c, 2));
        } else if constexpr (PAIRED) {
            float2 f[6];
#pragma unroll
            for (int j = 0; j < 6; ++j)
                f[j] = *reinterpret_cast<const float2 *>(box + box_at<true>(C_F0 + c, ncell, cell + j * st));
#pragma unroll
            for (int j = 0; j < 5; ++j) X[c][j] = {__ffma2_rn(make_float2(-1.0f, -1.0f), f[j], f[j + 1])};
            X0[c] = m::fma_(m::fma_(Real(6), X[c][2].v.x, X[c][1].v.x) - X[c][3].v.x, Real(1.0 / 12.0), f[2].x);
        } else {
            const int qF = C_F0 + c;
            const int qU = c == 0 ? C_RHOQ : c == 1 ? C_MN : c == 2 ? C_MT1 : c == 3 ? C_MT2 : c == 4 ? C_BT1
                           : c == 5 ? C_BT2 : C_E;
            Real f[6], u[6];
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                f[j] = SMQ(qF, j);
                u[j] = SMQ(qU, j);
            }
#pragma unroll
            for (int j = 0; j < 5; ++j) X[c][j] = make_pair2(f[j + 1] - f[j], u[j + 1] - u[j]);
            X0[c] = m::fma_(m::fma_(Real(6), f[3] - f[2], f[2] - f[1]) - (f[4] - f[3]), Real(1.0 / 12.0), f[2]);
        }
    }
    // interface state: mean of the primitives of cells i and i+1
    auto mean = [&](int q) { return m::half_(SMQ(q, 2) + SMQ(q, 3)); };
    const Real r = mean(C_RHO), vn = mean(C_VN), vt1 = mean(C_VT1), vt2 = mean(C_VT2);
    const Real Bn = mean(C_BN), Bt1 = mean(C_BT1), Bt2 = mean(C_BT2), P = mean(C_P);
    // Lax-Friedrichs speeds alpha(m) from the cell eigenvalues
    const Real vL = SMQ(C_VN, 2), vR = SMQ(C_VN, 3);
    auto alpha = [&](Real cL, Real cR) { return m::max_nonneg(m::abs_(vL + cL), m::abs_(vR + cR)); };
    const Real cfL = SMQ(C_CF, 2), cfR = SMQ(C_CF, 3);
    const Real caL = SMQ(C_CA, 2), caR = SMQ(C_CA, 3);
    const Real csL = SMQ(C_CSL, 2), csR = SMQ(C_CSL, 3);
    // twice the transport fluxes <B_n v_t> of the two cells
    const Real bvt1 = m::fma_(SMQ(C_BN, 2), SMQ(C_VT1, 2), SMQ(C_BN, 3) * SMQ(C_VT1, 3));
    const Real bvt2 = m::fma_(SMQ(C_BN, 2), SMQ(C_VT2, 2), SMQ(C_BN, 3) * SMQ(C_VT2, 3));

    // ---- eigen scalars at the interface state (Appendix A)
    const Real v2 = m::fma_(vt2, vt2, m::fma_(vt1, vt1, vn * vn));
    const Real hv2 = m::half_(v2);
    const FaceEigen<Real> e = face_eigen<Real, MM>(r, v2, Bn, Bt1, Bt2, P, K);
    const Real b1 = e.b1, b2 = e.b2, sg = e.sg;
    const Real pre = m::half_(e.ics2);
    const Real tau = K.gm1 * e.ics2;
    const Real afcf = e.af * e.cf, ascl = e.as * e.csl;
    const Real sas = sg * ascl, saf = sg * afcf;
    const Real eps3 = Real(1.0 / 3.0) * K.eps_w;   // 4 eps / 12: see weno_field

    // ---- projections.  With Y = X_m - v X_rho (the momentum differences in
    // the frame of the interface) the left eigenvectors of Appendix A are
    // combinations of
    //   g = X_E - v^2/2 X_rho - v.Y - |B_t| h,   h = b.X_B,   k = b.Y_t,
    //   L_fast    = pre ((gamma - 1) a_f g + sqrt(rho) c_s a_s h -+ a_f c_f Y_n +- sg a_s c_slow k),
    //   L_slow    = pre ((gamma - 1) a_s g - sqrt(rho) c_s a_f h -+ a_s c_slow Y_n -+ sg a_f c_f k),
    //   L_Alfven  = sg/2 (b x Y_t -+ ... ) = sg/2 [b_1 Y_t2 - b_2 Y_t1 +- sg sqrt(rho) (b_1 X_B2 - b_2 X_B1)],
    //   L_entropy = X_rho - (gamma - 1) g / c_s^2.
    // (g's field part -B_t is taken as -|B_t| b.  Where |B_t|^2 <= eps_B the
    // default b is not B_t / |B_t|; there |B_t| is taken as 0, which leaves out
    // at most |B_t| |X_B| <= 1e-15 |X_B|.)  The Alfven fields are carried
    // without their factor sg/2: phi_N is linear up to epsilon, which scales
    // by 4 with them, and the factor joins the back-projection.
    P2 F[7][5];
    const Real cF = pre * (K.gm1 * e.af), cS = pre * (K.gm1 * e.as);
    const Real srcs = pre * (e.sr * e.cs);
    const Real hF = srcs * e.as, hS = -(srcs * e.af);
    const Real nF = -(pre * afcf), nS = -(pre * ascl), kF = pre * sas, kS = -(pre * saf);
    const Real ssr = sg * e.sr;
    const Real a5 = ssr * b1, a4 = -(ssr * b2);
    // The seven fields at one position of the stencil: the fast, slow and
    // Alfven pairs (members u, l), entropy
    auto project = [&](const P2 (&x7)[7], P2 (&f)[7]) {
        const P2 Yn = pfma(-vn, x7[0], x7[1]);
        const P2 Y1 = pfma(-vt1, x7[0], x7[2]);
        const P2 Y2 = pfma(-vt2, x7[0], x7[3]);
        P2 mh, mk, mx, mF, mS;
        pmul3(b2, x7[5], Y2, Y1, mh, mk, mx);
        const P2 h = pfma(b1, x7[4], mh);
        const P2 k = pfma(b1, Y1, mk);
        const P2 x = pfma(b1, Y2, mx);
        pmul2(hF, hS, h, mF, mS);
        P2 g = pfma(-hv2, x7[0], x7[6]);
        g = pfma(-vn, Yn, g);
        g = pfma(-vt1, Y1, g);
        g = pfma(-vt2, Y2, g);
        g = pfma(-e.bt, h, g);
        mode_pair(pfma(cF, g, mF), nF, Yn, kF, k, f[0], f[1]);
        mode_pair(pfma(cS, g, mS), nS, Yn, kS, k, f[2], f[3]);
        mode_pair(x, a4, x7[4], a5, x7[5], f[4], f[5]);
        f[6] = pfma(-tau, g, x7[0]);
    };
    // ---- WENO parts of the fields: sums and differences of the pairs, upper
    // members m = 1 (v - c_f), 3 (v - c_slow), 2 (v - c_A)
    Real sf, df, ss, ds, sa, da, Fe;
    if constexpr (std::is_same<Real, float>::value) {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            P2 x7[7], f[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) x7[c] = X[c][j];
            project(x7, f);
#pragma unroll
            for (int mo = 0; mo < 7; ++mo) F[mo][j] = f[mo];
        }
        auto fields = [&](const P2 (&u)[5], const P2 (&l)[5], Real cL, Real cR, Real ep, Real &sum, Real &dif) {
            const Real Fu = weno_field<Real, VAR>(u, alpha(-cL, -cR), ep);
            const Real Fl = weno_field<Real, VAR>(l, alpha(cL, cR), ep);
            sum = Fu + Fl;
            dif = Fu - Fl;
        };
        fields(F[0], F[1], cfL, cfR, eps3, sf, df);
        fields(F[2], F[3], csL, csR, eps3, ss, ds);
        fields(F[4], F[5], caL, caR, Real(4) * eps3, sa, da);
        Fe = weno_field<Real, VAR>(F[6], m::max_nonneg(m::abs_(vL), m::abs_(vR)), eps3);
    } else {
        // double: loops over the positions and over the fields, the projections
        // in local memory.  With integer products and double-word interpolants
        // the unrolled face function is 100 to 200 KB of code, which no
        // instruction cache of an SM holds, and the loops need no more than 168
        // registers, three blocks per SM without spills: 256^3 WENO-Z step 388
        // ms unrolled, 353 looped with the products of the projections and
        // quotients on the integer pipes (396 and more unrolled); 128^3 step
        // with double-word weights 49.0 -> 39.7 ms.
#pragma unroll 1
        for (int j = 0; j < 5; ++j) {
            P2 x7[7], f[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                const int qU = c == 0 ? C_RHOQ : c == 1 ? C_MN : c == 2 ? C_MT1 : c == 3 ? C_MT2
                               : c == 4 ? (DIFF ? (int)C_DU4 : (int)C_BT1) : c == 5 ? (DIFF ? (int)C_DU5 : (int)C_BT2) : C_E;
                if constexpr (DIFF)
                    x7[c] = make_pair2(SMQ(C_DF0 + c, j), SMQ(qU, j));
                else
                    x7[c] = make_pair2(SMQ(C_F0 + c, j + 1) - SMQ(C_F0 + c, j), SMQ(qU, j + 1) - SMQ(qU, j));
            }
            project(x7, f);
#pragma unroll
            for (int mo = 0; mo < 7; ++mo) F[mo][j] = f[mo];
        }
        Real V[7];
        const Real cL[7] = {-cfL, cfL, -csL, csL, -caL, caL, Real(0)}, cR[7] = {-cfR, cfR, -csR, csR, -caR, caR, Real(0)};
#pragma unroll 1
        for (int mo = 0; mo < 7; ++mo) {
            P2 f[5];
#pragma unroll
            for (int j = 0; j < 5; ++j) f[j] = F[mo][j];
            V[mo] = weno_field<Real, VAR, DWW>(f, alpha(cL[mo], cR[mo]), mo == 4 || mo == 5 ? Real(4) * eps3 : eps3);
        }
        sf = V[0] + V[1];
        df = V[0] - V[1];
        ss = V[2] + V[3];
        ds = V[2] - V[3];
        sa = V[4] + V[5];
        da = V[4] - V[5];
        Fe = V[6];
    }
#undef SMQ
    if (!e.apart) {
        // Appendix A's fallback: the central part through L and R, in the
        // units of the WENO parts, in place of the unprojected one
        const Real u = Real(1) / kWenoScale<Real>;
        const Real Yn = X0[1] - vn * X0[0], Y1 = X0[2] - vt1 * X0[0], Y2 = X0[3] - vt2 * X0[0];
        const Real h = b1 * X0[4] + b2 * X0[5], k = b1 * Y1 + b2 * Y2;
        const Real g = X0[6] - hv2 * X0[0] - vn * Yn - vt1 * Y1 - vt2 * Y2 - e.bt * h;
        const Real u2 = Real(2) * u;
        sf += u2 * (cF * g + hF * h);
        df += u2 * (nF * Yn + kF * k);
        ss += u2 * (cS * g + hS * h);
        ds += u2 * (nS * Yn + kS * k);
        sa += u2 * (b1 * Y2 - b2 * Y1);
        da += u2 * (a4 * X0[4] + a5 * X0[5]);
        Fe += u * (X0[0] - tau * g);
#pragma unroll
        for (int c = 0; c < 7; ++c) X0[c] = Real(0);
    }

    // ---- back-projection: central + sum over fields of (WENO part) x (right
    // eigenvector).  The right eigenvectors of the fast pair (Rc +- Rs), seen
    // from the frame of the interface (v = 0),
    //   Rc = (a_f, 0, c_s a_s b / sqrt(rho), a_f (c_f^2 - g2 c_s^2)),
    //   Rs = rows (1, 2, 3): (-a_f c_f, c_slow a_s b sg),
    // of the slow pair (a_f, c_f -> a_s, c_slow and a_s, c_slow -> -a_f, c_f
    // in Rc's field rows and Rs), of the Alfven pair and of the entropy field
    // (1, 0, 0, 0) combine into a few scalars; the boost back to the lab adds
    // v S1 to the momentum and v^2/2 S1 + v.T to the energy.
    {
        const Real kw = kWenoScale<Real>;
        const Real mg = m::fma_(e.af, sf, e.as * ss);              // magnetosonic density
        const Real S1 = mg + Fe;
        const Real S2 = (e.cs * e.isr) * m::fma_(e.as, sf, -(e.af * ss));
        const Real hsa = m::half_(sa), hda = m::half_(da) * (sg * e.isr);   // (sg/2)^2, sg/2 of the Alfven fields
        const Real Tn = -m::fma_(afcf, df, ascl * ds);
        const Real Tk = m::fma_(sas, df, -(saf * ds));
        const Real T1 = m::fma_(Tk, b1, -(hsa * b2));
        const Real T2 = m::fma_(Tk, b2, hsa * b1);
        const Real en6 = m::fma_(afcf * e.cf, sf, m::fma_(ascl * e.csl, ss, -((K.g2 * e.cs2) * mg)));
        Ff[0] = m::fma_(kw, S1, X0[0]);
        Ff[1] = m::fma_(kw, m::fma_(S1, vn, Tn), X0[1]);
        Ff[2] = m::fma_(kw, m::fma_(S1, vt1, T1), X0[2]);
        Ff[3] = m::fma_(kw, m::fma_(S1, vt2, T2), X0[3]);
        Ff[4] = m::fma_(kw, m::fma_(S2, b1, -(hda * b2)), X0[4]);
        Ff[5] = m::fma_(kw, m::fma_(S2, b2, hda * b1), X0[5]);
        Ff[6] = m::fma_(kw, m::fma_(hv2, S1, m::fma_(vn, Tn, m::fma_(vt1, T1, m::fma_(vt2, T2, en6)))), X0[6]);
    }
    s1 = m::fma_(Real(0.5), bvt1, Ff[4]);
    s2 = m::fma_(Real(0.5), bvt2, Ff[5]);
}

}  // namespace w5ct
