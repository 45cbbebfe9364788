// hgks_math.cuh -- device arithmetic of the hybrid WENO-AO gas-kinetic scheme
// (arXiv 2304.05572) for sm_103a, FP64.
//
// Two kinds of code live here:
//  * decision-carrying reconstruction (troubled-cell indicator, normal-direction
//    linear and characteristic WENO-AO reconstruction, positivity test).  Its
//    outputs feed later troubled-cell decisions, so it is evaluated in one fixed
//    IEEE order with no FMA contraction: every operation goes through the
//    `ex` wrapper, whose operators map to __dadd_rn / __dmul_rn / __ddiv_rn and
//    whose fma is explicit.  Any implementation that evaluates the same formulas
//    in the same order (as written below) takes bit-identical decisions.
//  * the Gauss-point (tangential) reconstruction and the gas-kinetic flux, which
//    only feed the update and are written for few FP64 instructions: closed-form
//    micro-slope solves, one erfc and one exp per side, exp(-dt/(2 tau)) squared
//    for exp(-dt/tau), and the S2O4 flux combinations formed on scalar
//    coefficients before the moment vectors are combined.
#pragma once

#include <cstdint>
#include <cmath>

#include "hgks_fluxconst.h"
#if defined(__CUDACC__)
#include "hgks_fixed.cuh"
#endif

// flux arithmetic is also compiled for the host (unit checks of the formulas)
#define HGKS_HD __host__ __device__

namespace hgks {

// ---------------------------------------------------------------- exact-order FP64
struct ex {
    double v;
    __device__ __forceinline__ ex() {}
    __device__ __forceinline__ ex(double x) : v(x) {}
};
__device__ __forceinline__ ex operator+(ex a, ex b) { return ex(__dadd_rn(a.v, b.v)); }
__device__ __forceinline__ ex operator-(ex a, ex b) { return ex(__dsub_rn(a.v, b.v)); }
__device__ __forceinline__ ex operator*(ex a, ex b) { return ex(__dmul_rn(a.v, b.v)); }
#if defined(__CUDACC__)
// IEEE quotients and roots in integers: the same bits, where the compiler's sequences take 10 to 15
// FP64 instructions; those remain for zeros, subnormals, infinities, NaNs and the ends of the range.
// WENO-AO everywhere on 500^2: normal passes 4.65 -> 3.85 ms per step; dt at 1024^2 97 -> 46 us.
__device__ __noinline__ double div_far(double a, double b) { return __ddiv_rn(a, b); }
__device__ __noinline__ double sqrt_far(double a) { return __dsqrt_rn(a); }
__device__ __forceinline__ ex operator/(ex a, ex b)
{
    double q;
    if (!fixed::div_rn(a.v, b.v, q)) q = div_far(a.v, b.v);
    return ex(q);
}
__device__ __forceinline__ ex xsqrt(ex a)
{
    double q;
    if (!fixed::sqrt_rn(a.v, q)) q = sqrt_far(a.v);
    return ex(q);
}
#else
__device__ __forceinline__ ex operator/(ex a, ex b) { return ex(__ddiv_rn(a.v, b.v)); }
__device__ __forceinline__ ex xsqrt(ex a) { return ex(__dsqrt_rn(a.v)); }
#endif
__device__ __forceinline__ ex operator-(ex a) { return ex(-a.v); }
__device__ __forceinline__ ex xfma(ex a, ex b, ex c) { return ex(__fma_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ ex xabs(ex a) { return ex(fabs(a.v)); }

// 1/x and 1/sqrt(x) in free-order arithmetic (the flux, the tangential WENO-AO pass), in fixed
// point on the device: no FP64 instruction where the hardware's approximation and two
// Newton-Raphson steps take 4 and 7 of the pipe's 64-cycle slots; within 1 ulp of the correctly
// rounded quotient and within 2 ulps of IEEE division by the IEEE square root (hgks_check_reciprocal).
// The host build divides.
HGKS_HD __forceinline__ double rcp_nr(double x)
{
#ifdef __CUDA_ARCH__
    return fixed::rcp(x);
#else
    return 1.0 / x;
#endif
}

HGKS_HD __forceinline__ double rsqrt_nr(double x)
{
#ifdef __CUDA_ARCH__
    return fixed::rsqrt(x);
#else
    return 1.0 / sqrt(x);
#endif
}

// x > 0, x = 0: integer tests on the device, where a comparison occupies the FP64 pipe too
HGKS_HD __forceinline__ bool positive(double x)
{
#ifdef __CUDA_ARCH__
    return fixed::is_pos(x);
#else
    return x > 0.0;
#endif
}

HGKS_HD __forceinline__ bool is_zero(double x)
{
#ifdef __CUDA_ARCH__
    return fixed::is_zero(x);
#else
    return x == 0.0;
#endif
}

// x 2^K; exp(-y), y >= 0
template <int K>
HGKS_HD __forceinline__ double scale2(double x)
{
#ifdef __CUDA_ARCH__
    return fixed::scale2<K>(x);
#else
    return x * (K > 0 ? (double)(1 << (K > 0 ? K : 0)) : 1.0 / (double)(1 << (K < 0 ? -K : 0)));
#endif
}

HGKS_HD __forceinline__ double exp_neg(double y)
{
#ifdef __CUDA_ARCH__
    const unsigned hi = (unsigned)__double2hiint(y);
    if (hi < 0x40862000u) return fixed::exp_value(fixed::exp_neg(y));       // y < 708
    return hi <= 0x7FF00000u ? 0.0 : y;     // below the normal range; NaN
#else
    return exp(-y);
#endif
}

// x 2^K with the bits of the FP64 multiplication.  INT: an integer add to the exponent (the multiplication
// itself where the result could leave the normal range): for kernels bound by the FP64 pipe.  A lane
// group's short dependent chain is no faster with it (128 against 125 us on the 512^2 step's normal
// passes) and multiplies.
template <int K, bool INT>
__device__ __forceinline__ ex xscale(ex x)
{
    constexpr double f = K > 0 ? (double)(1 << (K > 0 ? K : 0)) : 1.0 / (double)(1 << (K < 0 ? -K : 0));
#if defined(__CUDACC__)
    if constexpr (INT) {
        const unsigned e = (unsigned)(__double2hiint(x.v) >> 20) & 0x7FFu;
        return e - 8u < 2032u || fixed::is_zero(x.v) ? ex(fixed::scale2<K>(x.v)) : x * ex(f);
    }
#endif
    return x * ex(f);
}

// Troubled-cell indicator, Sec. 2.3.1 Steps 1-3, on the window q[0..4] = Q_{i-2..i+2}
// (cell units).  Step 1: |D| <= Z1 with D = (4Q_{i-2}+Q_{i-1}) + (4Q_{i+2}+Q_{i+1}) - 10 Q_i
// and Z1 = 17 zeta1 dx^2 (Eq. (24): abar2 = D/34).  Step 2: xbar = -abar1/(2 abar2) with
// abar1 = -N/10, N = (2Q_{i-2}+Q_{i-1}) - (2Q_{i+2}+Q_{i+1}); inside iff |xbar| <= 5/2.
// Step 3: xhat from the conservative 3-cell quadratic; non-troubled iff |xbar - xhat| <= 1/4.
__device__ __forceinline__ int indicator_exact(ex q0, ex q1, ex q2, ex q3, ex q4, double Z1)
{
    ex D = xfma(ex(-10.0), q2, xfma(ex(4.0), q0, q1) + xfma(ex(4.0), q4, q3));
    if (fabs(D.v) <= Z1) return 0;
    ex N = xfma(ex(2.0), q0, q1) - xfma(ex(2.0), q4, q3);
    ex a1 = -(N / ex(10.0));
    ex a2 = D / ex(34.0);
    ex xbar = (-a1) / (ex(2.0) * a2);
    if (!(fabs(xbar.v) <= 2.5)) return 0;
    ex ah1 = ex(0.5) * (q3 - q1);
    ex ah2 = ex(0.5) * ((q1 + q3) - ex(2.0) * q2);
    ex den = ex(2.0) * ah2 + ex(ah2.v == 0.0 ? 1e-30 : 0.0);
    ex xhat = (-ah1) / den;
    if (fabs((xbar - xhat).v) <= 0.25) return 0;
    return 1;
}

#if defined(__CUDACC__)
__device__ __noinline__ int indicator_exact_nl(ex q0, ex q1, ex q2, ex q3, ex q4, double Z1)
{
    return indicator_exact(q0, q1, q2, q3, q4, Z1);
}

// The same decision with few or no FP64 instructions (a comparison and a conversion occupy the FP64
// pipe as long as an addition), f[j] = q[j] truncated to FP32 (fixed::to_float).  Each test is first taken in
// FP32 with a margin above its rounding errors; only a test that falls inside its margin is decided by
// the exact chain.
//   Step 1: |D| against Z1 from the truncated window: truncation (2^-23) and four roundings (2^-24) of terms
//     |c| m with coefficients summing to 20, m = max |q|: error below 20 m (2^-23 + 4 2^-24) = 7.2e-6 m.  A
//     value below 2^-126 counts as 0, which adds up to 20 2^-126 = 2.4e-37: within the 1e-6 Z1 kept back
//     for Z1 above 1e-30, below which the test is not taken.
//   Steps 2, 3 on D, N, d = q3 - q1, s = (q1 + q3) - 2 q2, rounded as the exact chain rounds them (10 FP64
//     operations): xbar = 1.7 N/D and xhat = -d/(2 s) (s = 2 ah2, the halves are exact), their FP32 ratios
//     within 2^-20 relative; margins 1e-5.  Quantities outside 1e-30..1e30 go to the exact chain, and
//     s = 0 does unless d = 0, where xhat = 0.
// The exact chain takes 5 FP64 slots of the pipe on smooth data and, behind Step 1, four IEEE
// divisions more, where one troubled lane holds up its warp.  Raw flags per step at 1024^2: normal
// 253 -> 163 us, tangential 702 -> 220 us (with the shared row loads of b_raw_tflags).
// CALL: the exact chain behind a call, for b_tang_small, whose three uses would each hold a copy of it (the
// large sweeps' tangential flags unroll four and are 31 % slower behind a call: 220 -> 288 us at 1024^2).
template <bool CALL>
__device__ __forceinline__ int indicator_raw(const double* q, const float* f, double Z1)
{
    const float m = fmaxf(fmaxf(fmaxf(fabsf(f[0]), fabsf(f[1])), fmaxf(fabsf(f[3]), fabsf(f[4]))), fabsf(f[2]));
    const float Df = fmaf(-10.0f, f[2], fmaf(4.0f, f[0], f[1]) + fmaf(4.0f, f[4], f[3]));
    // (an infinity among the f makes the sum infinite or a NaN: the comparison fails)
    const float Zf = fixed::to_float(Z1);
    if (Zf > 1e-30f && fmaf(8.0e-6f, m, fabsf(Df)) < 0.999999f * Zf) return 0;
    const ex q0(q[0]), q1(q[1]), q2(q[2]), q3(q[3]), q4(q[4]);
    const ex D = xfma(ex(-10.0), q2, xfma(ex(4.0), q0, q1) + xfma(ex(4.0), q4, q3));
    if (fixed::abs_le(D.v, Z1)) return 0;
    const ex N = xfma(ex(2.0), q0, q1) - xfma(ex(2.0), q4, q3);
    const float Dt = fixed::to_float(D.v), Nt = 1.7f * fixed::to_float(N.v);
    const bool range = fabsf(Dt) > 1e-30f && fabsf(Dt) < 1e30f;
    if (range && fabsf(Nt) > 2.50003f * fabsf(Dt)) return 0;
    const ex d = q3 - q1, s = xfma(ex(-2.0), q2, q1 + q3);
    const float sf = fixed::to_float(s.v), df = fixed::to_float(d.v);
    const bool flat = fixed::is_zero(s.v) && fixed::is_zero(d.v);
    if (range && fabsf(Nt) < 2.49997f * fabsf(Dt) && (flat || (fabsf(sf) > 1e-30f && fabsf(sf) < 1e30f && fabsf(df) < 1e30f))) {
        const float xb = __fdividef(Nt, Dt);
        const float xh = flat ? 0.0f : __fdividef(-0.5f * df, sf);
        const float gap = fabsf(xb - xh), tol = 1e-5f * (1.0f + fabsf(xh));
        if (gap < 0.25f - tol) return 0;
        if (gap > 0.25f + tol) return 1;
    }
    return CALL ? indicator_exact_nl(q0, q1, q2, q3, q4, Z1) : indicator_exact(q0, q1, q2, q3, q4, Z1);
}
#endif

// Step 5, Eqs. (26)-(27): value and derivative at x_{i+1/2} from cell i's window.
__device__ __forceinline__ void linear_left(const double* q, double inv12h, double& val, double& der)
{
    ex t = xfma(ex(-13.0), ex(q[1]), ex(2.0) * ex(q[0]));
    t = xfma(ex(47.0), ex(q[2]), t);
    t = xfma(ex(27.0), ex(q[3]), t);
    t = xfma(ex(-3.0), ex(q[4]), t);
    val = (t * ex(1.0 / 60.0)).v;
    ex s = xfma(ex(-15.0), ex(q[2]), ex(q[1]));
    s = xfma(ex(15.0), ex(q[3]), s);
    s = s - ex(q[4]);
    der = (s * ex(inv12h)).v;
}

// Eqs. (28)-(29): value and derivative at x_{i-1/2}, the mirror image of linear_left.
__device__ __forceinline__ void linear_right(const double* q, double inv12h, double& val, double& der)
{
    ex t = xfma(ex(-13.0), ex(q[3]), ex(2.0) * ex(q[4]));
    t = xfma(ex(47.0), ex(q[2]), t);
    t = xfma(ex(27.0), ex(q[1]), t);
    t = xfma(ex(-3.0), ex(q[0]), t);
    val = (t * ex(1.0 / 60.0)).v;
    ex s = xfma(ex(-15.0), ex(q[2]), ex(q[3]));
    s = xfma(ex(15.0), ex(q[1]), s);
    s = s - ex(q[0]);
    der = (-(s * ex(inv12h))).v;
}

// WENO-AO constants: linear weights of Eq. (35) and derived ratios.
struct AOConst {
    double g[4];      // gamma_0..2 (sub-stencils, S1 central), gamma_3 (large stencil)
    double g3inv;     // 1/gamma_3
    double gr[3];     // gamma_k / gamma_3
    double eps;
};

// Smoothness indicators of Eq. (39) in cell units, in the evaluation order the decisions need
// (factors 2, 4, 1/2, 1/4, 1/16 are exact).
template <bool INT>
__device__ __forceinline__ void ao_betas(const ex* q, ex* b)
{
    const ex q1_2 = xscale<1, INT>(q[1]), q2_2 = xscale<1, INT>(q[2]), q3_2 = xscale<1, INT>(q[3]);
    const ex s0 = (q[0] - q1_2) + q[2], t0 = (q[0] - xscale<1, INT>(q1_2)) + ex(3.0) * q[2];
    const ex s1 = (q[1] - q2_2) + q[3], t1 = q[1] - q[3];
    const ex s2 = (q[2] - q3_2) + q[4], t2 = (ex(3.0) * q[2] - xscale<1, INT>(q3_2)) + q[4];
    b[0] = ex(13.0 / 12.0) * (s0 * s0) + xscale<-2, INT>(t0 * t0);
    b[1] = ex(13.0 / 12.0) * (s1 * s1) + xscale<-2, INT>(t1 * t1);
    b[2] = ex(13.0 / 12.0) * (s2 * s2) + xscale<-2, INT>(t2 * t2);
    const ex a13 = q[1] + q[3], a04 = q[0] + q[4];
    const ex c1 = ex(17.0 / 24.0) * (q[3] - q[1]) - ex(5.0 / 48.0) * (q[4] - q[0]);
    const ex c2 = ((ex(0.75) * a13 - xscale<-4, INT>(a04)) - ex(1.375) * q[2]);
    const ex c3 = ex(1.0 / 6.0) * t1 - ex(1.0 / 12.0) * (q[0] - q[4]);
    const ex c4 = ((ex(1.0 / 24.0) * a04 - ex(1.0 / 6.0) * a13) + xscale<-2, INT>(q[2]));
    b[3] = ((((c1 * c1 + xscale<-1, INT>(c1 * c3)) + ex(13.0 / 3.0) * (c2 * c2)) + ex(21.0 / 5.0) * (c2 * c4))
            + ex(3129.0 / 80.0) * (c3 * c3)) + ex(87617.0 / 140.0) * (c4 * c4);
}

// Normalised nonlinear weights, Eqs. (37), (38), (40), with the ratio delta/(beta_k + eps) squared.
template <bool INT>
__device__ __forceinline__ void ao_weights(const ex* q, const AOConst& k, ex* wb)
{
    ex b[4], w[4], r[4];
    ao_betas<INT>(q, b);
    const ex d = ((xabs(b[3] - b[0]) + xabs(b[3] - b[1])) + xabs(b[3] - b[2])) * ex(1.0 / 3.0);
#pragma unroll
    for (int j = 0; j < 4; j++) r[j] = d / (b[j] + ex(k.eps));
#pragma unroll
    for (int j = 0; j < 4; j++) w[j] = ex(k.g[j]) * (ex(1.0) + r[j] * r[j]);
    const ex inv = ex(1.0) / (((w[0] + w[1]) + w[2]) + w[3]);
#pragma unroll
    for (int j = 0; j < 4; j++) wb[j] = w[j] * inv;
}

// AO(5,3) polynomial of Eq. (41) applied to point values p[0..3].
__device__ __forceinline__ ex ao_combine(const ex* wb, const AOConst& k, const ex* p)
{
    return wb[3] * (p[3] * ex(k.g3inv) - ((ex(k.gr[0]) * p[0] + ex(k.gr[1]) * p[1]) + ex(k.gr[2]) * p[2]))
         + ((wb[0] * p[0] + wb[1] * p[1]) + wb[2] * p[2]);
}

// Face values / cell-unit derivatives of the three quadratics (Eqs. (32), (43), with the
// p_2(x_{i+1/2}) coefficient corrected to -1/6) and of the quartic (Eqs. (36), (44)).
template <bool INT>
__device__ __forceinline__ void face_polys(const ex* q, int side, ex* pv, ex* pd)
{
    if (side > 0) {
        pv[0] = ((xscale<1, INT>(q[0]) - ex(7.0) * q[1]) + ex(11.0) * q[2]) * ex(1.0 / 6.0);
        pv[1] = ((-q[1] + ex(5.0) * q[2]) + xscale<1, INT>(q[3])) * ex(1.0 / 6.0);
        pv[2] = ((xscale<1, INT>(q[2]) + ex(5.0) * q[3]) - q[4]) * ex(1.0 / 6.0);
        pv[3] = ((((xscale<1, INT>(q[0]) - ex(13.0) * q[1]) + ex(47.0) * q[2]) + ex(27.0) * q[3]) - ex(3.0) * q[4]) * ex(1.0 / 60.0);
        pd[0] = (q[0] - ex(3.0) * q[1]) + xscale<1, INT>(q[2]);
        pd[1] = q[3] - q[2];
        pd[2] = q[3] - q[2];
        pd[3] = (((q[1] - ex(15.0) * q[2]) + ex(15.0) * q[3]) - q[4]) * ex(1.0 / 12.0);
    } else {
        pv[0] = ((-q[0] + ex(5.0) * q[1]) + xscale<1, INT>(q[2])) * ex(1.0 / 6.0);
        pv[1] = ((xscale<1, INT>(q[1]) + ex(5.0) * q[2]) - q[3]) * ex(1.0 / 6.0);
        pv[2] = ((ex(11.0) * q[2] - ex(7.0) * q[3]) + xscale<1, INT>(q[4])) * ex(1.0 / 6.0);
        pv[3] = ((((-ex(3.0) * q[0] + ex(27.0) * q[1]) + ex(47.0) * q[2]) - ex(13.0) * q[3]) + xscale<1, INT>(q[4])) * ex(1.0 / 60.0);
        pd[0] = q[2] - q[1];
        pd[1] = q[2] - q[1];
        pd[2] = (-xscale<1, INT>(q[2]) + ex(3.0) * q[3]) - q[4];
        pd[3] = (((q[0] - ex(15.0) * q[1]) + ex(15.0) * q[2]) - q[3]) * ex(1.0 / 12.0);
    }
}

// Left (L = R^{-1}, rows) and right (R, columns) eigenvectors of dF/dQ (local normal direction) at Q, the
// entries that are not 0 or 1 by construction (2D: L[2] = (-V, 0, 1, 0), R's third column (0, 0, 1, V)):
// a factor 1 and a term 0 leave the other operands' bits as they are.
template <int NV, bool INT>
__device__ __forceinline__ void eigvec(double gam, const ex* Q, ex (*L)[NV], ex (*R)[NV])
{
    const ex gm1 = ex(gam) - ex(1.0);
    const ex rho = Q[0], ri = ex(1.0) / rho;
    const ex U = Q[1] * ri;
    ex V(0.0), q2 = U * U;
    if constexpr (NV == 4) { V = Q[2] * ri; q2 = q2 + V * V; }
    const ex p = gm1 * (Q[NV - 1] - xscale<-1, INT>(rho) * q2);
    const ex c2 = (ex(gam) * p) * ri, c = xsqrt(c2), ci = ex(1.0) / c;
    const ex H = (Q[NV - 1] + p) * ri;
    const ex b1 = gm1 / c2, b1h = xscale<-1, INT>(b1), b2 = b1h * q2, bU = b1 * U, uci = U * ci, uc = U * c;
    constexpr int E = NV - 1;
    R[0][0] = ex(1.0);   R[0][1] = ex(1.0);        R[0][E] = ex(1.0);
    R[1][0] = U - c;      R[1][1] = U;              R[1][E] = U + c;
    R[E][0] = H - uc;     R[E][1] = xscale<-1, INT>(q2); R[E][E] = H + uc;
    L[0][0] = xscale<-1, INT>(b2 + uci); L[0][1] = -xscale<-1, INT>(bU + ci); L[0][E] = b1h;
    L[1][0] = ex(1.0) - b2;         L[1][1] = bU;                    L[1][E] = -b1;
    L[E][0] = xscale<-1, INT>(b2 - uci); L[E][1] = -xscale<-1, INT>(bU - ci); L[E][E] = b1h;
    if constexpr (NV == 4) {
        const ex bV = b1 * V;
        R[0][2] = ex(0.0); R[1][2] = ex(0.0); R[2][0] = V; R[2][1] = V; R[2][2] = ex(1.0); R[2][3] = V; R[3][2] = V;
        L[0][2] = -xscale<-1, INT>(bV); L[1][2] = bV; L[3][2] = L[0][2];
        L[2][0] = -V; L[2][1] = ex(0.0); L[2][2] = ex(1.0); L[2][3] = ex(0.0);
    }
}

// y = L x and y = R x with the summation order ((m0 x0 + m1 x1) + m2 x2) + m3 x3.
template <int NV>
__device__ __forceinline__ void project(const ex (*L)[NV], const ex* x, ex* y)
{
#pragma unroll
    for (int r = 0; r < NV; r++) {
        if (NV == 4 && r == 2) { y[2] = L[2][0] * x[0] + x[2]; continue; }
        ex s = L[r][0] * x[0] + L[r][1] * x[1];
#pragma unroll
        for (int c = 2; c < NV; c++) s = s + L[r][c] * x[c];
        y[r] = s;
    }
}

template <int NV>
__device__ __forceinline__ void project_back(const ex (*R)[NV], const ex* x, ex* y)
{
    y[0] = (x[0] + x[1]) + x[NV - 1];
    y[1] = (R[1][0] * x[0] + R[1][1] * x[1]) + R[1][NV - 1] * x[NV - 1];
    ex s = R[NV - 1][0] * x[0] + R[NV - 1][1] * x[1];
    if constexpr (NV == 4) {
        y[2] = ((R[2][0] * x[0] + R[2][1] * x[1]) + x[2]) + R[2][3] * x[3];
        s = s + R[3][2] * x[2];
    }
    y[NV - 1] = s + R[NV - 1][NV - 1] * x[NV - 1];
}

// Characteristic WENO-AO at the face of side (+1: x_{i+1/2}, -1: x_{i-1/2}) of the cell whose
// window (cells i-2..i+2) is Qw[j][comp], projected with the eigenvectors at Qs in the local
// normal direction.  Returns conservative value and cell-unit derivative.
template <int NV>
__device__ __forceinline__ void weno_ao_face(double gam, const AOConst& k, const double (*Qw)[NV], const double* Qs,
                                             int side, double* val, double* der)
{
    ex L[NV][NV], R[NV][NV], Uc[5][NV], uv[NV], ud[NV], qs[NV];
#pragma unroll
    for (int c = 0; c < NV; c++) qs[c] = ex(Qs[c]);
    eigvec<NV, true>(gam, qs, L, R);
#pragma unroll
    for (int j = 0; j < 5; j++) {
        ex x[NV];
#pragma unroll
        for (int c = 0; c < NV; c++) x[c] = ex(Qw[j][c]);
        project<NV>(L, x, Uc[j]);
    }
#pragma unroll
    for (int c = 0; c < NV; c++) {
        ex q[5], wb[4], pv[4], pd[4];
#pragma unroll
        for (int j = 0; j < 5; j++) q[j] = Uc[j][c];
        ao_weights<true>(q, k, wb);
        face_polys<true>(q, side, pv, pd);
        uv[c] = ao_combine(wb, k, pv);
        ud[c] = ao_combine(wb, k, pd);
    }
    ex v[NV], d[NV];
    project_back<NV>(R, uv, v);
    project_back<NV>(R, ud, d);
#pragma unroll
    for (int c = 0; c < NV; c++) { val[c] = v[c].v; der[c] = d[c].v; }
}

#if defined(__CUDACC__)   // lane-group functions: device code only (the host count compiles the flux alone)
// Row r of M for a per-lane r, selected without indexing local memory.
template <int NV, typename T>
__device__ __forceinline__ void select_row(const T (*M)[NV], int r, T* row)
{
#pragma unroll
    for (int c = 0; c < NV; c++) {
        T v = M[0][c];
#pragma unroll
        for (int k = 1; k < NV; k++) v = r == k ? M[k][c] : v;
        row[c] = v;
    }
}

// The characteristic WENO-AO face reconstruction of weno_ao_face, spread over the 4 lanes of an
// aligned lane group (lane q = threadIdx.x & 3): lane q projects the window onto characteristic
// field q (row q of L), runs the nonlinear weights and the AO combination of that field alone,
// the 4 fields' results are exchanged with shuffles, and lane q projects back component q (row q
// of R); the components are exchanged again so that every lane returns the whole state val[]
// (for the positivity test) and its own component's derivative derq.  Every value is formed by
// the same operations in the same order as in weno_ao_face, so the results are bit-identical;
// the per-lane work, and so the latency of an item on the narrow FP64 pipe, is about a quarter.
// Lanes q >= NV (1D) duplicate field NV-1.  All 4 lanes of the group must call this together
// (mask gmask).
template <int NV>
__device__ __forceinline__ void weno_ao_face_x4(double gam, const AOConst& k, const double (*Qw)[NV], const double* Qs,
                                                int side, unsigned gmask, double* val, double& derq)
{
    const int q = threadIdx.x & 3;
    const int qc = q < NV ? q : NV - 1;
    const int lane0 = threadIdx.x & 28;
    ex L[NV][NV], R[NV][NV], qs[NV];
#pragma unroll
    for (int c = 0; c < NV; c++) qs[c] = ex(Qs[c]);
    eigvec<NV, false>(gam, qs, L, R);
    ex Lq[NV], Rq[NV];
    select_row<NV>(L, qc, Lq);
    select_row<NV>(R, qc, Rq);
    ex u[5], wb[4], pv[4], pd[4];
#pragma unroll
    for (int j = 0; j < 5; j++) {
        ex s = Lq[0] * ex(Qw[j][0]) + Lq[1] * ex(Qw[j][1]);
#pragma unroll
        for (int c = 2; c < NV; c++) s = s + Lq[c] * ex(Qw[j][c]);
        u[j] = s;
    }
    ao_weights<false>(u, k, wb);
    face_polys<false>(u, side, pv, pd);
    const double uvq = ao_combine(wb, k, pv).v, udq = ao_combine(wb, k, pd).v;
    ex uv[NV], ud[NV];
#pragma unroll
    for (int c = 0; c < NV; c++) {
        uv[c] = ex(__shfl_sync(gmask, uvq, lane0 + c));
        ud[c] = ex(__shfl_sync(gmask, udq, lane0 + c));
    }
    // row qc of R times uv and ud, in the summation order of project_back
    ex v = Rq[0] * uv[0] + Rq[1] * uv[1], d = Rq[0] * ud[0] + Rq[1] * ud[1];
#pragma unroll
    for (int c = 2; c < NV; c++) { v = v + Rq[c] * uv[c]; d = d + Rq[c] * ud[c]; }
#pragma unroll
    for (int c = 0; c < NV; c++) val[c] = __shfl_sync(gmask, v.v, lane0 + c);
    derq = d.v;
}
#endif

// Reading (no safeguard is printed): rho <= 0 or p <= 0 after reconstruction -> first order.
// For rho > 0 (and gamma > 1), p > 0 exactly when rho E - ke > 0, ke = 0.5 (m_x^2 + m_y^2);
// tested in that division-free form, in this order.
template <int NV>
__device__ __forceinline__ bool nonphysical_exact(const double* Q)
{
    ex ke;
    if constexpr (NV == 4) ke = ex(0.5) * (ex(Q[1]) * ex(Q[1]) + ex(Q[2]) * ex(Q[2]));
    else ke = ex(0.5) * (ex(Q[1]) * ex(Q[1]));
    ex pr = ex(Q[NV - 1]) * ex(Q[0]) - ke;
    return !(positive(Q[0]) && positive(pr.v));
}

// First in FP32 (fixed::surely_physical); only a state next to vacuum takes the exact test.
#if defined(__CUDACC__)
template <int NV>
__device__ __forceinline__ bool nonphysical(const double* Q)
{
    if (fixed::surely_physical(fixed::to_float(Q[0]), fixed::to_float(Q[1]), NV == 4 ? fixed::to_float(Q[2]) : 0.0f,
                        fixed::to_float(Q[NV - 1])))
        return false;
    return nonphysical_exact<NV>(Q);
}

// The same for a state spread over an aligned group of 4 lanes (lane q component q; mask gmask): the FP32 test
// converts one component a lane.
template <int NV>
__device__ __forceinline__ bool nonphysical_x4(double v, int lane0, unsigned gmask)
{
    const float f = fixed::to_float(v);
    const float rho = __shfl_sync(gmask, f, lane0), mx = __shfl_sync(gmask, f, lane0 + 1);
    const float my = NV == 4 ? __shfl_sync(gmask, f, lane0 + 2) : 0.0f, E = __shfl_sync(gmask, f, lane0 + NV - 1);
    if (fixed::surely_physical(rho, mx, my, E)) return false;             // the same for the 4 lanes
    double Q[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) Q[k] = __shfl_sync(gmask, v, lane0 + k);
    return nonphysical_exact<NV>(Q);
}
#endif

// ---------------------------------------------------------------- Gauss-point reconstruction
#if defined(__CUDACC__)
// Quartic of the window q at the two Gauss points: v[0] at -g, v[1] at +g, and (DER) its derivatives
// there times inv_ht (`inv` the same as a fixed-point factor).  In fixed point (fixed::quartic_pair); FP64
// for exponents outside its range, infinities and NaNs.
template <bool DER>
__device__ __forceinline__ void gauss_linear(const double* q, fixed::Scale inv, double inv_ht, double* v, double* d)
{
    if (fixed::quartic_pair<DER>(q, inv, v, d)) return;
    const double s1 = q[1] + q[3], s2 = q[0] + q[4], d1 = q[3] - q[1], d2 = q[4] - q[0];
    const double even = fma(719.0 / 720.0, q[2], fma(1.0 / 1080.0, s1, (-1.0 / 4320.0) * s2));
    const double odd = fma(0.20046884346862004, d1, -0.028065638085606807 * d2);      // 25 sqrt3/216, 7 sqrt3/432
    v[0] = even - odd; v[1] = even + odd;
    if (DER) {
        const double n = fma(2.0 / 3.0, d1, (-1.0 / 12.0) * d2);
        // 4 sqrt3/9, 13 sqrt3/54, sqrt3/54
        const double t = fma(-0.76980035891950105, q[2], fma(0.4169751944147297, s1, -0.032075014954979206 * s2));
        d[0] = (n - t) * inv_ht; d[1] = (n + t) * inv_ht;
    }
}
#endif

// The tangential WENO-AO pass (free-order arithmetic: the outputs only feed the flux).
//
// AO reconstruction of one characteristic field at the two Gauss points xi = -+g, g^2 = 1/12: v[0], v[1], and
// (der) its derivatives d[0], d[1] in cell units.  With t_k/2 the slope at the cell's centre and s_k the
// curvature of sub-stencil k (the terms its smoothness indicator is made of) and c1..c4 the quartic's
// coefficients, the polynomials' values there are
//     p_k = q2 +- g t_k/2,           p_k' = t_k/2 +- g s_k          (xi^2 - 1/12 vanishes),
//     p_3 = q2 - c4/180 +- g (c1 + c3/12),   p_3' = c1 + c3/4 +- 2 g (c2 + c4/6),
// so the combination of Eq. (41) takes two sums over the sub-stencils and the indicators' own terms: 27
// FP64 operations in place of 72 on the tabulated point values of each polynomial.  With the shared rows of
// the projections (tang_project, tang_back) WENO-AO everywhere on 500^2 went from 7.35 to 3.45 ms per
// step of tangential passes, the 1024^2 four-quadrant step's from 0.25 to 0.14 ms.
__device__ __forceinline__ void gauss_ao(const double* q, const AOConst& k, bool der, double* v, double* d)
{
    const double q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3], q4 = q[4];
    // smoothness indicators, Eq. (39), as ao_betas
    const double s0 = fma(-2.0, q1, q0) + q2, s1 = fma(-2.0, q2, q1) + q3, s2 = fma(-2.0, q3, q2) + q4;
    const double d13 = q3 - q1, d04 = q4 - q0, a13 = q1 + q3, a04 = q0 + q4;
    const double t0 = fma(3.0, q2, fma(-4.0, q1, q0)), t1 = d13, t2 = fma(-3.0, q2, fma(4.0, q3, -q4));
    const double c1 = fma(17.0 / 24.0, d13, (-5.0 / 48.0) * d04);
    const double c2 = fma(-1.375, q2, fma(0.75, a13, -0.0625 * a04));
    const double c3 = fma(-1.0 / 6.0, d13, (1.0 / 12.0) * d04);
    const double c4 = fma(0.25, q2, fma(-1.0 / 6.0, a13, (1.0 / 24.0) * a04));
    constexpr double b1312 = 13.0 / 12.0;
    const double b0 = fma(b1312 * s0, s0, (0.25 * t0) * t0);
    const double b1 = fma(b1312 * s1, s1, (0.25 * t1) * t1);
    const double b2 = fma(b1312 * s2, s2, (0.25 * t2) * t2);
    const double b3 = fma(c1, fma(0.5, c3, c1), fma(c2, fma(13.0 / 3.0, c2, 4.2 * c4),
                      fma((3129.0 / 80.0) * c3, c3, ((87617.0 / 140.0) * c4) * c4)));
    // nonlinear weights, Eqs. (37), (38), not yet normalised (the reciprocals take no FP64 operation)
    const double dl = ((fabs(b3 - b0) + fabs(b3 - b1)) + fabs(b3 - b2)) * (1.0 / 3.0);
    const double r0 = dl * rcp_nr(b0 + k.eps), r1 = dl * rcp_nr(b1 + k.eps), r2 = dl * rcp_nr(b2 + k.eps), r3 = dl * rcp_nr(b3 + k.eps);
    const double w0 = fma(k.g[0] * r0, r0, k.g[0]), w1 = fma(k.g[1] * r1, r1, k.g[1]);
    const double w2 = fma(k.g[2] * r2, r2, k.g[2]), w3 = fma(k.g[3] * r3, r3, k.g[3]);
    const double inv = rcp_nr((w0 + w1) + (w2 + w3));
    // weights of the polynomials in the combination: sub-stencil k: w_k - w3 g_k/g3; quartic: w3/g3
    const double m0 = fma(-w3, k.gr[0], w0), m1 = fma(-w3, k.gr[1], w1), m2 = fma(-w3, k.gr[2], w2);
    const double m3 = w3 * k.g3inv, m32 = scale2<1>(m3);
    const double B = fma(m0, t0, fma(m1, t1, m2 * t2));
    const double ev = (m3 * (-1.0 / 180.0)) * c4;
    const double od = 0.14433756729740644 * fma(m32, fma(1.0 / 12.0, c3, c1), B);          // g/2
    v[0] = fma(inv, ev - od, q2);
    v[1] = fma(inv, ev + od, q2);
    if (der) {
        const double C = fma(m0, s0, fma(m1, s1, m2 * s2));
        const double De = fma(m32, fma(0.25, c3, c1), B), Do = fma(m32, fma(1.0 / 6.0, c4, c2), C);
        const double ih = scale2<-1>(inv);
        d[0] = ih * fma(-0.57735026918962576, Do, De);                                     // 2g
        d[1] = ih * fma(0.57735026918962576, Do, De);
    } else {
        d[0] = d[1] = 0.0;
    }
}

// Eigenvectors of the flux Jacobian in the tangential direction at the face average Qs: the projections onto
// and from the fields in the few terms their rows share (L and R have zeros and repeated entries).
struct TangEig { double U, V, c, H, hq2, b1h, ci2; };

__device__ __forceinline__ void tang_eig(double gam, const double* Qs, TangEig& e)
{
    const double gm1 = gam - 1.0, ri = rcp_nr(Qs[0]);
    e.U = Qs[1] * ri;
    e.V = Qs[2] * ri;
    e.hq2 = scale2<-1>(fma(e.U, e.U, e.V * e.V));
    const double p = gm1 * fma(-Qs[0], e.hq2, Qs[3]);
    const double c2 = (gam * p) * ri, ci = rsqrt_nr(c2);
    e.c = c2 * ci;
    e.H = (Qs[3] + p) * ri;
    e.ci2 = scale2<-1>(ci);
    e.b1h = (scale2<-1>(gm1) * ci) * ci;
}

// Fields of one state x
__device__ __forceinline__ void tang_project(const TangEig& e, const double* x, double* f)
{
    const double w = e.b1h * fma(e.hq2, x[0], fma(-e.U, x[1], fma(-e.V, x[2], x[3])));
    const double z = e.ci2 * fma(e.V, x[0], -x[2]);
    f[0] = w + z;
    f[1] = fma(-2.0, w, x[0]);
    f[2] = fma(e.U, x[0], -x[1]);
    f[3] = w - z;
}

__device__ __forceinline__ void tang_back(const TangEig& e, const double* f, double* x)
{
    const double s = f[0] + f[3], cd = e.c * (f[3] - f[0]);
    x[0] = s + f[1];
    x[1] = fma(e.U, x[0], -f[2]);
    x[2] = fma(e.V, x[0], cd);
    x[3] = fma(e.H, s, fma(e.hq2, f[1], fma(-e.U, f[2], e.V * cd)));
}

// One pass (4 components, one lane) at the two Gauss points: projection of the 5 line values x[s][],
// gauss_ao per field, projection back.
__device__ __forceinline__ void tang_ao(const TangEig& e, const double (*x)[4], const AOConst& ak, bool der,
                                        double (*v)[2], double (*d)[2])
{
    // all projections first: the line values are dead before the four fields' weights are formed
    double uc[5][4];
#pragma unroll
    for (int s = 0; s < 5; s++) tang_project(e, x[s], uc[s]);
    double cv[2][4], cd[2][4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const double u[5] = {uc[0][c], uc[1][c], uc[2][c], uc[3][c], uc[4][c]};
        double vv[2], dd[2];
        gauss_ao(u, ak, der, vv, dd);
#pragma unroll
        for (int g = 0; g < 2; g++) { cv[g][c] = vv[g]; cd[g][c] = dd[g]; }
    }
#pragma unroll
    for (int g = 0; g < 2; g++) {
        double xv[4], xd[4] = {0.0, 0.0, 0.0, 0.0};
        tang_back(e, cv[g], xv);
        if (der) tang_back(e, cd[g], xd);
#pragma unroll
        for (int r = 0; r < 4; r++) { v[r][g] = xv[r]; d[r][g] = xd[r]; }
    }
}

#if defined(__CUDACC__)
// The same pass spread over the 4 lanes of an aligned lane group: lane q projects the 5 line values onto
// field q with its row of L, runs gauss_ao for it, the fields' Gauss-point values and derivatives are
// exchanged with shuffles, and lane q forms its own component with its row of R: vq[g], dq[g].
__device__ __forceinline__ void tang_ao_x4(const TangEig& e, const double (*x)[4], const AOConst& ak, bool der,
                                           unsigned gmask, double* vq, double* dq)
{
    const int q = threadIdx.x & 3;
    const int lane0 = threadIdx.x & 28;
    const double bU = e.b1h * e.U, bV = e.b1h * e.V, b2h = e.b1h * e.hq2, Vci = e.V * e.ci2, Vc = e.V * e.c;
    auto pick = [&](double a, double b, double c, double d) { return q == 0 ? a : q == 1 ? b : q == 2 ? c : d; };
    const double l0 = pick(b2h + Vci, fma(-2.0, b2h, 1.0), e.U, b2h - Vci), l1 = pick(-bU, scale2<1>(bU), -1.0, -bU);
    const double l2 = pick(-(bV + e.ci2), scale2<1>(bV), 0.0, e.ci2 - bV), l3 = pick(e.b1h, -scale2<1>(e.b1h), 0.0, e.b1h);
    double u[5];
#pragma unroll
    for (int s = 0; s < 5; s++) u[s] = fma(l3, x[s][3], fma(l2, x[s][2], fma(l1, x[s][1], l0 * x[s][0])));
    double cv[2], cd[2];
    gauss_ao(u, ak, der, cv, cd);
    const double r0 = pick(1.0, e.U, e.V - e.c, e.H - Vc), r1 = pick(1.0, e.U, e.V, e.hq2);
    const double r2 = pick(0.0, -1.0, 0.0, -e.U), r3 = pick(1.0, e.U, e.V + e.c, e.H + Vc);
#pragma unroll
    for (int g = 0; g < 2; g++) {
        auto back = [&](double f) {
            const double f0 = __shfl_sync(gmask, f, lane0), f1 = __shfl_sync(gmask, f, lane0 + 1);
            const double f2 = __shfl_sync(gmask, f, lane0 + 2), f3 = __shfl_sync(gmask, f, lane0 + 3);
            return fma(r3, f3, fma(r2, f2, fma(r1, f1, r0 * f0)));
        };
        vq[g] = back(cv[g]);
        dq[g] = der ? back(cd[g]) : 0.0;          // `der` is the same for the 4 lanes
    }
}
#endif

// ---------------------------------------------------------------- gas-kinetic flux
// Every Maxwellian is handled in the frame that moves with its own tangential velocity V (2D):
// there the peculiar tangential velocity c = v - V is one more internal degree of freedom beside
// xi, odd moments of c vanish, and <psi (a.psi) u^n> takes the 1D form with Kt = K + 1 internal
// degrees (1D: Kt = K) plus one product for the tangential momentum; the moments' sums are moved
// back out of the frame.  On this part the flux is bound by the FP64 issue rate (one warp
// instruction per 64 cycles and scheduler), so what counts is the number of FP64 instructions.
// Operations per Gauss point (first / second stage) and flux launch at 1024^2:
//   lab-frame moments in both directions, solves for the micro-slopes      1433 / 1389   8.26 ms
//   moving frames, simplified time coefficients                             897 /  824   6.22 ms
//   divisions, roots, exp, erfc and the Gauss-point quartics in integers,
//   doubled energy sums                                                     893 /  820   3.79 ms
//   micro-slopes as derivatives of the primitives (struct Slope)            829 /  756   3.49 ms

// Primitive description of one Maxwellian (Eq. (3)) in its own tangential frame: h = p/rho.
template <int DIM>
struct MState {
    double rho, ri, U, hU, V, hV, p, h;   // hU, hV: halves
    double u2, H;                          // U^2 + h; H = (E + p)/rho, E without the tangential kinetic energy
};

// W_k-direction d in the frame of s, with what the closed forms share: R = d1 - U d0 (rho dU),
// S = d1 + R, dp (pressure), d2, d3 in the frame.
struct Dir { double d0, d1, d2, d3, R, S, dp; };

template <int NV>
HGKS_HD __forceinline__ double dotv(const double* a, const double* b)
{
    double s = a[0] * b[0];
#pragma unroll
    for (int k = 1; k < NV; k++) s = fma(a[k], b[k], s);
    return s;
}

template <int DIM>
HGKS_HD __forceinline__ bool make_state(const double* W, const FluxConst& fc, MState<DIM>& s)
{
    s.rho = W[0];
    s.ri = rcp_nr(s.rho);
    s.U = W[1] * s.ri;
    s.hU = scale2<-1>(s.U);
    double E = W[DIM + 1];
    if constexpr (DIM == 2) {
        s.V = W[2] * s.ri;
        s.hV = scale2<-1>(s.V);
        E = fma(-s.hV, W[2], E);
    } else {
        s.V = s.hV = 0.0;
    }
    s.p = fc.gm1 * fma(-s.hU, W[1], E);
    s.h = s.p * s.ri;
    s.u2 = fma(s.U, s.U, s.h);
    s.H = fma(s.hU, s.U, fc.gq * s.h);
    return positive(s.rho) && positive(s.p);
}

// A direction d of the conserved variables (lab frame) in the frame of s.
template <int DIM>
HGKS_HD __forceinline__ void in_frame(const MState<DIM>& s, const FluxConst& fc, const double* d, Dir& D)
{
    D.d0 = d[0]; D.d1 = d[1];
    if constexpr (DIM == 2) {
        D.d2 = fma(-s.V, d[0], d[2]);
        D.d3 = fma(-s.V, fma(-s.hV, d[0], d[2]), d[3]);
    } else {
        D.d2 = 0.0;
        D.d3 = d[2];
    }
    D.R = fma(-s.U, D.d0, D.d1);
    D.S = D.d1 + D.R;
    D.dp = fc.gm1 * fma(-s.hU, D.S, D.d3);
}

// The Euler x-flux derivative dF/dW d in the frame of s.
template <int DIM>
HGKS_HD __forceinline__ void jac_x(const MState<DIM>& s, const Dir& d, double* out)
{
    out[0] = d.d1;
    out[1] = fma(s.U, d.S, d.dp);
    if constexpr (DIM == 2) out[2] = s.U * d.d2;
    out[DIM + 1] = fma(s.H, d.R, s.U * (d.d3 + d.dp));
}

// -W_t of the slopes d (x) and e (y) from the Euler compatibility (Eq. (9)) at fixed lab
// position, as a direction in the frame of s: dF/dW d + dG/dW e with no tangential velocity, plus
// V e for the motion of the frame.
template <int DIM>
HGKS_HD __forceinline__ void minus_w_t(const MState<DIM>& s, const FluxConst& fc, const Dir& d, const Dir& e, Dir& n)
{
    if constexpr (DIM == 2) {
        const double sum = d.d1 + e.d2;
        n.d0 = fma(s.V, e.d0, sum);
        n.d1 = fma(s.V, e.d1, fma(s.U, sum + d.R, d.dp));
        n.d2 = fma(s.V, e.d2, fma(s.U, d.d2, e.dp));
        n.d3 = fma(s.V, e.d3, fma(s.H, d.R + e.d2, s.U * (d.d3 + d.dp)));
    } else {
        double f[3];
        jac_x<1>(s, d, f);
        n.d0 = f[0]; n.d1 = f[1]; n.d2 = 0.0; n.d3 = f[2];
    }
    n.R = fma(-s.U, n.d0, n.d1);
    n.S = n.d1 + n.R;
    n.dp = fc.gm1 * fma(-s.hU, n.S, n.d3);
}

// Micro-slope of one side (Eq. (8)).  <a> = dW/rho makes (a.psi) g the derivative of g along d,
// so it is kept as the derivatives of the primitives, al = d ln rho, be = dU, ga = dV, de = dh,
// ka = Kt dh, and every moment is the derivative of a half-line moment: no solve for a, moments up to
// u^4 rather than u^6, and the time slope from the primitive Euler equations (14 operations against
// 24 through the conserved ones).
struct Slope { double al, be, ga, de, ka; };

// What the conversion from conserved derivatives needs: lU = U/(2h); e = (gamma-1)/rho;
// z = |(U, V)|^2/2 - h/(gamma-1).
struct SlopeC { double lU, e, z; };

template <int DIM>
HGKS_HD __forceinline__ void slope_of(const MState<DIM>& s, const FluxConst& fc, const SlopeC& k, const double* d, Slope& a)
{
    a.al = s.ri * d[0];
    a.be = s.ri * fma(-s.U, d[0], d[1]);
    double x = fma(-s.U, d[1], fma(k.z, d[0], d[DIM + 1]));
    if constexpr (DIM == 2) {
        a.ga = s.ri * fma(-s.V, d[0], d[2]);
        x = fma(-s.V, d[2], x);
    } else {
        a.ga = 0.0;
    }
    a.de = k.e * x;
    a.ka = fc.Kt * a.de;
}

// -W_t of the slopes a (x) and b (y) from the Euler compatibility (Eq. (9)), as a slope: the Euler
// equations in the primitives.
template <int DIM>
HGKS_HD __forceinline__ void slope_minus_t(const MState<DIM>& s, const FluxConst& fc, const Slope& a, const Slope& b, Slope& c)
{
    const double px = fma(s.h, a.al, a.de), gh = fc.gm1 * s.h;        // p_x/rho
    if constexpr (DIM == 2) {
        const double div = a.be + b.ga;
        c.al = fma(s.U, a.al, fma(s.V, b.al, div));
        c.be = fma(s.U, a.be, fma(s.V, b.be, px));
        c.ga = fma(s.U, a.ga, fma(s.V, b.ga, fma(s.h, b.al, b.de)));
        c.de = fma(s.U, a.de, fma(s.V, b.de, gh * div));
    } else {
        c.al = fma(s.U, a.al, a.be);
        c.be = fma(s.U, a.be, px);
        c.ga = 0.0;
        c.de = fma(s.U, a.de, gh * a.be);
    }
    c.ka = fc.Kt * c.de;
}

// Half-line moments: u[n] = rho <u^n> on one half line (n <= 4) with the multiples that the
// derivatives need, G = d u[0]/dU (the density at u = 0, signed), hG its half, and Kh = Kt h = <c^2 + xi^2>.
struct Mom { double u[5], G, hG, u1x2, u1x3, u2x3, u2x6, u3x4, Kh; };

// T(n) = <u^n (a.psi)>, the derivative of u[n]: d/dh = (d/dU)^2/2, d u[0]/dU = G, d u[1]/dU = u[0].
HGKS_HD __forceinline__ double mom_t0(const Slope& a, const Mom& m, const SlopeC& k) { return fma(a.al, m.u[0], fma(-k.lU, a.de, a.be) * m.G); }
HGKS_HD __forceinline__ double mom_t1(const Slope& a, const Mom& m) { return fma(a.al, m.u[1], fma(a.be, m.u[0], a.de * m.hG)); }
HGKS_HD __forceinline__ double mom_t2(const Slope& a, const Mom& m) { return fma(a.al, m.u[2], fma(a.be, m.u1x2, a.de * m.u[0])); }
HGKS_HD __forceinline__ double mom_t3(const Slope& a, const Mom& m) { return fma(a.al, m.u[3], fma(a.be, m.u2x3, a.de * m.u1x3)); }
HGKS_HD __forceinline__ double mom_t4(const Slope& a, const Mom& m) { return fma(a.al, m.u[4], fma(a.be, m.u3x4, a.de * m.u2x6)); }

// <u^n psi (a.psi)> in the frame, given T(n), T(n+1), T(n+2).  The energy component (of u^2 + Kt h) is doubled
// here and in every sum over the sides; flux_finish halves the sums (an exponent decrement).
template <int DIM>
HGKS_HD __forceinline__ void mom_g(const Slope& a, const Mom& m, int n, double t0, double t1, double t2, double* out)
{
    out[0] = t0;
    out[1] = t1;
    if constexpr (DIM == 2) out[2] = a.ga * m.u[n];
    out[DIM + 1] = fma(m.Kh, t0, fma(a.ka, m.u[n], t2));
}

// acc (+)= the moment vector c of the frame of s as seen from the lab; TWICE: with doubled energy
// component, which then gains V (2 c2 + V c0) where the energy gains V (c2 + V c0/2).
template <int DIM, bool FIRST, bool TWICE>
HGKS_HD __forceinline__ void add_lab(const MState<DIM>& s, const double* c, double* acc)
{
    double l[DIM + 2];
    l[0] = c[0];
    l[1] = c[1];
    if constexpr (DIM == 2) {
        const double in = TWICE ? fma(s.V, c[0], scale2<1>(c[2])) : fma(s.hV, c[0], c[2]);
        l[2] = FIRST ? fma(s.V, c[0], c[2]) : fma(s.V, c[0], acc[2] + c[2]);
        l[3] = FIRST ? fma(s.V, in, c[3]) : fma(s.V, in, acc[3] + c[3]);
    } else {
        l[2] = FIRST ? c[2] : acc[2] + c[2];
    }
    acc[0] = FIRST ? l[0] : acc[0] + l[0];
    acc[1] = FIRST ? l[1] : acc[1] + l[1];
#pragma unroll
    for (int k = 2; k < DIM + 2; k++) acc[k] = l[k];
}

// The same for <u^n psi g> = (u_n, u_n+1, 0, (u_n+2 + Kt h u_n)/2), energy doubled.
template <int DIM, bool FIRST>
HGKS_HD __forceinline__ void add_psi_lab(const MState<DIM>& s, const Mom& m, int n, double* acc)
{
    const double en = fma(m.Kh, m.u[n], m.u[n + 2]);
    if constexpr (DIM == 2) {
        const double v = s.V * m.u[n];
        acc[2] = FIRST ? v : acc[2] + v;
        acc[3] = FIRST ? fma(s.V, v, en) : fma(s.V, v, acc[3] + en);
    } else {
        acc[2] = FIRST ? en : acc[2] + en;
    }
    acc[0] = FIRST ? m.u[n] : acc[0] + m.u[n];
    acc[1] = FIRST ? m.u[n + 1] : acc[1] + m.u[n + 1];
}

#if defined(__CUDACC__)
__device__ __noinline__ double erfc_far(double y) { return erfc(y); }
#endif

// exp(-x^2) and erfc(|x|): below |x| = 8 from the fixed-point exponential and erfcx(|x|) =
// exp(x^2) erfc(|x|), the library erfc beyond.
HGKS_HD __forceinline__ void exp_erfc(double x, double& ex2, double& E)
{
    const double x2 = x * x;
#ifdef __CUDA_ARCH__
    if ((unsigned)__double2hiint(x2) < 0x40500000u) { fixed::exp_erfc(fabs(x), x2, ex2, E); return; }
    ex2 = exp_neg(x2);
    E = erfc_far(fabs(x));
#else
    ex2 = exp(-x2);
    E = erfc(fabs(x));
#endif
}

// Half-line moments of the left state over u > 0 (sign = +1) or of the right state over
// u < 0 (sign = -1), carrying the density: u[n] = rho <u^n> on the half line, with
// <1> = erfc(-+sqrt(lam) U)/2, <u> = U <1> +- exp(-lam U^2)/(2 sqrt(pi lam)) and
// <u^(n+2)> = U <u^(n+1)> + (n+1) h <u^n>; lam = 1/(2h), sl its root.
// With x = sqrt(lam) U, erfc(-+x) is formed from E = erfc(|x|): the half line that the mean
// velocity points into holds 1 - E/2 of the mass, the other E/2.
template <int DIM>
HGKS_HD __forceinline__ void half_moments(const MState<DIM>& s, double sl, int sign, const FluxConst& fc, Mom& m)
{
    const double x = sl * s.U;
    double ex2, E;
    exp_erfc(x, ex2, E);
    const double g0 = ex2 * (0.56418958354775628695 * sl);          // sqrt(lam/pi) exp(-lam U^2)
    const double e = s.p * g0, G = s.rho * g0;                      // rho h = p
    m.G = sign > 0 ? G : -G;
    m.hG = scale2<-1>(m.G);
#ifdef __CUDA_ARCH__
    const bool neg = __double2hiint(x) < 0;         // (at x = 0 both forms below give half the mass)
#else
    const bool neg = x < 0.0;
#endif
    const bool into = (sign > 0) != neg;
    const double hr = scale2<-1>(s.rho);
    m.u[0] = into ? fma(-hr, E, s.rho) : hr * E;
    m.u[1] = fma(s.U, m.u[0], sign > 0 ? e : -e);
    m.u[2] = fma(s.U, m.u[1], s.h * m.u[0]);
    m.u1x2 = scale2<1>(m.u[1]);
    m.u1x3 = 3.0 * m.u[1];
    m.u[3] = fma(s.U, m.u[2], s.h * m.u1x2);
    m.u2x3 = 3.0 * m.u[2];
    m.u2x6 = scale2<1>(m.u2x3);
    m.u[4] = fma(s.U, m.u[3], s.h * m.u2x3);
    m.u3x4 = scale2<2>(m.u[3]);
    m.Kh = fc.Kt * s.h;
}

// Sums over the two sides (left over u > 0, right over u < 0), lab frame, energy components doubled
// (one multiplication less per vector; the flux launch went from
// 4.02 to 3.79 ms at 1024^2): the equilibrium state and its slopes (Eqs. (46)-(47))
// and the moments int u psi of the three non-equilibrium terms of Eq. (10): S4 (g^k), S5 ((a1 u +
// a2 v) g^k), S6n (-A^k g^k).  D5, D6n: the density moments int psi of the last two (Prandtl fix only).
template <int DIM>
struct FluxSums { double Wc[DIM + 2], Wx[DIM + 2], Wy[DIM + 2], S4[DIM + 2], S5[DIM + 2], S6n[DIM + 2], D5[DIM + 2], D6n[DIM + 2]; };

// One side's share of the sums (left: over u > 0, else over u < 0), from its state and its normal (x) and
// tangential (y) derivatives; FIRST: stored, else added.
// Returns false if the state is non-physical.
template <int DIM, bool PRFIX, bool FIRST>
HGKS_HD __forceinline__ bool flux_side(const FluxConst& fc, const double* W, const double* Wx, const double* Wy, bool left,
                                       FluxSums<DIM>& q, double& p)
{
    constexpr int NV = DIM + 2;
    MState<DIM> s;
    if (!make_state<DIM>(W, fc, s)) return false;
    p = s.p;
    const double sl = rsqrt_nr(scale2<1>(s.h));      // sqrt(lambda)
    Mom m;
    half_moments<DIM>(s, sl, left ? +1 : -1, fc, m);
    add_psi_lab<DIM, FIRST>(s, m, 0, q.Wc);
    SlopeC k;
    k.lU = sl * (sl * s.U);
    k.e = fc.gm1 * s.ri;
    k.z = fma(s.hU, s.U, -(fc.rgm1 * s.h));
    if constexpr (DIM == 2) k.z = fma(s.hV, s.V, k.z);
    Slope a, b;
    double g[NV];
    slope_of<DIM>(s, fc, k, Wx, a);
    const double ta0 = mom_t0(a, m, k), ta1 = mom_t1(a, m), ta2 = mom_t2(a, m);
    mom_g<DIM>(a, m, 0, ta0, ta1, ta2, g);
    add_lab<DIM, FIRST, true>(s, g, q.Wx);
    // int u psi (a1 u + a2 v) g of this side (L5) and, for the Prandtl fix, int psi (a1 u + a2 v) g
    double L5[NV], L[NV];
    const bool noneq = !fc.tau_zero;
    if (noneq) {
        const double ta3 = mom_t3(a, m), ta4 = mom_t4(a, m);
        mom_g<DIM>(a, m, 2, ta2, ta3, ta4, L5);
        if constexpr (PRFIX) mom_g<DIM>(a, m, 1, ta1, ta2, ta3, L);
    }
    if constexpr (DIM == 2) {
        slope_of<DIM>(s, fc, k, Wy, b);
        const double tb0 = mom_t0(b, m, k), tb1 = mom_t1(b, m), tb2 = mom_t2(b, m);
        mom_g<DIM>(b, m, 0, tb0, tb1, tb2, g);
        add_lab<DIM, FIRST, true>(s, g, q.Wy);
        if (noneq) {
            // v = V + c: the c part has <u^n c psi (b.psi)> = dV u_n, dV u_(n+1), h T_b(n) + dh u_n
            // and dV (u_(n+2) + (Kt + 2) h u_n) (doubled)
            const double kc = fc.ktp2 * s.h;
            if constexpr (PRFIX) {
                L[0] = fma(s.V, g[0], fma(b.ga, m.u[0], L[0]));
                L[1] = fma(s.V, g[1], fma(b.ga, m.u[1], L[1]));
                L[2] = fma(s.V, g[2], fma(s.h, tb0, fma(b.de, m.u[0], L[2])));
                L[3] = fma(s.V, g[3], fma(b.ga, fma(kc, m.u[0], m.u[2]), L[3]));
                add_lab<DIM, FIRST, true>(s, L, q.D5);
            }
            const double tb3 = mom_t3(b, m);
            mom_g<DIM>(b, m, 1, tb1, tb2, tb3, g);
            L5[0] = fma(s.V, g[0], L5[0] + g[2]);
            L5[1] = fma(s.V, g[1], fma(b.ga, m.u[2], L5[1]));
            L5[2] = fma(s.V, g[2], fma(s.h, tb1, fma(b.de, m.u[1], L5[2])));
            L5[3] = fma(s.V, g[3], fma(b.ga, fma(kc, m.u[1], m.u[3]), L5[3]));
        }
    } else if constexpr (PRFIX) {
        if (noneq) add_lab<DIM, FIRST, true>(s, L, q.D5);
    }
    if (!noneq) return true;
    add_lab<DIM, FIRST, true>(s, L5, q.S5);
    add_psi_lab<DIM, FIRST>(s, m, 1, q.S4);
    // time slope A from <a1 u + a2 v + A> = 0 (Eq. (9)), with the opposite sign
    Slope c;
    slope_minus_t<DIM>(s, fc, a, b, c);
    const double tc1 = mom_t1(c, m), tc2 = mom_t2(c, m), tc3 = mom_t3(c, m);
    mom_g<DIM>(c, m, 1, tc1, tc2, tc3, g);
    add_lab<DIM, FIRST, true>(s, g, q.S6n);
    if constexpr (PRFIX) {
        mom_g<DIM>(c, m, 0, mom_t0(c, m, k), tc1, tc2, g);
        add_lab<DIM, FIRST, true>(s, g, q.D6n);
    }
    return true;
}

// M2 = int u psi (abar1 u + abar2 v) g0 in the frame of s: since <abar> = d makes (abar.psi) g0 the
// derivative of g0 along d, it is Pi'(W) d + Sigma'(W) e + V dF/dW e with Pi = int u^2 psi g and
// Sigma = int u c psi g, no solve for abar needed (chain rule through rho, U, V, h at V = 0).
template <int DIM>
HGKS_HD __forceinline__ void m2_term(const MState<DIM>& s, const FluxConst& fc, const Dir& d, const Dir& e, double* out)
{
    constexpr int NV = DIM + 2;
    const double U = s.U, h = s.h, U2 = U * U;
    const double rdh = fma(-h, d.d0, d.dp);
    const double k6h = fc.k6 * h, k3h = fc.k3 * h, uk = U2 + k6h;
    const double p3 = 0.5 * fma(U2, uk, k3h * h);
    const double p3U = fma(2.0, U2, k6h);           // times U
    const double p3h = fma(fc.hk6, U2, k3h);
    out[0] = fma(U, d.S, d.dp);
    out[1] = fma(U, fma(3.0, rdh, fma(3.0, h, U2) * d.d0), (3.0 * s.u2) * d.R);
    out[NV - 1] = fma(p3, d.d0, fma(p3U, U * d.R, p3h * rdh));
    if constexpr (DIM == 2) {
        double f[4];
        jac_x<2>(s, e, f);
        out[0] = fma(s.V, f[0], out[0] + f[2]);
        out[1] = fma(s.V, f[1], fma(s.u2, e.d2, out[1]));
        out[2] = fma(s.V, f[2], fma(s.u2, d.d2, fma(U, e.dp, h * e.R)));
        out[3] = fma(s.V, f[3], fma(s.hU * (uk - h), e.d2, out[3]));
    }
}

// Time coefficients.  With e_d = exp(-d/tau) and P_d = tau (1 - e_d) the integrals over [0, d] of the
// factors of Eq. (10) are
//   C0 = d - P, C1 = tau (2P - d (1 + e)), C2 = tau P + d^2/2 - tau d, C3 = P, C4 = tau (d e - 2P), C5 = -tau P;
// the stages' combinations of d = dt and dt/2 simplify (o = 1 - e_{dt/2}, P = tau o, Q = dt e_{dt/2} - 2P):
//   STAGE 0: A0 = C(dt/2) and A1 = (8 C(dt/2) - C(dt))/3 from their C3 and C4 alone;
//   STAGE 1: (4/3)(C(dt) - 2 C(dt/2)) = (4/3) (P o, P Q, dt^2/4 - P^2, -P o, -P Q, P^2).
template <int STAGE>
HGKS_HD __forceinline__ void time_coefs(double dt, double tau, double* A0, double* A1)
{
    const double e = exp_neg(0.5 * dt * rcp_nr(tau));
    const double o = 1.0 - e, P = tau * o, dte = dt * e;
    if constexpr (STAGE == 0) {
        const double hd = 0.5 * dt, td = tau * dt;
        const double c4 = tau * fma(0.5, dte, -2.0 * P);                  // C4(dt/2)
        const double Pd = fma(P, e, P);                                    // P_dt
        const double c4d = tau * fma(dte, e, -2.0 * Pd);                  // C4(dt)
        A0[0] = hd - P; A0[3] = P; A0[4] = c4; A0[5] = -(tau * P);
        A0[1] = fma(-0.5, td, -c4);
        A0[2] = fma(0.125 * dt, dt, fma(-0.5, td, -A0[5]));
        A1[3] = (1.0 / 3.0) * fma(8.0, P, -Pd);
        A1[4] = (1.0 / 3.0) * fma(8.0, c4, -c4d);
        A1[5] = -(tau * A1[3]);
        A1[0] = dt - A1[3];
        A1[1] = -td - A1[4];
        A1[2] = fma((1.0 / 6.0) * dt, dt, -td - A1[5]);
    } else {
        const double kP = (4.0 / 3.0) * P;
        const double Q = fma(-2.0, P, dte);
        A0[0] = kP * o; A0[1] = kP * Q;
        A0[3] = -A0[0]; A0[4] = -A0[1]; A0[5] = kP * P;
        A0[2] = fma((1.0 / 3.0) * dt, dt, -A0[5]);
    }
}

// Gas-kinetic flux at one Gauss point from the sums over the two sides and their pressures.
template <int DIM, int STAGE, bool PRFIX>
HGKS_HD __forceinline__ bool flux_finish(const FluxConst& fc, FluxSums<DIM>& q, double pl, double pr, double dt,
                                         double* o0, double* o1)
{
    constexpr int NV = DIM + 2;
    // the sums' energies are doubled
    q.Wc[NV - 1] = scale2<-1>(q.Wc[NV - 1]);
    q.Wx[NV - 1] = scale2<-1>(q.Wx[NV - 1]);
    if constexpr (DIM == 2) q.Wy[NV - 1] = scale2<-1>(q.Wy[NV - 1]);
    if (!fc.tau_zero) {
        q.S4[NV - 1] = scale2<-1>(q.S4[NV - 1]);
        q.S5[NV - 1] = scale2<-1>(q.S5[NV - 1]);
        q.S6n[NV - 1] = scale2<-1>(q.S6n[NV - 1]);
        if constexpr (PRFIX) {
            q.D5[NV - 1] = scale2<-1>(q.D5[NV - 1]);
            q.D6n[NV - 1] = scale2<-1>(q.D6n[NV - 1]);
        }
    }
    MState<DIM> sc;
    if (!make_state<DIM>(q.Wc, fc, sc)) return false;

    // equilibrium flux moments in the frame of Wc: M1 = int u psi g0 = F(Wc), M3 = int u psi Abar g0 =
    // dF/dW Wc_t (formed with the opposite sign), M2 = int u psi (abar1 u + abar2 v) g0
    Dir dx, dy, dn;
    double M1[NV], M3n[NV];
    in_frame<DIM>(sc, fc, q.Wx, dx);
    if constexpr (DIM == 2) in_frame<DIM>(sc, fc, q.Wy, dy);
    minus_w_t<DIM>(sc, fc, dx, dy, dn);
    jac_x<DIM>(sc, dn, M3n);
    M1[0] = q.Wc[1];
    M1[1] = fma(q.Wc[1], sc.U, sc.p);
    M1[NV - 1] = q.Wc[1] * sc.H;

    // collision time (Sec. 3 preamble)
    const double jump = fabs((pl - pr) * rcp_nr(pl + pr));
    double tau;
    if (fc.tau_zero) tau = 0.0;
    else if (fc.viscous) tau = fma(fc.c2 * jump, dt, fc.mu * rcp_nr(sc.p));
    else tau = fma(fc.c2, jump, fc.c1) * dt;

    double A0[6], A1[6];
    const bool eq_only = is_zero(tau);
    if (eq_only) {
        // F(d) = d M1 + d^2/2 M3
        A0[0] = STAGE == 0 ? 0.5 * dt : 0.0;
        A0[2] = STAGE == 0 ? 0.125 * dt * dt : (1.0 / 3.0) * dt * dt;
        A1[0] = dt;
        A1[2] = (1.0 / 6.0) * dt * dt;
    } else {
        time_coefs<STAGE>(dt, tau, A0, A1);
    }
    double c0[NV], c1[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) {
        const double m0 = -(A0[2] * M3n[k]), m1 = STAGE == 0 ? -(A1[2] * M3n[k]) : 0.0;
        c0[k] = DIM == 2 && k == 2 ? m0 : fma(A0[0], M1[k], m0);
        if constexpr (STAGE == 0) c1[k] = DIM == 2 && k == 2 ? m1 : fma(A1[0], M1[k], m1);
    }
    double M2[NV];
    if (!eq_only) {
        m2_term<DIM>(sc, fc, dx, dy, M2);
#pragma unroll
        for (int k = 0; k < NV; k++) {
            c0[k] = fma(A0[1], M2[k], c0[k]);
            if constexpr (STAGE == 0) c1[k] = fma(A1[1], M2[k], c1[k]);
        }
    }
    add_lab<DIM, true, false>(sc, c0, o0);
    if constexpr (STAGE == 0) add_lab<DIM, true, false>(sc, c1, o1);
    if (eq_only) return true;
#pragma unroll
    for (int k = 0; k < NV; k++) {
        o0[k] = fma(A0[3], q.S4[k], fma(A0[4], q.S5[k], fma(-A0[5], q.S6n[k], o0[k])));
        if constexpr (STAGE == 0) o1[k] = fma(A1[3], q.S4[k], fma(A1[4], q.S5[k], fma(-A1[5], q.S6n[k], o1[k])));
    }
    if constexpr (PRFIX) {
        // Prandtl-number fix (an extension: the paper's BGK flux has Pr = 1).  The energy flux
        // gains (1/Pr - 1) q, q the time-integrated heat flux of the distribution of Eq. (10)
        // relative to the equilibrium velocity (Uc, Vc).  With l = (|Uc|^2/2, -Uc, -Vc, 1),
        // int (u - Uc)(|u - Uc|^2 + xi^2)/2 phi = l.(int u psi phi) - Uc l.(int psi phi) for
        // every term phi of Eq. (10); the g0 term carries no heat flux, the density moments of
        // the (abar u) g0 and Abar g0 terms are -Wc_t and Wc_t (compatibility, Eq. (9)), those of
        // g^k sum to Wc (Eq. (46)).  The equilibrium terms are in the frame of Wc, where l has no
        // tangential part.  (a compile-time variant, so that the Pr = 1 flux keeps its registers)
        double lf[NV], lv[NV], Qh[6];
        lf[0] = sc.hU * sc.U; lf[1] = -sc.U; lf[NV - 1] = 1.0;
        lv[0] = lf[0]; lv[1] = lf[1]; lv[NV - 1] = 1.0;
        if constexpr (DIM == 2) { lf[2] = 0.0; lv[0] = fma(sc.hV, sc.V, lf[0]); lv[2] = -sc.V; }
        auto frame_dot = [&](const double* x) { return fma(lf[0], x[0], fma(lf[1], x[1], x[NV - 1])); };
        const double lN = fma(lf[0], dn.d0, fma(lf[1], dn.d1, dn.d3));       // -l.Wc_t
        Qh[1] = fma(-sc.U, lN, frame_dot(M2));
        Qh[2] = fma(sc.U, lN, -frame_dot(M3n));
        Qh[3] = fma(-sc.U, dotv<NV>(lv, q.Wc), dotv<NV>(lv, q.S4));
        Qh[4] = fma(-sc.U, dotv<NV>(lv, q.D5), dotv<NV>(lv, q.S5));
        Qh[5] = fma(sc.U, dotv<NV>(lv, q.D6n), -dotv<NV>(lv, q.S6n));
        double q0 = 0.0, q1 = 0.0;
#pragma unroll
        for (int j = 1; j < 6; j++) {
            q0 = fma(A0[j], Qh[j], q0);
            if constexpr (STAGE == 0) q1 = fma(A1[j], Qh[j], q1);
        }
        o0[NV - 1] = fma(fc.prfix, q0, o0[NV - 1]);
        if constexpr (STAGE == 0) o1[NV - 1] = fma(fc.prfix, q1, o1[NV - 1]);
    }
    return true;
}

// Gas-kinetic flux at one Gauss point in the local frame (x = normal); Sec. 2.1, Eqs. (6)-(12),
// (46)-(47), collision time of Sec. 3.  Inputs: side states and their normal (x) and tangential
// (y, 2D) derivatives.  With Fd = F(dt), Fh = F(dt/2) of Eq. (12):
//   STAGE 0: o0 = Fh (for W*, Eq. (19)),  o1 = (8 Fh - Fd)/3 = dt F^n + dt^2/6 dF^n (Eqs. (17)-(18), (20))
//   STAGE 1: o0 = (4/3)(Fd - 2 Fh) = dt^2/3 dF* (Eqs. (18), (20))
// Returns false if a side or the equilibrium state is non-physical.
template <int DIM, int STAGE, bool PRFIX = false>
HGKS_HD __forceinline__ bool gks_flux(const FluxConst& fc, const double* Wl, const double* Wlx, const double* Wly,
                                         const double* Wr, const double* Wrx, const double* Wry, double dt,
                                         double* o0, double* o1)
{
    FluxSums<DIM> q;
    double pl, pr;
    const bool okl = flux_side<DIM, PRFIX, true>(fc, Wl, Wlx, Wly, true, q, pl);
    const bool okr = okl && flux_side<DIM, PRFIX, false>(fc, Wr, Wrx, Wry, false, q, pr);
    if (!okr) return false;
    return flux_finish<DIM, STAGE, PRFIX>(fc, q, pl, pr, dt, o0, o1);
}

}  // namespace hgks
