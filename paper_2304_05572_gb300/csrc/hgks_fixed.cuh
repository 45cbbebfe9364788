// hgks_fixed.cuh -- reciprocal, reciprocal square root, exponential and erfc of the flux in 64-bit
// fixed point.
//
// The FP64 pipe of this part takes one warp instruction per 64 cycles and scheduler (measured
// 65-76, comparisons and conversions from and to doubles included), while the integer pipe issues a
// 32 x 32 + 64 bit multiply-add in 2 and everything else in 1 (a 64 x 64 -> 64 bit high product: 10-22).  A function whose arguments and results have a known
// range is therefore cheaper in integers, at more bits than a double carries: each routine below
// works with 61-63 fraction bits, rounds once, and is within one unit in the last place of the exact
// result (tests/test_fixed_point.py, which compiles this header for the host).
// In place of the FP64 sequences (4 operations for 1/x, 7 for 1/sqrt(x), about 20 for an exponential,
// 17 for erfc; 7, 2, 3 and 2 of them per Gauss point) the flux launch at 1024^2 went from 6.22 to
// 5.18 ms.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define HGKS_FX __device__ __forceinline__
#define HGKS_FX_DATA __device__
#else
#include <cmath>
#include <cstring>
#define HGKS_FX inline
#define HGKS_FX_DATA
#endif

namespace hgks {
namespace fixed {

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;

#ifdef __CUDACC__
HGKS_FX u64 bits_of(double x) { return (u64)__double_as_longlong(x); }
HGKS_FX double of_bits(u64 b) { return __longlong_as_double((long long)b); }
HGKS_FX u32 float_bits(float x) { return __float_as_uint(x); }
HGKS_FX float float_of(u32 b) { return __uint_as_float(b); }
HGKS_FX float approx_rcp(float x) { float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
HGKS_FX float approx_rsqrt(float x) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r; }
HGKS_FX int clz32(u32 x) { return __clz((int)x); }
#else
HGKS_FX u64 bits_of(double x) { u64 b; memcpy(&b, &x, 8); return b; }
HGKS_FX double of_bits(u64 b) { double x; memcpy(&x, &b, 8); return x; }
HGKS_FX u32 float_bits(float x) { u32 b; memcpy(&b, &x, 4); return b; }
HGKS_FX float float_of(u32 b) { float x; memcpy(&x, &b, 4); return x; }
#ifndef HGKS_FX_OWN_SEEDS               // (a check may bring seeds as far off as the hardware's may be)
HGKS_FX float approx_rcp(float x) { return 1.0f / x; }
HGKS_FX float approx_rsqrt(float x) { return 1.0f / std::sqrt(x); }
#endif
HGKS_FX int clz32(u32 x) { return __builtin_clz(x); }
#endif

// floor(a b / 2^64) less at most 2: the low halves' product is dropped
HGKS_FX u64 umulhi(u64 a, u64 b)
{
    const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
    const u64 x = (u64)ah * bl, y = (u64)al * bh;
    return (u64)ah * bh + (x >> 32) + (y >> 32);
}

HGKS_FX u64 umulhi_exact(u64 a, u64 b)
{
#ifdef __CUDACC__
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}

// A signed factor in halves: v = hi 2^32 + 2 lo (the last bit dropped), so that every partial product is a
// signed 32 x 32 bit one.
struct Half { int hi, lo; };
HGKS_FX Half halves(i64 v) { return Half{(int)(v >> 32), (int)((u32)v >> 1)}; }

// a b / 2^64 within 3 units; |a|, |b| < 2^63 with |a| + |b| <= 2^63.6
HGKS_FX i64 smulhi(Half a, Half b)
{
    const i64 cross = (i64)a.hi * b.lo + (i64)a.lo * b.hi;
    return (i64)a.hi * b.hi + (cross >> 31);
}

// x > 0 (false for a NaN), x = 0, x finite, |x| <= y for y >= 0 (false for a NaN): on the bit patterns
HGKS_FX bool is_pos(double x) { return bits_of(x) - 1u < 0x7FF0000000000000ull; }
HGKS_FX bool is_zero(double x) { return bits_of(x) << 1 == 0u; }
HGKS_FX bool is_finite(double x) { return ((u32)(bits_of(x) >> 32) & 0x7FF00000u) != 0x7FF00000u; }
HGKS_FX bool abs_le(double x, double y) { return (bits_of(x) & 0x7FFFFFFFFFFFFFFFull) <= bits_of(y); }

// x rounded towards zero to a float; below 2^-126 to zero, from 2^128 on (and a NaN) to an infinity
HGKS_FX float to_float(double x)
{
    const u64 b = bits_of(x);
    const u32 hi = (u32)(b >> 32), e = hi & 0x7FF00000u;
    u32 f = (u32)(b >> 29) - 0xC0000000u;
    f = e < 0x38100000u ? 0u : e > 0x47E00000u ? 0x7F800000u : f;
    return float_of((f & 0x7FFFFFFFu) | (hi & 0x80000000u));
}

// Whether rho > 0 and rho E - (mx^2 + my^2)/2 > 0 beyond doubt, from the components truncated to FP32
// (to_float): truncations and products err by less than 2^-20 of each term, so a difference above 4e-6 of
// rho E is positive (both factors within 1e-12..1e12, where no product leaves the range).
HGKS_FX bool surely_physical(float rho, float mx, float my, float E)
{
    const float re = rho * E, ke = 0.5f * (mx * mx + my * my);
    return rho > 1e-12f && rho < 1e12f && E > 1e-12f && E < 1e12f && re - ke > 4e-6f * re;
}

// y 2^Q rounded down, for 0 <= y < 2^(64-Q)
HGKS_FX u64 to_fixed(double y, int q)
{
    const u64 b = bits_of(y);
    const u32 e = (u32)(b >> 52);
    const u32 s = 1086u - (u32)q - e;                                      // >= 0 in range
    const u64 m = (b << 11) | 0x8000000000000000ull;
    return s < 64u ? m >> s : 0u;
}

// x 2^k for a finite x (zeros and subnormals stay as they are, infinities and NaNs too): an integer
// add to the exponent in place of an FP64 multiplication
template <int K>
HGKS_FX double scale2(double x)
{
    const u64 b = bits_of(x);
    const u32 hi = (u32)(b >> 32), e = hi & 0x7FF00000u;
    const u32 h = e - 0x00100000u < 0x7FE00000u ? hi + (u32)(K * 0x00100000) : hi;
    return of_bits(((u64)h << 32) | (u32)b);
}

// A starting value for the two below: the approximation, which may lie a rounding outside [1/2, 1) at the
// mantissa's ends, brought inside and as a fraction in 2^-32.
HGKS_FX u32 seed(float y0)
{
    y0 = y0 < 0.99999994f ? y0 : 0.99999994f;
    y0 = y0 > 0.5f ? y0 : 0.5f;
    return (float_bits(y0) << 8) | 0x80000000u;
}

// 1/m for m in [1, 2) given in units of 2^-63, as r 2^-63, r in (2^62, 2^63], within 2 units: the 23-bit
// reciprocal of the leading bits and one third-order Newton step, 1/m = y (1 + e + e^2), e = 1 - m y.
HGKS_FX u64 rcp_mantissa(u64 m)
{
    const u32 y = seed(approx_rcp(float_of(0x3F800000u | (u32)(m << 1 >> 41))));
    const u64 p = (u64)(u32)(m >> 32) * y + (((u64)(u32)m * y) >> 32);     // m y, 2^-63
    const i64 e = (i64)(0x8000000000000000ull - p);                        // |e| < 2^42
    const i64 eh = (int)(e >> 12);
    const i64 s = e + ((eh * eh) >> 39);
    return ((u64)y << 31) + (u64)((i64)((int)(s >> 32)) * (i64)y) + (((u64)(u32)s * y) >> 32);
}

// 1/sqrt(m) for m in [1, 4) in units of 2^-62 (frac: 23 fraction bits of m or m/2, odd: m < 2), as r 2^-63:
// the same with 1/sqrt(m) = y (1 + e/2 + 3 e^2/8), e = 1 - m y^2.
HGKS_FX u64 rsqrt_mantissa(u64 m, u32 frac, u32 odd)
{
    const u32 y = seed(approx_rsqrt(float_of((odd ? 0x3F800000u : 0x40000000u) | frac)));
    const u64 p = umulhi(m, (u64)y * y);                                   // m y^2, 2^-62
    const i64 e = (i64)(0x4000000000000000ull - p);                        // e in 2^-62 = e/2 in 2^-63
    const i64 eh = (int)(e >> 11);                                         // 2^-51
    const i64 s = e + ((eh * eh) >> 42) * 3;
    return ((u64)y << 31) + (u64)((i64)((int)(s >> 32)) * (i64)y) + (((u64)(u32)s * y) >> 32);
}

// 1/x.  Out of range: |x| >= 2^1022 gives 0; zero, subnormal, infinite and NaN arguments give a NaN
// (which the flux's physical-state tests reject).
HGKS_FX double rcp(double x)
{
    const u64 b = bits_of(x);
    const u32 hi = (u32)(b >> 32), e0 = (hi >> 20) & 0x7FF;
    const u64 r = rcp_mantissa((b << 11) | 0x8000000000000000ull);
    const u64 mant = ((u64)(2044u - e0) << 52) + ((r + 512u) >> 10);
    const bool in = e0 - 1u < 2044u;
    const u32 h = in ? (u32)(mant >> 32) : e0 - 2045u < 2u ? 0u : 0x7FF80000u;
    return of_bits((((u64)(h | (hi & 0x80000000u))) << 32) | (in ? (u32)mant : 0u));
}

// 1/sqrt(x); a NaN unless x is positive, normal and finite.
HGKS_FX double rsqrt(double x)
{
    const u64 b = bits_of(x);
    const u32 hi = (u32)(b >> 32), e0 = hi >> 20;                          // with the sign bit
    const u32 odd = e0 & 1u;                                               // odd biased exponent: m in [1, 2)
    const u64 r = rsqrt_mantissa(((b << 11) | 0x8000000000000000ull) >> odd, (hi << 3 & 0x007FFFF8u) | ((u32)b >> 29), odd);
    const u64 mant = ((u64)(1021u - (u32)(((int)e0 - 1023) >> 1)) << 52) + ((r + 512u) >> 10);
    const u32 h = e0 - 1u < 2046u ? (u32)(mant >> 32) : 0x7FF80000u;
    return of_bits(((u64)h << 32) | (u32)mant);
}

// IEEE a / b (round to nearest) where a is zero or normal, b normal and the quotient normal and
// below 2^1023; false elsewhere.  The quotient of the mantissas to 61 bits, rounded to 53 and corrected by the sign of the
// exact remainder against half a unit (a quotient of two doubles is never half way between two).
HGKS_FX bool div_rn(double a, double b, double& q)
{
    const u64 ab = bits_of(a), bb = bits_of(b);
    const u32 ah = (u32)(ab >> 32), bh = (u32)(bb >> 32);
    const u32 ea = (ah >> 20) & 0x7FFu, eb = (bh >> 20) & 0x7FFu;
    const u64 ma = (ab & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull, mb = (bb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const u64 t = umulhi(ma << 11, rcp_mantissa(mb << 11));                // ma/mb in 2^-62, (1/2, 2)
    const u32 small = t < 0x4000000000000000ull ? 1u : 0u;                 // quotient below 1
    const u32 sh = 10u - small;
    u64 c = (t + (256ull << (1u - small))) >> sh;                          // 53 bits, unit 2^-52 or 2^-53
    const i64 r2 = (i64)((ma << (52u + small)) - c * mb) * 2;              // twice the remainder (its low 64 bits are all of it)
    c += r2 > (i64)mb ? 1u : 0u;
    c -= r2 < -(i64)mb ? 1u : 0u;
    const u32 e = ea + 1022u - eb - small;                                 // exponent field less 1 (c carries the hidden bit)
    const u64 z = ((u64)e << 52) + c;
    const bool zero = ab << 1 == 0u;
    q = of_bits((zero ? 0u : z) | ((ab ^ bb) & 0x8000000000000000ull));
    return eb - 1u < 2046u && (zero || (ea - 1u < 2046u && e < 2045u));
}

// IEEE sqrt(x) (round to nearest) for positive normal x; false elsewhere.  Rounded from x/sqrt(x) in 2^-61
// and corrected by the remainder x - c^2, which must lie in (-c, c].
HGKS_FX bool sqrt_rn(double x, double& q)
{
    const u64 b = bits_of(x);
    const u32 hi = (u32)(b >> 32), e0 = hi >> 20;
    const u32 odd = e0 & 1u;
    const u64 m = ((b << 11) | 0x8000000000000000ull) >> odd;              // [1, 4) in 2^-62
    const u64 t = umulhi(m, rsqrt_mantissa(m, (hi << 3 & 0x007FFFF8u) | ((u32)b >> 29), odd));   // 2^-61, [1, 2)
    u64 c = (t + 256u) >> 9;
    const u64 m53 = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const i64 r = (i64)((m53 << (53u - odd)) - c * c);                     // low 64 bits of m 2^104 - c^2
    c += r > (i64)c ? 1u : 0u;
    c -= r <= -(i64)c ? 1u : 0u;
    q = of_bits((((u64)(u32)(((int)e0 - 1023) >> 1) + 1022u) << 52) + c);
    return e0 - 1u < 2046u;
}

#include "exp2_table.inc"
HGKS_FX_DATA const u64 c_exp2[64] = HGKS_EXP2_TABLE;

// exp(-y) = r 2^-62 2^-n, r in [2^61, 2^62], for 0 <= y < 708: with y log2(e) = n + j/64 + f,
// exp(-y) = 2^-n 2^(-j/64) exp(-f ln 2), the last factor by its Taylor series to z^6/720 (z < 0.0109,
// remainder 2^-58).  y enters with 57 fraction bits below 64 and with 53 (exactly) above.
struct Exp { u64 r; int n; };

HGKS_FX u64 load_exp2(u32 j)
{
#ifdef __CUDACC__
    return __ldg(c_exp2 + j);
#else
    return c_exp2[j];
#endif
}

HGKS_FX Exp exp_neg(double y)
{
    const int q = (u32)(bits_of(y) >> 32) < 0x40500000u ? 57 : 53;                   // y < 64
    const u64 yf = to_fixed(y, q);                                         // y in 2^-q
    const u64 t = umulhi_exact(yf, 0xB8AA3B295C17F0BCull), tl = yf * 0xB8AA3B295C17F0BCull;   // y log2(e), 2^-(q+63)
    Exp r;
    r.n = (int)(t >> (q - 1));
    const u64 f = (t << (65 - q)) | (tl >> (q - 1));                       // fraction, 2^-64
    const u64 w = umulhi(f << 6, 0xB17217F7D1CF79ABull);                    // w = 64 z, 2^-64
    const u32 w32 = (u32)(w >> 32);
    // A = 1/24 - z/120 + z^2/720 in 2^-36; then 1/6 - z A, 1/2 - z (.), 1 - z (.), 1 - z (.)
    u32 a = 572662306u - (u32)(((u64)w32 * 95443718u) >> 38);
    a = 2863311531u - (u32)(((u64)w32 * a) >> 38);
    u64 p = 0x2AAAAAAAAAAAAAABull - (((u64)w32 * a) >> 10);                // 2^-64
    p = 0x8000000000000000ull - (umulhi(w, p) >> 6);                       // 2^-64
    p = 0x8000000000000000ull - (umulhi(w, p) >> 7);                       // 2^-63
    p = 0x8000000000000000ull - (umulhi(w, p) >> 6);                       // 2^-63
    r.r = umulhi(load_exp2((u32)(f >> 58)), p);                            // 2^-62
    return r;
}

HGKS_FX double exp_value(Exp e)
{
    return of_bits((((u64)(1021 - e.n)) << 52) + ((e.r + 256u) >> 9));
}

// A positive fixed-point number v 2^(-62-n), 2^32 <= v < 2^63, rounded to a double.
HGKS_FX double pack(u64 v, int n)
{
    const int lz = clz32((u32)(v >> 32));
    const u64 s = v << lz;
    return of_bits((((u64)(1023 - lz - n)) << 52) + (s >> 11) + ((s >> 10) & 1u));
}

#include "erfcx_table.inc"

// erfcx(y) = exp(y^2) erfc(y) on [0, 8): per interval [k/4, (k+1)/4) a degree-11 polynomial in
// t = y - (k + 1/2)/4 (Chebyshev interpolant, relative error 2.1e-16; gen_erfcx_table.py).  Here in
// the variable 4t, |4t| <= 1/2: coefficient j in units of 2^-62 4^j.
struct ErfcxQ { i64 b[HGKS_ERFCX_INTERVALS * (HGKS_ERFCX_DEGREE + 1)]; };
constexpr ErfcxQ make_erfcx_q()
{
    constexpr double a[HGKS_ERFCX_INTERVALS * (HGKS_ERFCX_DEGREE + 1)] = HGKS_ERFCX_TABLE;
    ErfcxQ q{};
    for (int k = 0; k < HGKS_ERFCX_INTERVALS; k++) {
        double unit = 4611686018427387904.0;
        for (int j = 0; j <= HGKS_ERFCX_DEGREE; j++) {
            q.b[k * (HGKS_ERFCX_DEGREE + 1) + j] = (i64)(a[k * (HGKS_ERFCX_DEGREE + 1) + j] * unit);
            unit *= 0.25;
        }
    }
    return q;
}
HGKS_FX_DATA constexpr ErfcxQ c_erfcx_q = make_erfcx_q();

// erfcx(y) in 2^-62 for 0 <= y < 8
HGKS_FX u64 erfcx_q(double y)
{
    const u64 yf = to_fixed(y, 58);                                        // 2^-58
    u32 k = (u32)(yf >> 56);
    k = k < HGKS_ERFCX_INTERVALS ? k : HGKS_ERFCX_INTERVALS - 1;
    const i64 t = (i64)(yf - ((u64)k << 56)) - (1ll << 55);                // y - centre, 2^-58
    const Half th = halves((i64)((u64)t << 8));                            // 4t in 2^-64
    const i64* a = c_erfcx_q.b + k * (HGKS_ERFCX_DEGREE + 1);
    i64 c[HGKS_ERFCX_DEGREE + 1];
#ifdef __CUDACC__
#pragma unroll
    for (int j = 0; j <= HGKS_ERFCX_DEGREE; j += 2) {
        const longlong2 v = __ldg((const longlong2*)(a + j));
        c[j] = v.x; c[j + 1] = v.y;
    }
#else
    for (int j = 0; j <= HGKS_ERFCX_DEGREE; j++) c[j] = a[j];
#endif
    i64 p = c[HGKS_ERFCX_DEGREE];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = HGKS_ERFCX_DEGREE - 1; j >= 0; j--) p = c[j] + smulhi(halves(p), th);
    return (u64)p;
}

// exp(-y^2) and erfc(y), y2 = y^2, for 0 <= y < 8
HGKS_FX void exp_erfc(double y, double y2, double& ex, double& er)
{
    const Exp e = exp_neg(y2);
    ex = exp_value(e);
    er = pack(umulhi(e.r << 1, erfcx_q(y) << 1), e.n);
}

// ---------------------------------------------------------------- linear forms of a 5-value window
// Five values in one unit, v[j] = q[j] 2^(1083-E) truncated, E the largest biased exponent among them
// (|v| < 2^61: 60 fraction bits of the window's largest value, where a double sum rounds to 53 of it).
// False where the exponents leave the range in which every result below is a normal double (or a
// value is infinite or a NaN); a window of zeros gives zeros.
HGKS_FX bool window(const double* q, i64* v, int& E)
{
    u32 top = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 5; j++) {
        const u32 h = (u32)(bits_of(q[j]) >> 32) & 0x7FFFFFFFu;
        top = h > top ? h : top;
    }
    const u32 e = top >> 20;
    E = e == 0 ? 100 : (int)e;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int j = 0; j < 5; j++) {
        const u64 b = bits_of(q[j]);
        const u32 hi = (u32)(b >> 32);
        const u32 s = 3u + (u32)E - ((hi >> 20) & 0x7FFu);
        const u64 m = (b << 11) | 0x8000000000000000ull;
        const u64 a = s < 64u ? m >> s : 0u;
        v[j] = (int)hi < 0 ? (i64)(0u - a) : (i64)a;
    }
    return e == 0 || e - 200u < 1700u;
}

// r 2^(E-1023-F) as a double
HGKS_FX double from_fixed(i64 r, int E, int F)
{
    const u64 a = r < 0 ? 0u - (u64)r : (u64)r;
    const u32 h = (u32)(a >> 32);
    const int lz = h ? clz32(h) : 32 + clz32((u32)a | 1u);
    const u64 m = a << lz;
    const u64 d = ((u64)(u32)(E + 62 - F - lz) << 52) + (m >> 11) + ((m >> 10) & 1u);
    return of_bits(a == 0 ? 0u : d | ((u64)r & 0x8000000000000000ull));
}

// Multiplier in [1, 2) as 2^-62 halves, and its exponent
struct Scale { Half m; int e; };
HGKS_FX Scale scale_of(double x)
{
    const u64 b = bits_of(x);
    return Scale{halves((i64)((b << 10 & 0x3FFFFFFFFFFFFC00ull) | 0x4000000000000000ull)), (int)(b >> 52) - 1023};
}

// The quartic through the averages of cells i-2..i+2 at its two Gauss points xi = -+1/(2 sqrt 3): v[0], v[1],
// and (DER) its derivatives there times `inv` (1/h), d[0], d[1].  The values at +-xi are the sum and the
// difference of an even and an odd form, on q2, q1 + q3, q0 + q4 and q3 - q1, q4 - q0, so that both points take 5
// products together (5 more for the derivatives).  Coefficients in 2^-62 (719/720, 1/1080, -1/4320;
// 25 sqrt3/216, -7 sqrt3/432; 2/3, -1/12; -4 sqrt3/9, 13 sqrt3/54, -sqrt3/54), with the last places of one
// of each set chosen so that constants and linear data come out exactly.  Products keep 58 fraction
// bits of the window's largest value: values within 2^-54 of it, derivatives within 2^-53 of it times
// inv, beside their rounding (the FP64 chain: up to 2^-52 and 2^-50).
// A product of halves drops the two low halves' term, and the partial sums stay below 2^63:
// |hi| <= 2^30 for a sum of two values, 3.8 2^61 for the largest set.
HGKS_FX void dot2(Half a, Half ca, Half b, Half cb, i64& hi, i64& cross)
{
    cross += (i64)a.hi * ca.lo + (i64)a.lo * ca.hi;
    hi += (i64)a.hi * ca.hi;
    cross += (i64)b.hi * cb.lo + (i64)b.lo * cb.hi;
    hi += (i64)b.hi * cb.hi;
}

HGKS_FX i64 form2(Half a, i64 ca, Half b, i64 cb)
{
    i64 hi = 0, cross = 0;
    dot2(a, halves(ca), b, halves(cb), hi, cross);
    return hi + (cross >> 31);
}

HGKS_FX i64 form3(Half c, i64 cc, Half a, i64 ca, Half b, i64 cb)
{
    const Half k = halves(cc);
    i64 hi = (i64)c.hi * k.hi, cross = (i64)c.hi * k.lo + (i64)c.lo * k.hi;
    dot2(a, halves(ca), b, halves(cb), hi, cross);
    return hi + (cross >> 31);
}

template <bool DER>
HGKS_FX bool quartic_pair(const double* q, Scale inv, double* v, double* d)
{
    i64 w[5];
    int E;
    if (!window(q, w, E) || (DER && (u32)(E + inv.e - 100) > 1900u)) return false;
    const Half c = halves(w[2]), s1 = halves(w[1] + w[3]), s2 = halves(w[0] + w[4]);
    const Half d1 = halves(w[3] - w[1]), d2 = halves(w[4] - w[0]);
    const i64 even = form3(c, 4605280898957349864ll, s1, 4270079646692026ll, s2, -1067519911673006ll);
    const i64 odd = form2(d1, 924499362554543698ll, d2, -129429910757636118ll);
    v[0] = from_fixed(even - odd, E, 58);
    v[1] = from_fixed(even + odd, E, 58);
    if (DER) {
        const i64 n = form2(d1, 3074457345618258602ll, d2, -384307168202282325ll);
        const i64 s = form3(c, -3550077552209447800ll, s1, 1922958674113450892ll, s2, -147919898008726992ll);
        d[0] = from_fixed(smulhi(halves(n - s), inv.m), E + inv.e, 56);
        d[1] = from_fixed(smulhi(halves(n + s), inv.m), E + inv.e, 56);
    }
    return true;
}

}  // namespace fixed
}  // namespace hgks
