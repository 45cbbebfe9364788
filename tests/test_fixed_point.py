"""The fixed-point reciprocal, reciprocal square root, exponential and erfc of the flux kernel
(csrc/hgks_fixed.cuh), compiled for the host, against long-double references.

Bounds in units of the result's last place: one rounding (1/2), the approximations' own remainders
(2^-9 for the two reciprocals; for the exponential 2^-5 for the argument's 57 fraction bits and
2^-4 for series and truncations, bounded here by 1/4), and for erfc the table's 2.1e-16 (up to 1.9
units) beside the exponential's.  The Gauss-point quartic (quartic_pair) loses, beside its rounding,
at most 1.5 2^-60 by the window's truncation and 1.5 2^-58 per product and set (values: 5 products, 2
sets; derivatives the same and 3 2^-56 for the factor 1/h) of the window's largest value: within
2^-54 and 2^-53."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_05572_gb300", "csrc")

SRC = r"""
#include "hgks_fixed.cuh"
#include <cfloat>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <random>
using namespace hgks::fixed;
static double ulps(double a, long double r)
{
    int e; std::frexp((double)r, &e);
    return (double)(std::fabs((long double)a - r) / std::ldexp(1.0L, e - 53));
}
int main(int argc, char** argv)
{
    const char* what = argv[1];
    std::mt19937_64 g(20230415);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    double worst = 0.0;
    if (!strcmp(what, "quartic")) {
        // error beyond one rounding, relative to the window's largest value (and 1/h): values, derivatives
        const long double r3 = std::sqrt(3.0L);
        double wv = 0.0, wd = 0.0;
        bool ok = true;
        for (long i = 0; i < 200000; i++) {
            double q[5], v[2], d[2], mx = 0.0;
            const double base = i & 1 ? 6.0 * U(g) - 3.0 : 0.0, amp = i & 1 ? std::exp(-U(g) * 40.0) : 1.0;
            const double sc = std::ldexp(1.0, (int)(U(g) * 600.0) - 300), inv = std::exp(40.0 * U(g) - 20.0);
            for (double& x : q) x = sc * (base + amp * (2.0 * U(g) - 1.0) * (i & 4 ? std::exp(-U(g) * 20.0) : 1.0));
            if (i % 50 == 0) for (int j = 1; j < 5; j++) q[j] = q[0];
            if (i % 50 == 1) { q[0] = q[1] = 0.0; q[3] = -q[3]; }
            for (double x : q) mx = std::fmax(mx, std::fabs(x));
            ok = ok && quartic_pair<true>(q, scale_of(inv), v, d);
            double u[2];
            ok = ok && quartic_pair<false>(q, scale_of(inv), u, nullptr) && u[0] == v[0] && u[1] == v[1];
            if (i % 50 == 0) ok = ok && v[0] == q[0] && v[1] == q[0];
            for (int k = 0; k < 2; k++) {
                const long double s = k ? r3 : -r3;
                const long double c[5] = {-1 / 4320.0L + 7 * s / 432, 1 / 1080.0L - 25 * s / 216, 719 / 720.0L,
                                          1 / 1080.0L + 25 * s / 216, -1 / 4320.0L - 7 * s / 432};
                const long double e[5] = {1 / 12.0L - s / 54, -2 / 3.0L + 13 * s / 54, -4 * s / 9, 2 / 3.0L + 13 * s / 54, -1 / 12.0L - s / 54};
                long double a = 0, b = 0;
                for (int j = 0; j < 5; j++) { a += c[j] * q[j]; b += e[j] * q[j]; }
                b *= inv;
                wv = std::fmax(wv, (double)((std::fabs(v[k] - a) - std::fabs(a) * 0x1p-53L) / mx));
                wd = std::fmax(wd, (double)((std::fabs(d[k] - b) - std::fabs(b) * 0x1p-53L) / (mx * (long double)inv)));
            }
        }
        double z[5] = {0.0, -0.0, 0.0, 0.0, 0.0}, v[2], d[2];
        ok = ok && quartic_pair<true>(z, scale_of(3.0), v, d) && v[0] == 0 && v[1] == 0 && d[0] == 0 && d[1] == 0;
        for (double bad : {std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN(), 1e-280, 1e280}) {
            z[1] = bad;
            ok = ok && !quartic_pair<true>(z, scale_of(3.0), v, d);
        }
        printf("%d %.6f %.6f\n", ok ? 1 : 0, std::ldexp(wv, 54), std::ldexp(wd, 53));
        return 0;
    }
    if (!strcmp(what, "ieee")) {
        // quotients and roots: the host's bits on random operands, on short mantissas and on operands made
        // so that the result lies next to the middle between two doubles
        long wrong = 0, taken = 0, n = 400000;
        for (long i = 0; i < n; i++) {
            auto draw = [&](bool wide) {
                u64 m = g() & 0xFFFFFFFFFFFFFull, e = wide ? 1 + g() % 2046 : 900 + g() % 200;
                const int sh = (int)(g() % 53);
                if (i % 4 == 1) m &= ~((1ull << sh) - 1);
                if (i % 4 == 2) m |= (1ull << sh) - 1;
                return of_bits((g() & 0x8000000000000000ull) | (e << 52) | m);
            };
            double a = draw(i & 1), b = draw(i & 1), q;
            if (i % 5 == 0) a = of_bits(bits_of(b * draw(false)) + g() % 3 - 1);
            if (i % 1000 == 0) a = std::copysign(0.0, a);
            if (div_rn(a, b, q)) { taken++; wrong += bits_of(q) != bits_of(a / b); }
            double x = std::fabs(draw(i & 1));
            if (i % 3 == 0) { const double y = draw(false); x = of_bits(bits_of(y * y) + g() % 3 - 1); }
            if (sqrt_rn(x, q)) wrong += bits_of(q) != bits_of(std::sqrt(x));
        }
        const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
        double q;
        for (double v : {0.0, -0.0, 1e-310, inf, nan}) wrong += div_rn(1.0, v, q) + sqrt_rn(v, q) + (v == 0.0 ? 0 : div_rn(v, 1.0, q));
        wrong += sqrt_rn(-1.0, q) + div_rn(1e300, 1e-300, q) + div_rn(1e-300, 1e300, q) + div_rn(1e-200, 1e108, q);
        printf("%ld %d\n", wrong, taken > n / 2 ? 1 : 0);
        return 0;
    }
    if (!strcmp(what, "physical")) {
        // never true for a state that is not physical; true from 1e-5 of rho E on
        long wrong = 0, missed = 0, yes = 0;
        for (long i = 0; i < 400000; i++) {
            const double rho = std::exp(40.0 * U(g) - 20.0), u = 2000.0 * (U(g) - 0.5), v = i & 1 ? 2000.0 * (U(g) - 0.5) : 0.0;
            const double rel = (i % 3 ? 1.0 : -1.0) * std::exp(-U(g) * 25.0), ke = 0.5 * rho * (u * u + v * v);
            const double E = ke / (1.0 - (rel < 0.9 ? rel : 0.9));
            const long double pr = (long double)E * rho - 0.5L * ((long double)(rho * u) * (rho * u) + (long double)(rho * v) * (rho * v));
            const bool s = surely_physical(to_float(rho), to_float(rho * u), to_float(rho * v), to_float(E));
            wrong += s && !(pr > 0);
            yes += s;
            missed += !s && rel > 1e-5 && E < 1e12 && E > 1e-12 && rho > 1e-12 && rho < 1e12;
        }
        for (double bad : {0.0, -1.0, std::numeric_limits<double>::infinity(), std::numeric_limits<double>::quiet_NaN(), 1e-320, 1e300})
            wrong += surely_physical(to_float(bad), 0.0f, 0.0f, 1.0f) + surely_physical(1.0f, 0.0f, 0.0f, to_float(bad))
                   + (std::isfinite(bad) && std::fabs(bad) < 1.4 ? 0 : surely_physical(1.0f, to_float(bad), 0.0f, 1.0f));
        printf("%ld %d\n", wrong + missed, yes > 100000 ? 1 : 0);
        return 0;
    }
    if (!strcmp(what, "special")) {
        const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
        bool ok = true;
        for (double v : {0.0, -0.0, 1e-310, -1e-310, inf, -inf, nan}) ok = ok && std::isnan(rcp(v));
        ok = ok && rcp(std::ldexp(1.3, 1022)) == 0.0 && rcp(std::ldexp(-1.0, 1023)) == 0.0;
        for (double v : {0.0, -0.0, 1e-310, -1.0, -inf, inf, nan}) ok = ok && std::isnan(rsqrt(v));
        for (double v : {0.0, -0.0, 3.0, -1e200, inf, -inf, 1e-300}) ok = ok && scale2<1>(v) == 2 * v && scale2<-1>(v) == 0.5 * v;
        ok = ok && std::isnan(scale2<1>(nan)) && rcp(1.0) == 1.0 && rcp(-2.0) == -0.5 && rsqrt(4.0) == 0.5 && rsqrt(1.0) == 1.0;
        ok = ok && exp_value(exp_neg(0.0)) == 1.0 && rcp(std::ldexp(1.0, 1021)) == std::ldexp(1.0, -1021) && rcp(std::ldexp(1.0, -1022)) == std::ldexp(1.0, 1022);
        printf("%d\n", ok ? 1 : 0);
        return 0;
    }
    for (long i = 0; i < 400000; i++) {
        // edges of the ranges, neighbours of powers of two, log-uniform and uniform arguments
        double x = std::exp((U(g) - 0.5) * 1300.0), y = i & 1 ? U(g) : std::exp(-U(g) * 40.0);
        if (i < 4000) { x = std::ldexp(1.0 + (i / 4) * DBL_EPSILON, (i & 3) - 1); if (i & 2) x = std::nextafter(x, 0.0); }
        if (!strcmp(what, "rcp")) worst = std::fmax(worst, std::fmax(ulps(rcp(x), 1.0L / x), ulps(-rcp(-x), 1.0L / x)));
        if (!strcmp(what, "rsqrt")) worst = std::fmax(worst, ulps(rsqrt(x), 1.0L / std::sqrt((long double)x)));
        if (!strcmp(what, "exp")) {
            double a = i % 3 ? y * 64.0 : 64.0 + U(g) * (708.0 - 64.0);
            if (i == 0) a = 64.0;
            if (i == 1) a = std::nextafter(64.0, 0.0);
            if (i == 2) a = std::nextafter(708.0, 0.0);
            worst = std::fmax(worst, ulps(exp_value(exp_neg(a)), std::exp(-(long double)a)));
        }
        if (!strcmp(what, "erfc")) {
            double a = y * 8.0, a2, ex, er;
            if (i < 96) { a = (i / 3) / 4.0 + (i % 3 == 1 ? 0.125 : 0.0); if (i % 3 == 2) a = std::nextafter(a, 8.0); }
            if (i == 96) a = std::nextafter(8.0, 0.0);
            a2 = a * a;
            if (!(a2 < 64.0)) continue;
            exp_erfc(a, a2, ex, er);
            // the exponential is taken of the rounded square
            const long double ref = std::erfc((long double)a) * std::exp((long double)a * a - (long double)a2);
            worst = std::fmax(worst, ulps(er, ref));
        }
    }
    printf("%.6f\n", worst);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("what,bound", [("rcp", 0.51), ("rsqrt", 0.51), ("exp", 0.75), ("erfc", 2.7)])
def test_within_bounds(exe, what, bound):
    worst = float(subprocess.run([exe, what], check=True, capture_output=True, text=True).stdout)
    assert worst <= bound, worst


def test_special_arguments(exe):
    assert subprocess.run([exe, "special"], check=True, capture_output=True, text=True).stdout.strip() == "1"


def test_gauss_point_quartic(exe):
    ok, wv, wd = subprocess.run([exe, "quartic"], check=True, capture_output=True, text=True).stdout.split()
    assert ok == "1" and float(wv) <= 1.0 and float(wd) <= 1.0, (ok, wv, wd)


@pytest.mark.parametrize("what", ["ieee", "physical"])
def test_exact_decisions(exe, what):
    """IEEE quotients and roots bit for bit; the FP32 positivity test against the exact sign."""
    assert subprocess.run([exe, what], check=True, capture_output=True, text=True).stdout.split() == ["0", "1"]
