"""The fixed-point reciprocal and reciprocal square root (csrc/hgks_fixed.cuh) with starting values as
far off as the device's single-precision approximations may be, on either side: one unit in the last
place for rcp.approx.ftz.f32, 2^-22.9 relative for rsqrt.approx.ftz.f32.  The mantissa's ends are where
it matters: the exact value lies one rounding above 1/2 there, so a seed may lie below 1/2.

Bounds as with correctly rounded seeds: the third-order remainder (2^-22.9 + 2^-24)^3 stays below 2^-66,
so a result is within one rounding and 2^-9 of a unit, and quotients and roots are IEEE's bits."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_05572_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
static int side;                       // -1, 0, +1: seeds low, correctly rounded, high
#define HGKS_FX_OWN_SEEDS
namespace hgks { namespace fixed {
inline float approx_rcp(float x)
{
    const float r = (float)(1.0L / x);
    return side < 0 ? std::nextafter(r, 0.0f) : side > 0 ? std::nextafter(r, 4.0f) : r;
}
inline float approx_rsqrt(float x)
{
    const long double r = 1.0L / std::sqrt((long double)x), d = side * std::exp2(-22.9L) * r;
    float f = (float)(r + d);          // the float next to the error bound that does not exceed it
    while (std::fabs((long double)f - r) > std::fabs(d) && side) f = std::nextafter(f, side < 0 ? 4.0f : 0.0f);
    return f;
}
} }
#include "hgks_fixed.cuh"
using namespace hgks::fixed;
static double ulps(double a, long double r)
{
    int e; std::frexp((double)r, &e);
    return (double)(std::fabs((long double)a - r) / std::ldexp(1.0L, e - 53));
}
int main(int argc, char** argv)
{
    side = std::atoi(argv[1]);
    std::mt19937_64 g(7);
    double worst = 0.0;
    long wrong = 0;
    for (long i = 0; i < 300000; i++) {
        // the ends of the leading 23 bits, their neighbourhoods, and random mantissas; both parities
        u64 m = i < 100000 ? (u64)(i / 4) << 29 : g() >> 12;
        if (i & 1) m = ~m;
        if (i % 16 == 2) m |= (1ull << 29) - 1;
        const double x = of_bits(((u64)(1023 - ((i >> 1) & 1)) << 52) | (m & 0xFFFFFFFFFFFFFull)), y = of_bits((1023ull << 52) | (g() >> 12));
        double q = 0.0;
        worst = std::fmax(worst, std::fmax(ulps(rcp(x), 1.0L / x), ulps(rsqrt(x), 1.0L / std::sqrt((long double)x))));
        wrong += !div_rn(y, x, q) || bits_of(q) != bits_of(y / x);
        wrong += !sqrt_rn(x, q) || bits_of(q) != bits_of(std::sqrt(x));
    }
    std::printf("%.6f %ld\n", worst, wrong);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("seeds")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("side", [-1, 0, 1])
def test_seeds_at_the_approximations_error_bounds(exe, side):
    worst, wrong = subprocess.run([exe, str(side)], check=True, capture_output=True, text=True).stdout.split()
    assert float(worst) <= 0.51 and wrong == "0", (worst, wrong)
