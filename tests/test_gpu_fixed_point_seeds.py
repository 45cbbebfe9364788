"""The fixed-point reciprocal, root, quotient and square root (csrc/hgks_fixed.cuh) on the device, from the
hardware's own single-precision approximations: every leading mantissa pattern the approximations see (2^23
for the reciprocal, both parities for the root) with the remaining bits at 0, at 1 and hashed, and
numerators and radicands next to a product, where a quotient or root lies next to a double or next to
the middle between two.  Quotients and roots are IEEE's bits; the reciprocal is within 1 unit in the
last place of IEEE's, the reciprocal root within 2 of the IEEE reciprocal of the IEEE root."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include "hgks_fixed.cuh"
namespace fx = hgks::fixed;
typedef fx::u64 u64;
__device__ u64 hash(u64 z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ u64 apart(double a, double b) { const u64 x = fx::bits_of(a), y = fx::bits_of(b); return x > y ? x - y : y - x; }
// out: largest distance of rcp, of rsqrt; wrong quotients, wrong roots
__global__ void check(unsigned long long* out)
{
    const u64 lead = (u64)blockIdx.x * blockDim.x + threadIdx.x;           // 2^23 threads
    for (int low = 0; low < 3; low++)
        for (int odd = 0; odd < 2; odd++) {
            const u64 h = hash(lead * 6 + low * 2 + odd);
            const u64 tail = low == 0 ? 0u : low == 1 ? (1u << 29) - 1 : h & ((1u << 29) - 1);
            const double x = fx::of_bits(((u64)(1023 - odd) << 52) | (lead << 29) | tail);
            const double y = fx::of_bits((1023ull << 52) | (h >> 12));
            atomicMax(out, apart(fx::rcp(x), __drcp_rn(x)));
            atomicMax(out + 1, apart(fx::rsqrt(x), __drcp_rn(__dsqrt_rn(x))));
            const double near = fx::of_bits(fx::bits_of(__dmul_rn(x, y)) + h % 3 - 1), square = fx::of_bits(fx::bits_of(__dmul_rn(x, x)) + h % 3 - 1);
            double q = 0.0;
            unsigned wq = !fx::div_rn(y, x, q) || fx::bits_of(q) != fx::bits_of(__ddiv_rn(y, x));
            wq += !fx::div_rn(near, x, q) || fx::bits_of(q) != fx::bits_of(__ddiv_rn(near, x));
            unsigned wr = !fx::sqrt_rn(x, q) || fx::bits_of(q) != fx::bits_of(__dsqrt_rn(x));
            wr += !fx::sqrt_rn(square, q) || fx::bits_of(q) != fx::bits_of(__dsqrt_rn(square));
            if (wq) atomicAdd(out + 2, (unsigned long long)wq);
            if (wr) atomicAdd(out + 3, (unsigned long long)wr);
        }
}
int main()
{
    unsigned long long *d, h[4];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
    check<<<1 << 15, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu %llu %llu\n", h[0], h[1], h[2], h[3]);
    return 0;
}
"""


def test_every_leading_pattern(tmp_path):
    from paper_2304_05572_gb300 import _build
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run([_build._nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-I", _build.CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    r, s, wq, wr = (int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert r <= 1 and s <= 2 and wq == 0 and wr == 0, (r, s, wq, wr)
