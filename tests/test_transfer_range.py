"""Which device buffers the state transfers' kernels may touch (csrc/hgks_internal.h, compiled for the host): only
those that lie in one allocation whole.  A buffer that reaches past its allocation's end, or whose end
wraps around, goes to the runtime's copies, which judge it as they always did."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_05572_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include "hgks_internal.h"
int main(int, char** argv)
{
    unsigned long long v[4];
    for (int k = 0; k < 4; k++) std::sscanf(argv[1 + k], "%llu", v + k);
    std::printf("%d\n", hgks::inside_allocation(v[0], v[1], v[2], v[3]) ? 1 : 0);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_2304_05572_gb300 import _build
    d = tmp_path_factory.mktemp("range")
    (d / "t.cpp").write_text(SRC)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc()))), "include")
    subprocess.run(["g++", "-std=gnu++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda, "-o", str(d / "t"),
                    str(d / "t.cpp")], check=True)
    return str(d / "t")


BASE, TOP = 0x7F0000000000, 2 ** 64 - 1


@pytest.mark.parametrize("base,size,p,n,inside", [
    (BASE, 4096, BASE, 4096, 1), (BASE, 4096, BASE + 1024, 3072, 1), (BASE, 4096, BASE, 8, 1),
    (BASE, 4096, BASE, 4104, 0), (BASE, 4096, BASE + 1032, 3072, 0), (BASE, 4096, BASE + 4096, 8, 0),
    (BASE, 4096, BASE - 8, 8, 0), (BASE, 4096, BASE + 8, TOP - BASE, 0), (BASE, 4096, BASE + 8, TOP, 0)])
def test_inside_allocation(exe, base, size, p, n, inside):
    out = subprocess.run([exe] + [str(x) for x in (base, size, p, n)], check=True, capture_output=True, text=True).stdout
    assert out.strip() == str(inside)
