"""Node order on several threads when none can be had: the bisection of
geometry.cu, compiled by itself with an operator new that fails from the k-th call
on, ends normally and gives the order of one thread."""
import os
import subprocess

import pytest

from paper_1709_08070_gb300 import build

MAIN = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <algorithm>
#include <exception>
#include <new>
#include <system_error>
#include <thread>
#include <vector>
static long allowed = -1;  // allocations still to succeed; -1: all
void* operator new(size_t n)
{
    if (allowed == 0) throw std::bad_alloc();
    if (allowed > 0) --allowed;
    return malloc(n);
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }
%s
int main()
{
    std::vector<RcbNode> a(100003), b;
    uint64_t s = 1;
    for (size_t i = 0; i < a.size(); ++i) {
        for (double& x : a[i].x) x = (double)((s = s * 6364136223846793005ull + 1442695040888963407ull) >> 40);
        a[i].idx = (int64_t)i;
    }
    b = a;
    rcb_split(a.data(), (int64_t)a.size(), 0);
    allowed = %d;
    rcb_split(b.data(), (int64_t)b.size(), 7);
    allowed = -1;
    for (size_t i = 0; i < a.size(); ++i)
        if (a[i].idx != b[i].idx) return 3;
    return 0;
}
"""


@pytest.mark.parametrize("allowed", [-1, 0, 1, 3])
def test_order_without_threads(tmp_path, allowed):
    with open(os.path.join(build.CSRC, "geometry.cu")) as f:
        text = f.read()
    part = text[text.index("constexpr int64_t kRcbLeaf"):text.index("// Reorders the nodes of a built geometry")]
    part = part[:part.rindex("}  // namespace")]
    src, exe = str(tmp_path / "rcb.cpp"), str(tmp_path / "rcb")
    with open(src, "w") as f:
        f.write(MAIN % (part, allowed))
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", src, "-o", exe], check=True)
    assert subprocess.run([exe], timeout=120).returncode == 0
