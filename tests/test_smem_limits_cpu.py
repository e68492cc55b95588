"""The record of the kernels' shared-memory limits (SmemLimits): a limit set on one
device says nothing about another, it only grows, and a refused one is not recorded."""
import subprocess

from paper_2105_06055_gb300 import build

SRC = """
#include <cstdio>
#include "pd_smem_limit.cuh"
int main()
{
    pd::SmemLimits l;
    int calls = 0, f = 0, g = 0;
    auto ok = [&]() { return ++calls, 0; };
    auto bad = [&]() { return ++calls, 7; };
    auto show = [&](int e) { std::printf("%d %d\\n", e, calls); };
    show(l.raise(0, &f, 60000, ok));   // set
    show(l.raise(0, &f, 50000, ok));   // below the limit
    show(l.raise(1, &f, 60000, ok));   // the same kernel on another device
    show(l.raise(1, &g, 60000, ok));   // another kernel
    show(l.raise(0, &f, 70000, bad));  // refused
    show(l.raise(0, &f, 70000, ok));   // not recorded: set now
    show(l.raise(0, &f, 70000, ok));
    return 0;
}
"""


def test_limits_are_kept_by_device_and_kernel(tmp_path):
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-I", build.CSRC, "-o", str(exe), str(src), "-pthread"])
    got = [tuple(map(int, r.split())) for r in subprocess.check_output([str(exe)], text=True).splitlines()]
    assert got == [(0, 1), (0, 1), (0, 2), (0, 3), (7, 4), (0, 5), (0, 5)]
