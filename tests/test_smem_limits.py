"""The dynamic shared-memory limits remembered per device and kernel (the CUDA
attribute is per device): a second device is raised on its own, smaller plans
leave a limit alone, and a refused raise is reported and tried again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "bd_smem.h"
struct Call { const void* fn; size_t bytes; };
int main()
{
    bd::SmemLimits l;
    std::vector<Call> calls;
    int answer = 0;
    auto set = [&](const void* f, size_t b) { calls.push_back({f, b}); return answer; };
    int k1 = 0, k2 = 0, bad = 0;
    auto expect = [&](int dev, const void* f, size_t b, int result, size_t n_calls) {
        const int r = l.raise(dev, f, b, 0, set);
        if (r != result || calls.size() != n_calls) {
            std::printf("device %d, %zu bytes: result %d, %zu calls (expected %d, %zu)\n", dev, b, r, calls.size(), result, n_calls);
            ++bad;
        }
    };
    expect(0, &k1, 50000, 0, 1);   // first use on device 0
    expect(0, &k1, 50000, 0, 1);
    expect(0, &k1, 20000, 0, 1);   // a smaller plan: the limit stays
    expect(0, &k2, 20000, 0, 2);   // another kernel
    expect(1, &k1, 50000, 0, 3);   // the same kernel on another device
    expect(1, &k1, 60000, 0, 4);
    expect(0, &k1, 60000, 0, 5);
    answer = 7;
    expect(0, &k1, 90000, 7, 6);   // refused: reported, not remembered
    answer = 0;
    expect(0, &k1, 60000, 0, 6);
    expect(0, &k1, 90000, 0, 7);
    return bad;
}
"""


def test_limits_are_kept_per_device_and_kernel(tmp_path):
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_2411_00991_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", inc, str(src), "-o", str(exe), "-pthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_limit_is_raised_through_the_one_place():
    csrc = os.path.join(ROOT, "paper_2411_00991_gb300", "csrc")
    uses = [f for f in os.listdir(csrc)
            for line in open(os.path.join(csrc, f)) if "cudaFuncSetAttribute(" in line]
    assert uses == ["bd_internal.h"]
