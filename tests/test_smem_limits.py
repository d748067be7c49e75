"""A kernel's shared-memory limit is raised once per device, not once per process.

The bookkeeping is host code: it is compiled with the C++ compiler and run against a fake
of the attribute call, with two devices, growing sizes, a failing call and threads.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cassert>
#include <stdexcept>
#include <thread>
#include <vector>
#include "smem_limits.h"

int main() {
    kpcg::SmemLimits limits;
    size_t attr[2][2] = {};  // [device][kernel]: what the runtime was told
    int calls = 0, kernels[2];
    auto allow = [&](int dev, int k, size_t bytes) {
        limits.allow(dev, &kernels[k], bytes, [&] { ++calls; attr[dev][k] = bytes; });
        assert(attr[dev][k] >= bytes);
    };
    allow(0, 0, 100000);
    allow(0, 0, 100000);
    assert(calls == 1);
    allow(1, 0, 100000);  // the same kernel on another device
    allow(0, 1, 50000);   // another kernel
    assert(calls == 3);
    allow(0, 0, 200000);
    allow(0, 0, 60000);   // a smaller launch keeps the higher limit
    assert(calls == 4 && attr[0][0] == 200000 && attr[1][0] == 100000);
    bool threw = false;
    try {
        limits.allow(1, &kernels[1], 70000, [] { throw std::runtime_error("refused"); });
    } catch (const std::runtime_error&) {
        threw = true;
    }
    assert(threw);
    allow(1, 1, 70000);   // tried again after a failure
    assert(calls == 5 && attr[1][1] == 70000);
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 1000; ++i)
                limits.allow(t & 1, &kernels[i & 1], 70000 + i, [&] { attr[t & 1][i & 1] = 70000 + i; });
        });
    for (auto& t : ts) t.join();
    assert(attr[0][0] == 200000 && attr[1][0] == 100000 && attr[0][1] == 70999 && attr[1][1] == 70999);
    return 0;
}
"""


def test_per_device(tmp_path):
    src = tmp_path / "limits.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "limits")
    inc = os.path.join(ROOT, "paper_1602_06693_gb300", "csrc")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-UNDEBUG", "-I", inc, str(src), "-o", exe])
    subprocess.check_call([exe], timeout=60)


def test_every_limit_goes_through_it():
    """No kernel keeps a flag of its own for the whole process."""
    csrc = os.path.join(ROOT, "paper_1602_06693_gb300", "csrc")
    users = [f for f in sorted(os.listdir(csrc)) if "cudaFuncSetAttribute" in
             open(os.path.join(csrc, f)).read()]
    assert users == ["api.cu"]
