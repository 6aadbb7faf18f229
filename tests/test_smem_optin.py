"""The bookkeeping of the kernels' shared-memory opt-in (csrc/bx_smem.h), compiled for the host with a fake of
the attribute call: once per device and size, on every device of a process, never lowered, a failure
tried again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_11125_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <vector>
#include <thread>
#include "bx_smem.h"
int main() {
    bx::SmemOptIn o;
    std::vector<std::pair<int, size_t>> calls;
    int fail = 0;
    auto need = [&](int dev, size_t n) {
        return o.ensure(dev, n, [&](size_t b) { calls.push_back({dev, b}); return fail; });
    };
    need(0, 1000); need(0, 1000); need(0, 800); need(1, 800); need(1, 1000); need(0, 1000); need(63, 5);
    fail = 7;
    printf("%d ", need(0, 2000));
    fail = 0;
    need(0, 2000); need(0, 1500); need(64, 9); need(64, 9);
    for (auto& c : calls) printf("%d:%zu ", c.first, c.second);
    bx::SmemOptIn p;
    size_t top = 0;
    std::vector<std::thread> t;
    for (int q = 0; q < 8; ++q)
        t.emplace_back([&, q] {
            for (size_t n = 1; n < 2000; ++n)
                p.ensure(3, n * (q + 1), [&](size_t b) { if (b < top) printf("lowered "); top = b; return 0; });
        });
    for (auto& x : t) x.join();
    printf("top %zu", top);
}
"""


def test_once_per_device_and_size(tmp_path):
    src, exe = tmp_path / "optin.cpp", tmp_path / "optin"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    out = subprocess.check_output([str(exe)], text=True)
    assert out == "7 0:1000 1:800 1:1000 63:5 0:2000 0:2000 64:9 64:9 top 15992"


def test_no_launcher_keeps_the_size_for_all_devices():
    """Every opt-in goes through the per-device record (the self-test, which sets it on each call, aside)."""
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        n = text.count("cudaFuncSetAttribute(")
        assert n == {"bx_internal.cuh": 1, "bx_fwd_tc.cu": 1}.get(f, 0), (f, n)
