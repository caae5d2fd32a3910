"""The bookkeeping of what is set once per device (the shared-memory limits of the convolution
kernels): the header compiled by the host compiler against a fake of the CUDA call."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_02245_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    pat::DeviceOnce a, b;
    std::atomic<int> calls[128] = {};
    int error = 0, device = 0;
    auto set = [&] { ++calls[device]; return error; };
    for (int rep = 0; rep < 3; ++rep)
        for (device = 0; device < 3; ++device) CHECK(a.run(device, set) == 0);
    for (int d = 0; d < 3; ++d) CHECK(calls[d] == 1);         // every device, once
    device = 1;
    CHECK(b.run(1, set) == 0 && calls[1] == 2);               // another kernel
    device = 5;
    error = 98;
    CHECK(a.run(5, set) == 98 && a.run(5, set) == 98 && calls[5] == 2);   // a failure is not kept
    error = 0;
    CHECK(a.run(5, set) == 0 && a.run(5, set) == 0 && calls[5] == 3);
    device = 100;
    CHECK(a.run(100, set) == 0 && a.run(100, set) == 0 && calls[100] == 2);   // past the table
    device = 0;
    CHECK(a.run(-1, set) == 0 && calls[0] == 2);
    pat::DeviceOnce c;
    std::atomic<int> n{0}, early{0};
    std::atomic<bool> is_set{false};
    std::vector<std::thread> ts;
    for (int i = 0; i < 16; ++i)
        ts.emplace_back([&] {
            c.run(2, [&] { ++n; std::this_thread::yield(); is_set = true; return 0; });
            if (!is_set) ++early;                             // nobody goes on before it is set
        });
    for (auto& t : ts) t.join();
    CHECK(n == 1 && early == 0);
    return 0;
}
"""


def test_every_device_is_set_once(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_convolutions_set_their_limits_per_device():
    """No launcher keeps the result of cudaFuncSetAttribute for the whole process."""
    text = open(os.path.join(CSRC, "conv.cu")).read()
    assert text.count("cudaFuncSetAttribute") == 1 and "static const cudaError_t" not in text
    assert text.count("raise_smem(once,") == 5
