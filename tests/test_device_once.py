"""Set-up that is made once per device (function attributes, loading of kernels): csrc/device_once.h, compiled for the host."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2510_15312_b200", "csrc")

PROGRAM = r"""
#include "device_once.h"
#include <cstdio>
#include <thread>
#include <vector>
static sdv::DeviceOnce once;
int main() {
    int runs[80] = {0};
    auto ok = [&](int d) { return once.run(d, [&]() { ++runs[d]; return 0; }); };
    // every device has its own set-up, and only one
    for (int d : {0, 1, 0, 1, 63, 63}) if (ok(d)) return 1;
    if (runs[0] != 1 || runs[1] != 1 || runs[63] != 1) return 2;
    // past the mask: every time
    ok(64); ok(64);
    if (runs[64] != 2) return 3;
    // a failure is handed back and tried again
    int tries = 0;
    auto twice = [&]() { return ++tries < 2 ? 7 : 0; };
    if (once.run(2, twice) != 7 || once.run(2, twice) != 0 || once.run(2, twice) != 0 || tries != 2) return 4;
    // threads on several devices: whoever returns finds its device set up
    sdv::DeviceOnce shared;
    std::atomic<int> ready[8] = {};
    std::atomic<int> bad{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 16; ++t)
        ts.emplace_back([&, t]() {
            for (int i = 0; i < 2000; ++i) {
                const int d = (t + i) % 8;
                if (shared.run(d, [&]() { ready[d].store(1, std::memory_order_relaxed); return 0; })) ++bad;
                if (!ready[d].load(std::memory_order_relaxed)) ++bad;
            }
        });
    for (auto& t : ts) t.join();
    return bad ? 5 : 0;
}
"""


def test_set_up_runs_once_per_device_and_again_after_a_failure(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


@pytest.mark.parametrize("name", ["cudaFuncSetAttribute", "cudaFuncGetAttributes"])
def test_every_function_attribute_is_set_up_per_device(name):
    """No flag of its own beside a call whose effect belongs to one device."""
    with open(os.path.join(CSRC, "sdv.cu")) as fh:
        text = fh.read()
    assert name in text and "static bool" not in text and "std::atomic<bool>" not in text
