"""per_device.h, the once-per-device set-up of kernel attributes: called once
for each device, from any thread, every caller given that device's result (a
once-per-process flag gave a second device nothing)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1606_00545_gb300", "csrc")

PROGRAM = r'''
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main()
{
    static hec::PerDevice<int> once;
    std::atomic<int> calls[70] = {};
    std::atomic<int> wrong{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&]() {
            for (int dev = 0; dev < 70; ++dev)
                if (once.get(dev, [&]() { ++calls[dev]; return 100 + dev; }) != 100 + dev)
                    ++wrong;
        });
    for (auto &t : ts)
        t.join();
    for (int dev = 0; dev < 64; ++dev)
        wrong += calls[dev] != 1;
    for (int dev = 64; dev < 70; ++dev) // past the slots: every call
        wrong += calls[dev] != 8;
    std::printf("wrong %d\n", wrong.load());
    return wrong.load() != 0;
}
'''


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "wrong 0\n", r.stdout
