"""The table of numbers that are looked up once per device, asked by several threads at once (host only)."""
import os
import subprocess

from conftest import ROOT

# A query that answers slowly and, as a launch's does, changes a number after it was first written: no caller may see
# the first version, and the query runs once per device.
PROGRAM = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "w2a8_table.h"
int main() {
    int bad = 0;
    for (int round = 0; round < 20; ++round) {
        w2a8::PerDeviceTable<9> table;
        std::atomic<int> asked{0}, wrong{0}, ready{0};
        std::vector<std::thread> threads;
        for (int t = 0; t < 16; ++t)
            threads.emplace_back([&, t] {
                const int dev = t % 2;
                ++ready;
                while (ready < 16) {}
                const int *row = table.get(dev, [&](int *n) {
                    ++asked;
                    for (int c = 1; c <= 8; c *= 2) n[c] = (148 - dev) / c;
                    std::this_thread::sleep_for(std::chrono::milliseconds(1));
                    n[8] = n[8] * 3 / 4;
                });
                if (row[8] != (148 - dev) / 8 * 3 / 4 || row[1] != 148 - dev) ++wrong;
            });
        for (auto &th : threads) th.join();
        bad += wrong != 0 || asked != 2;
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_threads_get_one_answer_per_device(tmp_path):
    src, exe = tmp_path / "table.cpp", tmp_path / "table"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", os.path.join(ROOT, "paper_2508_06753_b200", "csrc"),
                    "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
