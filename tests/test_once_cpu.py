"""The helper that sets a kernel's attributes once per device: a second device gets its own call, a failed one is
tried again, threads may race for the first."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <thread>
#include <vector>
#include "lbe_once.h"
int main() {
    static lbe::PerDevice once;
    int calls = 0;
    auto run = [&](int dev, int status) { return once(dev, [&] { ++calls; return status; }); };
    if (run(0, 0) != 0 || run(0, 7) != 0 || calls != 1) return 1;  // done once
    if (run(1, 5) != 5 || calls != 2) return 2;                    // another device, and its failure comes back
    if (run(1, 0) != 0 || run(1, 0) != 0 || calls != 3) return 3;  // tried again, then done
    if (run(64, 0) != 0 || run(64, 0) != 0 || calls != 5) return 4;  // beyond the mask: every time
    static lbe::PerDevice many;
    std::atomic<int> ran{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] { for (int i = 0; i < 1000; ++i) many(k % 4, [&] { ran++; return 0; }); });
    for (auto &x : t) x.join();
    return ran >= 4 && ran <= 8 ? 0 : 5;
}
"""


def test_once_per_device(tmp_path):
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "once")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_1202_3842_gb300", "csrc"),
                    str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
