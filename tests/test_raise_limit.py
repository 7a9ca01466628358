"""Two host threads that raise one kernel's shared-memory limit: what stands at the end is what is recorded."""

import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_08038_gb300", "csrc")

SOURCE = r"""
#include <atomic>
#include <chrono>
#include <thread>
#include "raise_limit.cuh"

// The smaller value is asked for first and takes longer to set.
int main() {
    int limit = 0, calls = 0;
    std::atomic<int> set{0};
    auto raise = [&](int want, int ms) {
        return rosar::raise_limit(&limit, want, [&, ms](int n) {
            ++calls;
            std::this_thread::sleep_for(std::chrono::milliseconds(ms));
            set = n;
            return 0;
        });
    };
    std::thread a([&] { raise(50000, 300); });
    std::this_thread::sleep_for(std::chrono::milliseconds(100));
    std::thread b([&] { raise(90000, 0); });
    a.join();
    b.join();
    if (limit != 90000 || set != limit) return 1;
    if (raise(60000, 0) != 0 || calls != 2) return 2;                                   // nothing to do
    if (rosar::raise_limit(&limit, 100000, [](int) { return 7; }) != 7 || limit != 90000) return 3;   // not recorded
    return 0;
}
"""


def test_the_recorded_limit_is_the_one_set(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
