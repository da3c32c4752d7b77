"""The idle-block totals (csrc/kc_idle.h) on the CPU: a device's share is its own,
and threads that reserve at the same time never pass it."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_03254_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <thread>
#include <vector>

#include "kc_idle.h"

int main() {
    static kcapi::IdleTotals t;
    if (!t.reserve(0, 90, 100)) return std::puts("device 0 refused"), 1;
    if (t.reserve(0, 20, 100)) return std::puts("device 0 over its share"), 1;
    if (!t.reserve(1, 90, 100)) return std::puts("device 1 charged for device 0's blocks"), 1;
    t.release(0, 90);
    if (t.held(0) != 0 || t.held(1) != 90) return std::puts("wrong totals"), 1;
    // what the threads have counted together, each thread's own part of it: never above the limit
    constexpr size_t kLimit = 1000;
    std::atomic<size_t> mine{0}, worst{0};
    std::vector<std::thread> pool;
    for (int i = 0; i < 8; ++i)
        pool.emplace_back([&, i] {
            for (int r = 0; r < 200000; ++r) {
                const size_t n = 1 + (r * 37 + i * 11) % 400;
                if (!t.reserve(2, n, kLimit)) continue;
                const size_t now = mine.fetch_add(n) + n;
                for (size_t w = worst.load(); w < now && !worst.compare_exchange_weak(w, now);) {}
                mine.fetch_sub(n);
                t.release(2, n);
            }
        });
    for (auto& th : pool) th.join();
    if (worst.load() > kLimit || t.held(2) != 0) return std::printf("%zu of %zu\n", worst.load(), kLimit), 1;
    return 0;
}
"""


def test_idle_totals(tmp_path):
    src, exe = tmp_path / "idle.cpp", tmp_path / "idle"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
