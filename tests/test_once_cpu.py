"""The once-per-device values of csrc/dir_once.h, asked for by many threads at
once: one of them fills the value, the others wait and get that one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "dir_once.h"

struct Value { int n[4]; };

int main() {
    constexpr int kThreads = 16;
    static dirk::OncePerDevice<Value, 3> table;
    std::atomic<int> fills{0}, wrong{0}, ready{0};
    for (int dev = 0; dev < 3; ++dev) {
        fills = ready = 0;
        std::vector<std::thread> threads;
        for (int k = 0; k < kThreads; ++k)
            threads.emplace_back([&, dev] {
                ++ready;
                while (ready < kThreads) std::this_thread::yield();
                const Value* v = table.get(dev, [&](Value& w) {
                    const int call = ++fills;  // a second filling would write other values
                    std::this_thread::sleep_for(std::chrono::milliseconds(20));
                    for (int& n : w.n) n = 10 * dev + call;
                });
                for (int n : v->n) wrong += n != 10 * dev + 1;
            });
        for (std::thread& t : threads) t.join();
        if (fills != 1) return 1;
    }
    if (wrong != 0) return 2;
    auto none = [](Value&) {};
    return table.get(-1, none) || table.get(3, none) ? 3 : 0;
}
"""


def test_filled_once_however_many_ask(tmp_path):
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "once"
    inc = os.path.join(ROOT, "paper_0909_0928_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", inc, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
