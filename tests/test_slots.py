"""The bounded set behind hlf_get_factor's copies (csrc/slots.h), compiled for the host:
as many threads as it has things hold one each at the same time, and the next one goes on
when one comes back."""

import subprocess

from paper_2103_00693_gb300 import build as hbuild

PROGRAM = """
#include <atomic>
#include <chrono>
#include <cstdio>
#include <set>
#include <thread>
#include <vector>
#include "slots.h"
int main()
{
    constexpr int N = 8;
    hlf::Slots<int, N> slots;
    std::set<int*> held;  // one thread: all of them, without waiting
    for (int i = 0; i < N; ++i) held.insert(slots.take());
    if (held.size() != N) return 1;
    std::atomic<bool> got{false};
    std::thread late([&] { slots.give(slots.take()); got = true; });
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    if (got) return 2;  // all are in use
    for (int* p : held) slots.give(p);
    late.join();
    std::atomic<int> in_use{0}, most{0}, bad{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 3 * N; ++t)
        ts.emplace_back([&] {
            for (int i = 0; i < 2000; ++i) {
                int* p = slots.take();
                const int u = ++in_use;
                int m = most;
                while (m < u && !most.compare_exchange_weak(m, u)) {}
                const int before = ++*p;  // nobody else has it
                std::this_thread::yield();
                bad += *p != before;
                --in_use;
                slots.give(p);
            }
        });
    for (auto& t : ts) t.join();
    return bad || most > N || most < 2 ? 3 : 0;
}
"""


def test_slots(tmp_path):
    (tmp_path / "slots.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", hbuild.CSRC, str(tmp_path / "slots.cpp"), "-o",
                    str(tmp_path / "slots")], check=True)
    assert subprocess.run([str(tmp_path / "slots")], timeout=60).returncode == 0
