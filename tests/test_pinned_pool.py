"""The staging kept for reads: bounded, shared by threads, given back with the
last context (counted through a fake allocator, no device needed)."""
import shutil
import subprocess

import pytest

from paper_1808_00270_gb300 import build as B

SRC = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include "pinned_pool.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d\n", __LINE__); return 1; } } while (0)
using namespace gld;
static std::atomic<int> live{0}, made{0};
static bool refuse = false;
int main() {
    PinnedPool pool([](size_t n) { if (refuse) return (void*)nullptr; ++live; ++made; return std::malloc(n); },
                    [](void* p) { --live; std::free(p); }, 1 << 20);
    pool.enter();
    Pinned a = pool.take(100000);
    pool.give(a);
    Pinned b = pool.take(90000);  // the same buffer again
    CHECK(b.p == a.p && made == 1);
    Pinned big = pool.take(2 << 20);
    pool.give(big);               // past the bound: freed at once
    CHECK(live == 1);
    refuse = true;
    CHECK(!pool.take(3 << 20).p);  // no room: an empty buffer
    refuse = false;
    pool.enter();
    pool.give(b);
    pool.leave();
    CHECK(live == 1);  // one context left
    pool.leave();
    CHECK(live == 0);  // none
    std::thread t[4];
    for (auto& x : t)
        x = std::thread([&] {
            for (int k = 0; k < 2000; ++k) {
                pool.enter();
                Pinned p = pool.take(1000 + 70000 * (k % 5)), q = pool.take(10);
                p.p[0] = q.p[0] = 1;
                pool.give(p);
                pool.give(q);
                pool.leave();
            }
        });
    for (auto& x : t) x.join();
    CHECK(live == 0);
    std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no C++ compiler")
def test_pool(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", B.CSRC, str(src), "-o", str(exe), "-lpthread"],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
