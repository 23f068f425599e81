"""The limits that the library raises for its kernels (shared memory per block) only grow, whichever threads
ask at once, and a refused request is not taken for a granted one (plain host code, compiled here)."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_09160_gb300", "csrc")
PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "wmcd_limits.h"
int main() {
    using namespace std::chrono_literals;
    wmcd::RaisedLimit limit;
    std::atomic<int> attribute{0}, calls{0};
    // a low request that is slow to take effect, and a high one that comes meanwhile
    std::thread low([&] { limit.raise(100, [&](int b) { calls++; std::this_thread::sleep_for(200ms); attribute = b; return true; }); });
    std::this_thread::sleep_for(50ms);
    std::thread high([&] { limit.raise(200, [&](int b) { calls++; attribute = b; return true; }); });
    low.join();
    high.join();
    if (attribute != 200 || calls != 2) { std::printf("a lower request undid a higher one: %d\n", (int)attribute); return 1; }
    if (!limit.raise(150, [&](int) { calls++; return true; }) || calls != 2) { std::printf("raised again\n"); return 1; }
    // refused: asked again the next time, and lower ones stay granted
    for (int k = 0; k < 2; k++)
        if (limit.raise(300, [&](int) { calls++; return false; })) { std::printf("refused request granted\n"); return 1; }
    return calls == 4 && limit.raise(200, [&](int) { return false; }) ? 0 : 1;
}
"""


def test_limits_only_grow(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", exe, str(tmp_path / "t.cpp")])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
