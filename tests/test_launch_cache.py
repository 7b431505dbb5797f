"""What the host keeps about a kernel between launches (csrc/launch_cache.h), compiled with the host C++ compiler against a
fake runtime: the shared memory limit never falls below what a launch was told it may use, on every device of its own, and
no thread sees another one's half-written shape."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_03510_gb300", "csrc")

HARNESS = r'''
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "launch_cache.h"
using namespace ccs;
int main() {
    // the fake runtime: a limit per device, 200 KB per SM; a call takes a while, so that threads meet in it
    static std::atomic<size_t> limit[80];
    static std::atomic<int> sets, queries, bad;
    LaunchCache cache;
    auto ask = [&](int dev, unsigned threads, size_t smem) {
        int active = -1;
        const int e = cache.blocks_per_sm<int>(dev, threads, smem,
            [&](size_t b) { std::this_thread::yield(); limit[dev < 0 ? 79 : dev] = b; ++sets; return 0; },
            [&](unsigned t, size_t b, int *a) { std::this_thread::yield(); ++queries; *a = (int)(200000 / (b + t)); return 0; },
            &active);
        // what a launch on this device needs from here on
        if (e != 0 || active != (int)(200000 / (smem + threads)) || limit[dev < 0 ? 79 : dev] < smem) ++bad;
    };
    std::vector<std::thread> pool;
    for (int t = 0; t < 8; ++t)
        pool.emplace_back([&, t] {
            for (int k = 0; k < 3000; ++k) ask((t + k) % 3, 32 * (1 + (t + k / 7) % 4), 1000 * (1 + (t * 5 + k) % 40));
        });
    for (auto &p : pool) p.join();
    printf("threads %d\n", (int)bad);
    for (int d : {0, 1, 2}) printf("limit %zu\n", (size_t)limit[d]);
    sets = queries = 0;
    LaunchCache one;
    int a = 0;
    auto set = [&](size_t) { ++sets; return 0; };
    auto query = [&](unsigned, size_t, int *x) { ++queries; *x = 3; return 0; };
    for (int k = 0; k < 5; ++k) one.blocks_per_sm<int>(0, 128, 5000, set, query, &a);
    printf("repeated %d %d\n", (int)sets, (int)queries);
    one.blocks_per_sm<int>(1, 128, 5000, set, query, &a);   // another device has an attribute of its own
    one.blocks_per_sm<int>(0, 128, 4000, set, query, &a);   // a smaller launch leaves the limit alone
    one.blocks_per_sm<int>(0, 64, 4000, set, query, &a);
    printf("device, shapes %d %d\n", (int)sets, (int)queries);
    for (int k = 0; k < 2; ++k) one.blocks_per_sm<int>(64, 128, 5000, set, query, &a);   // not in the table
    printf("beyond %d %d\n", (int)sets, (int)queries);
    // an error is returned, and nothing is kept of the call that made it
    LaunchCache err;
    const int e1 = err.blocks_per_sm<int>(0, 128, 10, [](size_t) { return 7; }, query, &a);
    queries = 0;
    const int e2 = err.blocks_per_sm<int>(0, 128, 10, set, [&](unsigned, size_t, int *) { return 9; }, &a);
    const int e3 = err.blocks_per_sm<int>(0, 128, 10, set, query, &a);
    printf("errors %d %d %d %d\n", e1, e2, e3, (int)queries);
    return 0;
}
'''


def test_limit_and_shape_under_threads_devices_and_errors(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")],
                   check=True)
    out = subprocess.run([str(tmp_path / "h")], capture_output=True, text=True, check=True).stdout.split("\n")
    assert out[0] == "threads 0"
    assert out[1:4] == ["limit 40000"] * 3
    assert out[4] == "repeated 1 1"
    assert out[5] == "device, shapes 2 4"
    assert out[6] == "beyond 4 6"
    assert out[7] == "errors 7 9 0 1"
