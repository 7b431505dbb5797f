"""Which ray a thread of the candidate pass takes (csrc/cand_plan.h), compiled with the host C++ compiler: the threads cover
every ray once for images with ragged bands and partial rows, and a width that makes no tile, up to the largest a caller
can pass, leaves the rays in their own order instead of wrapping around 32 bits."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_03510_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include <vector>
#include "cand_plan.h"
using namespace ccs;
int main() {
    unsigned n, w;
    while (scanf("%u %u", &n, &w) == 2) {
        const unsigned img = cand_tile_width(n, w), t = cand_threads(n, img);
        const char *what = "once";
        if (t < n || (unsigned)(t + 4095u) < t) what = "wrapped";
        else if (n <= 1u << 22) {
            std::vector<char> seen(t, 0);
            for (unsigned k = 0; k < t; ++k) {
                const unsigned r = cand_ray(k, img);
                if (r >= t || seen[r]++) { what = "twice"; break; }
            }
        } else {   // the ends
            for (unsigned k : {0u, 1u, 31u, 32u, t / 2, t - 33u, t - 1u})
                if (cand_ray(k, img) >= t) what = "outside";
            if (cand_ray(t - 1u, img) != t - 1u) what = "last";
        }
        printf("%u %u %s\n", img, t, what);
    }
    return 0;
}
'''

# rays, image width -> the tile width taken, the threads
CASES = {
    (1920 * 1080, 1920): (1920, 1920 * 1080), (336 * 211, 336): (336, 336 * 212), (336 * 211 - 5, 336): (336, 336 * 212),
    (64, 8): (8, 64), (8, 8): (8, 32), (7, 8): (0, 7), (1000, 0): (0, 1000), (333 * 211, 333): (0, 333 * 211),
    (1, 64): (0, 1), (100, 104): (0, 100), (104, 104): (104, 416),
    (1000, 1 << 20): (0, 1000), (1000, 1 << 30): (0, 1000), (1000, 1 << 31): (0, 1000), (1000, 2 ** 32 - 8): (0, 1000),
    (1 << 30, 1 << 30): (0, 1 << 30), (858993459, 858993456): (0, 858993459), (2 ** 32 - 4096, 8): (0, 2 ** 32 - 4096),
    (1 << 31, 1 << 16): (1 << 16, 1 << 31), ((1 << 31) - 1, 1 << 26): (1 << 26, 1 << 31),
}


def test_every_ray_once_and_widths_without_a_tile(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    text = "\n".join(f"{n} {w}" for n, w in CASES) + "\n"
    out = subprocess.run([str(tmp_path / "h")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for (case, (img, threads)), line in zip(CASES.items(), out):
        assert line == f"{img} {threads} once", (case, line)
