"""The engine of launches that leave it open (csrc/engine_plan.h), compiled with the host C++ compiler: calls of less than a
warp, shallow leaves in world axes and very large launches stay on the ray-persistent kernel, and the pair engine does not
run with a refill threshold of a whole warp."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_03510_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include "engine_plan.h"
int main() {
    unsigned n, p, local, depth, refill;
    while (scanf("%u %u %u %u %u", &n, &p, &local, &depth, &refill) == 5)
        printf("%d %u\n", (int)ccs::pairs_by_default(n, p, local != 0, depth), ccs::default_pairs_refill(refill));
    return 0;
}
'''

# rays, patches, local frames, leaf depth, refill -> the pair engine or not, its refill threshold
CASES = {
    (1, 96, 1, 8, 8): (0, 8), (31, 98304, 0, 8, 8): (0, 8), (32, 1536, 1, 8, 8): (1, 8), (32, 1536, 0, 8, 8): (1, 8),
    (0, 96, 1, 8, 8): (0, 8), (1 << 23, 96, 1, 8, 8): (1, 8), ((1 << 23) + 1, 96, 1, 8, 8): (0, 8),
    (4096, 1536, 0, 1, 8): (0, 8), (4096, 1536, 0, 3, 8): (0, 8), (4096, 1536, 0, 4, 8): (1, 8), (4096, 1536, 1, 1, 8): (1, 8),
    (4096, 96, 0, 2, 8): (1, 8), (16 * 96, 96, 0, 2, 8): (0, 8), (16 * 96 + 1, 96, 0, 2, 8): (1, 8),
    (230400, 24576, 0, 2, 8): (0, 8), (919911, 24576, 0, 2, 8): (1, 8), (1 << 23, 1 << 26, 0, 3, 8): (0, 8),
    (1000, 0, 0, 2, 8): (1, 8),
    (919911, 1536, 0, 8, 1): (1, 1), (919911, 1536, 0, 8, 24): (1, 24), (919911, 1536, 0, 8, 25): (1, 24),
    (919911, 1536, 0, 8, 32): (1, 24),
}


def test_rule_and_refill(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    text = "\n".join(" ".join(map(str, c)) for c in CASES) + "\n"
    out = subprocess.run([str(tmp_path / "h")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for (case, want), line in zip(CASES.items(), out):
        assert tuple(map(int, line.split())) == want, case
