"""Sizes of the Gregory box tables (csrc/table_plan.h), compiled with the host C++ compiler: what is stored fits its bytes, and
what an update of the points rebuilds stays within 10 levels and 2^16 nodes whatever the number of patches."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_03510_gb300", "csrc")

HARNESS = r'''
#include <cstdio>
#include "table_plan.h"
int main() {
    unsigned n; unsigned long long bytes;
    while (scanf("%u %llu", &n, &bytes) == 2) {
        const unsigned s = ccs::greg_table_levels(n, bytes);
        printf("%u %u %u\n", s, ccs::greg_update_levels(n, s), ccs::greg_update_blocks(n, s));
    }
    return 0;
}
'''

BIG = 1 << 33


def test_stored_and_updated_levels(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    cases = [(n, b) for n in (0, 1, 24, 64, 65, 96, 384, 1536, 4056, 16224, 32768, 32769, 64896, 1 << 22, (1 << 22) + 1, 1 << 26)
             for b in (0, 1 << 20, BIG)]
    text = "\n".join(f"{n} {b}" for n, b in cases) + "\n"
    out = subprocess.run([str(tmp_path / "h")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    got = {c: tuple(map(int, q.split())) for c, q in zip(cases, out)}
    for (n, b), (stored, update, blocks) in got.items():
        most = min(b, 1 << 28)
        assert stored <= 16 and (stored == 0 or (n << stored) * 64 <= most), (n, b)
        assert stored == 16 or n == 0 or (n << (stored + 1)) * 64 > most, (n, b)   # as deep as fits
        assert update <= min(stored, 10) and (update == 0 or n << update <= 1 << 16), (n, b)
        assert update == min(stored, 10) or n << (update + 1) > 1 << 16, (n, b)
        # a scene's blocks cover its own nodes, at least the depth word; a scene without a table has none
        assert blocks == (0 if stored == 0 else max(1, -(-(n << update) // 128)) if update else 1), (n, b)
    assert [got[(n, BIG)][1] for n in (24, 64, 65, 96, 1536, 4056, 32768, 32769, 64896)] == [10, 10, 9, 9, 5, 4, 1, 0, 0]
