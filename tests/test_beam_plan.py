"""Shared memory of the beam launches: whatever D and B, a pool has the plan (tables, lists) that the largest size gives it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_05330_b200", "csrc")

MAIN = r"""
#include "beam_plan.h"
#include "sdms.h"
#include <cstdio>
int main() {
  for (int d = 1; d <= SDMS_MAX_DRAFT; ++d)
    for (int b = 1; b <= SDMS_MAX_BEAMS; ++b) std::printf("%d %d %d\n", d, b, sdms::beam_bytes(d, b));
}
"""


def needs(M, D, B):
    """Bytes of the tables, and of tables and lists, of a pool with M matches."""
    cap = 64
    while cap < M + M // 4 + 1:
        cap *= 2
    row = -(-M // 32) * 32
    tables = D * (16 * cap + 2 * row) + 6 * cap + 2 * row
    return tables, tables + D * cap * B * 16


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("beam_plan")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "main.cpp"),
                    "-o", str(d / "main")], check=True)
    lines = subprocess.run([str(d / "main")], check=True, capture_output=True, text=True).stdout.splitlines()
    return {tuple(map(int, x.split()[:2])): int(x.split()[2]) for x in lines}


def test_no_pool_loses_its_place_in_shared_memory(sizes):
    full = 200 * 1024
    assert len(sizes) == 32 * 8
    for (D, B), have in sizes.items():
        fit = max((n for M in range(1, 6500) for n in needs(M, D, B) if n <= full), default=0)
        # every pool that fits at the largest size fits, and what it does not take stays cache
        assert have == next(x for x in (160 * 1024, 192 * 1024, full) if fit <= x), (D, B, have, fit)
