"""The sizes of the watertight check's edge table (csrc/emb_edges.cuh, host arithmetic): the
table that decides holds every edge a list can have, so that no probe walks a full table."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_01251_gb300", "csrc")

MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include "emb_edges.cuh"
int main(int n, char **a)
{
    for (int i = 1; i + 1 < n; i += 2)
        for (int k = 0; k < 2; ++k) {
            const EdgePlan P = emb_edge_plan(atoll(a[i]), atoll(a[i + 1]), k);
            printf("%s %s %d %d %d %llu\n", a[i], a[i + 1], k, (int)P.slots, (int)P.all, (unsigned long long)P.cap);
        }
}
"""


def test_the_last_table_holds_every_edge(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "plan.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "plan")
    subprocess.check_call([cxx, "-I", CSRC, str(src), "-o", exe])
    T = [1, 255, 256, 1024, 4096, 5461, 65535, 65536, 65537, 1 << 17, 1000003, 1398101, 1 << 22, 7197216, 1 << 30]
    pairs = [(v, t) for t in T for v in (3, t // 100 + 3, t // 2 + 2, 2 * t, 2 * t + 1, 3 * t)]
    out = subprocess.check_output([exe] + [str(x) for p in pairs for x in p], text=True)
    rows = [[int(x) for x in line.split()] for line in out.splitlines()]
    assert len(rows) == 2 * len(pairs)
    for v, t, attempt, slots, full, cap in rows:
        assert cap & (cap - 1) == 0 and cap >= 1024
        assert slots == (v <= 2 * t)
        # triangles without a common edge have 3 each; a list without slots is decided at once
        if full:
            assert 4 * 3 * t <= 3 * cap, (v, t, cap)
        assert full or (attempt == 0 and slots)
