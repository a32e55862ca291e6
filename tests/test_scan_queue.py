"""Places in the queue of deferred scans, on the host: whatever number of
scans a level asks for, no place is handed out twice."""
from __future__ import annotations

import subprocess

from paper_2212_00977_gb300 import build_lib

PROGRAM = r"""
#include <stdio.h>
#include "pspc_level.cuh"
using namespace pspc;
int main() {
    const unsigned cap = 1u << 26;
    decltype(LevelStatus::n_scan) asked = 0;
    unsigned long long next_free = 0, true_asked = 0;
    // a level's vertices: the first ones fill the queue, the others ask for more than 2^32 in all
    for (long k = 0; k < 600; ++k) {
        const unsigned want = k < 40 ? 1000003u : 16777213u;
        const unsigned q0 = scan_place(asked, cap);
        asked += want;
        true_asked += want;
        if (asked != true_asked) return printf("%ld: the count wrapped\n", k), 1;
        if (q0 > cap) return printf("%ld: place %u is outside\n", k, q0), 1;
        if (q0 < next_free) return printf("%ld: place %u is taken\n", k, q0), 1;
        next_free = (unsigned long long)q0 + want < cap ? (unsigned long long)q0 + want : cap;
    }
    return scan_place(0, cap) == 0 && scan_place(cap - 1, cap) == cap - 1 && scan_place(cap, cap) == cap ? 0 : 2;
}
"""


def test_no_place_twice_beyond_2_32(tmp_path):
    src = tmp_path / "queue.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "queue"
    subprocess.run([build_lib._nvcc(), *build_lib._flags(), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
