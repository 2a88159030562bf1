"""The shared-memory order of the 3D residual + full weighting (no GPU): restrict_turns.h, compiled with
the host compiler, gives which shared plane and which group of warps every coarse plane of a block
uses; for every pair of warps, each store into a shared plane must be ordered after the reads of what
the plane held before, and no barrier may be arrived at twice before it has completed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include "restrict_turns.h"

// Warp w has waited for barrier instance p (so that every warp has arrived at p, and done what it does
// before that) once it has passed coarse plane p in a turn of its own.
static bool waited_in(int w, int first, int last) {
    for (int p = first; p <= last; p++)
        if (r3_turn(p) == r3_group(w)) return true;
    return false;
}

int main(void) {
    const int warps = WARPS, planes = 24;
    for (int c = 0; c < planes; c++) {
        int sums = 0;
        for (int w = 0; w < 16; w++) sums += r3_turn(c) == r3_group(w);
        if (sums != 4) printf("plane %d is summed by %d warps\n", c, sums);
    }
    for (int r = 0; r < warps; r++)        // reads plane c in its own turn, after all have arrived at c
        for (int c = 0; c < planes; c++) {
            if (r3_turn(c) != r3_group(r)) continue;
            for (int w = 0; w < warps; w++)  // stores into the same shared plane at coarse plane d
                for (int d = c + 1; d < planes; d++)
                    if (r3_plane(d) == r3_plane(c) && w != r && !waited_in(w, c + 1, d - 1))
                        printf("warp %d stores plane %d while warp %d may read plane %d\n", w, d, r, c);
        }
    // barrier 1 + turn: instance d of a barrier must not be reached before instance c has completed
    for (int w = 0; w < warps; w++)
        for (int c = 0; c < planes; c++)
            for (int d = c + 1; d < planes; d++)
                if (r3_turn(d) == r3_turn(c) && !waited_in(w, c, d - 1))
                    printf("warp %d arrives at plane %d before the barrier of plane %d has completed\n", w, d, c);
    return 0;
}
"""


# 18 warps: one thread per node of the 33 x 17 fine region
@pytest.mark.parametrize("warps", [18])
def test_stores_follow_reads(tmp_path, warps):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "turns.cc", tmp_path / "turns"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-DWARPS=%d" % warps, "-I", os.path.join(ROOT, "paper_1012_4307_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out == "", out
