"""CPU check of the packed fill's offset ring (wavefront16.cuh): with the
constants of the source, no profile offset that a compute warp still reads can
be overwritten by an input warp that runs as far ahead as it may."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The last warp of a strip is the one that reads furthest back.  At the start of the chunk at step s0
# it has published min(n, s0 - lag) columns; its lanes read the offsets of columns s0 - 2 lane and on, in the
# sweep's first chunk also the one before.  A block's first strip starts one chunk left of the task.
MODEL = r"""
#include "sw.h"
#include "wavefront16.cuh"
#include <cstdio>
using namespace swgb;
int main() {
    for (int n = 1; n < 6000; n += n < 1400 ? 1 : 997)
        for (int start = -kP16CH; start <= 0; start += kP16CH)
            for (int s0 = start; s0 < n + kP16Lag; s0 += kP16CH) {
                const int past = s0 - kP16Lag, done = past < 0 ? 0 : (past < n ? past : n);
                const int first = s0 - 2 * 31 - (s0 == start ? 1 : 0);
                // the columns whose offsets may be in the ring: below the room; column c sits in slot c mod kQB
                if (first + kQB < p16_offset_room(done)) {
                    std::printf("n %d, chunk %d: column %d's slot may hold column %d\n", n, s0, first, first + kQB);
                    return 1;
                }
            }
    return 0;
}
"""


def test_offsets_in_use_are_never_overwritten(tmp_path):
    from paper_2211_10769_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, exe = tmp_path / "ring.cu", tmp_path / "ring"
    src.write_text(MODEL)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
