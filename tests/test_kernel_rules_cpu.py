"""CPU checks of rules that the kernels rely on, compiled from their headers
and run on the host: the packed fill's offset ring (wavefront16.cuh) and where a
walk starts (walk.cuh)."""
import subprocess

import pytest


def _run(tmp_path, text):
    from paper_2211_10769_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(text)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


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
    """With the constants of the source, no profile offset that a compute warp still reads can be
    overwritten by an input warp that runs as far ahead as it may."""
    _run(tmp_path, MODEL)


START = r"""
#include "sw.h"
#include "walk.cuh"
#include <cstdio>
using namespace swgb;
int main() {
    // an earlier call's candidate, far outside the pair that was refused
    for (int err : {kErrBadCode, kErrTimeout})
        for (bool local : {true, false}) {
            const WalkState w = walk_start(make_int4(4000, 8000, 8000, 0), local, err);
            if (w.done == 0 || w.i != 1 || w.j != 1) { std::printf("error %d: walks from %d, %d\n", err, w.i, w.j); return 1; }
        }
    const WalkState ok = walk_start(make_int4(7, 30, 40, 0), true, 0), none = walk_start(make_int4(0, 30, 40, 0), true, 0),
                    any = walk_start(make_int4(-7, 30, 40, 0), false, 0), edge = walk_start(make_int4(5, 0, 40, 0), false, 0);
    return !(ok.done == 0 && ok.i == 30 && ok.j == 40 && ok.state == 0 && ok.nruns == 0 && none.done == 3 &&
             any.done == 0 && any.i == 30 && any.j == 40 && edge.done == 3);
}
"""


def test_no_walk_after_an_error(tmp_path):
    """A walk that starts on the device starts nowhere when the error word is set: the candidates and
    decision words are then not this call's."""
    _run(tmp_path, START)
