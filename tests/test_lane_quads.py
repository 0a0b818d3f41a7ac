"""The walk over a warp's lanes in groups of four, which the first pass takes over the rows it updates: every group that
has a lane once, in order, and an end after the last one -- also when lanes 28 to 31 are among them. Checked on the
host, where a shift by the width of the mask neither ends the loop nor passes the sanitizer."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1708_06065_gb300", "csrc")

PROGRAM = r"""
#include "lane_quads.h"
// constant evaluation refuses undefined operations
static_assert(!lair::lanes_from(0xffffffffu, 32), "end");
static_assert(lair::lanes_from(0x80000000u, 28) && lair::lane_quad(0x80000000u, 28), "last group");
static_assert(!lair::lanes_from(0u, 0) && !lair::lanes_from(0xfu, 4) && !lair::lane_quad(0xfffffff0u, 0), "none");
int main() {
    for (unsigned groups = 0; groups < 256; ++groups)
        for (int lane = 0; lane < 4; ++lane) {   // the lane that stands for its group
            unsigned lanes = 0, seen = 0;
            for (int g = 0; g < 8; ++g)
                if (groups >> g & 1) lanes |= 1u << (4 * g + lane);
            int last = -4, steps = 0;
            for (int p = 0; lair::lanes_from(lanes, p); p += 4) {
                if (p % 4 || p <= last || ++steps > 8) return 1;
                if (!lair::lane_quad(lanes, p)) continue;
                last = p;
                seen |= 1u << (p / 4);
            }
            if (seen != groups) return 2;
        }
    return 0;
}
"""


def test_every_group_of_four_lanes_once(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "quads.cpp", tmp_path / "quads"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=20).returncode == 0
