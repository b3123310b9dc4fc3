"""Shared-memory staging of the finest level, checked on the CPU for every grid
side the library accepts: the rows a phase takes at a time fit the floats a
launch reserves, at least one row is taken, and the staging beside the largest
one-block tail fits the launch's shared memory."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_1653_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "fine_stage.h"
int main() {
    for (int side = 7; side <= %d; side = 2 * side + 1)
        std::printf("%%d %%d %%d %%d\n", side, gs::fine_stage_floats(side), gs::fine_restrict_chunk(side),
                    gs::fine_update_chunk(side));
}
"""


def constant(name, file):
    src = open(os.path.join(CSRC, file)).read()
    return eval(re.search(r"constexpr \w+ %s = ([^;]+);" % name, src).group(1))


def test_staging_fits_on_every_accepted_side(tmp_path):
    largest = constant("kIsaacsMaxSide", "common.cuh")
    (tmp_path / "t.cpp").write_text(PROGRAM % largest)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    rows = [list(map(int, line.split())) for line in subprocess.run([exe], check=True, capture_output=True, text=True)
            .stdout.splitlines()]
    assert rows[-1][0] == largest == 16383
    # the tail of a grid: five levels of up to 16^2 cells and the inverse of 49 unknowns
    rec, planes = 57, 4 * 18 * 18
    tail = 4 * sum(rec * m * m + planes for m in (1, 2, 4, 8, 16)) + 8 * (49 * 49 + 49)
    for side, floats, restrict, update in rows:
        half = (side + 1) // 2
        assert restrict >= 1 and (2 * restrict + 1) * half <= floats, side
        assert update >= 1 and update * (side + 1) <= floats, side
        assert tail + 256 + 4 * floats <= constant("kTiledSmemMax", "mgsolve.cuh"), side


def test_launch_reserves_what_the_phases_stage():
    """The launch's size and the phases take their sizes from the same functions."""
    mg = open(os.path.join(CSRC, "mgsolve.cu")).read()
    fine = open(os.path.join(CSRC, "fine.cuh")).read()
    assert "fine_stage_floats(a.L[0].side) * sizeof(float)" in mg
    assert "fine_restrict_chunk(V.side)" in fine and "fine_update_chunk(V.side)" in fine
    assert "kFineStage" not in mg + fine
