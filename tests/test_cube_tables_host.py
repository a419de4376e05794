"""CPU check of which thread of the cube's table kernel computes which half line.  The two
halves of a line are neighbouring lanes that exchange a pivot, and the grid is whole blocks of
64 threads, so up to 56 threads are past the end of the list."""
import os
import subprocess

from paper_1710_11259_gb300 import build_ext

PROGRAM = r"""
#include <cstdio>
#include "cube_unit.cuh"
int main()
{
    for (int shifts = 1; shifts <= 40; ++shifts)
        for (int raw = 0; raw < (8 * shifts + 63) / 64 * 64; ++raw)
            std::printf("%d %d %d\n", shifts, raw, fps::unit_table_thread(raw, shifts));
}
"""


def test_halves_of_a_line_are_a_lane_pair(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build_ext._nvcc())), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", f"-I{cuda}", f"-I{build_ext.CSRC}", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    ids = {}
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]:
        shifts, raw, i = map(int, line.split())
        ids[shifts, raw] = i
    for (shifts, raw), i in ids.items():
        assert 0 <= i < 8 * shifts
        assert ids[shifts, raw ^ 1] == i ^ 1, (shifts, raw)  # the partner holds the other half of the line
        if raw < 8 * shifts:
            assert i == raw
