"""CPU check of the rule that picks the launch of the segment recurrences: every line of the
accepted sizes (n <= 40000, so up to 625 segments of 32 unknowns) is covered by a CTA whose
registers fit an SM."""
import os
import subprocess

from paper_1710_11259_gb300 import build_ext

PROGRAM = r"""
#include <cstdio>
#include "sweep.cuh"
int main()
{
    for (int fp64 = 0; fp64 < 2; ++fp64)
        for (int mode = 0; mode < 3; ++mode)
            for (int nb = 1; nb <= 625; ++nb) {
                const int len = fps::chain_length(fp64, mode, nb);
                std::printf("%d %d %d %d %d\n", fp64, mode, nb, len, len ? fps::chain_warps(fp64, len) : 0);
            }
}
"""

REGISTERS = {(0, 8): 64, (0, 16): 96, (1, 8): 96}  # per thread, as stated beside the rule


def test_every_line_has_a_launch_that_fits(tmp_path):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build_ext._nvcc())), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", f"-I{cuda}", f"-I{build_ext.CSRC}", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    walks = set()
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]:
        fp64, mode, nb, length, warps = map(int, line.split())
        if length == 0:  # the walking kernel takes any number of segments
            walks.add((fp64, nb))
            continue
        assert -(-nb // length) <= warps <= 32, line
        assert 32 * warps * REGISTERS[fp64, length] <= 65536, line
    assert min(nb for f, nb in walks if f == 1) == 161 and min(nb for f, nb in walks if f == 0) == 321
