"""The launch shape of the sweeps, compiled for the host from the library's header (CPU).

A block's rows with work are those its MOs reach, so a colour's launch must stay
in proportion to its blocks and to the GPU, not grow with blocks x rows (the
square of the cluster): most of such a launch would have nothing to do.
"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1402_2880_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "sscf_internal.h"
int main() {
    int blocks, runs, warps, resident, waves, many;
    while (std::scanf("%d %d %d %d %d %d", &blocks, &runs, &warps, &resident, &waves, &many) == 6) {
        const sscf::SweepShape s = sscf::sweep_shape(blocks, runs, warps, resident, waves, many);
        std::printf("%d %d\n", s.shares, s.min_runs);
    }
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", include, str(d / "shape.cpp"), "-o", str(d / "shape")],
                   check=True, capture_output=True)

    def run(args):
        text = "\n".join(" ".join(map(str, a)) for a in args)
        out = subprocess.run([str(d / "shape")], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def _constant(name):
    with open(os.path.join(CSRC, "k_rotate.cu")) as f:
        return int(re.search(rf"constexpr int {name} = (\d+);", f.read()).group(1))


@pytest.mark.parametrize("mode", ["rotations", "combinations"])
def test_a_colours_launch_is_bounded(shapes, mode):
    waves = _constant("kWsRotWaves" if mode == "rotations" else "kWsCombWaves")
    many = 0 if mode == "rotations" else _constant("kWsManyRuns")
    args = []
    for n in (1, 8, 27, 100, 997, 4096, 8192, 65536, 91000):
        for blocks in (1, max(1, n // 16), max(1, n // 8)):
            for rows_per_run in (16 / 3, 32 / 3, 64 / 3):
                for warps, resident in ((1, 152), (4, 152 * 3), (4, 152 * 6)):
                    args.append((blocks, -(-n // int(rows_per_run)), warps, resident, waves, many))
    for (blocks, runs, warps, resident, _, _), (shares, min_runs) in zip(args, shapes(args)):
        assert min_runs in (warps, 2 * warps)
        assert 1 <= shares <= max(1, -(-runs // min_runs))
        # at most `waves` of the resident CTAs, and one CTA for every block
        assert shares * blocks <= waves * resident + blocks
        # a launch below the limit has a share for every run its blocks can have
        if -(-runs // min_runs) * blocks <= waves * resident:
            assert shares * min_runs >= runs
