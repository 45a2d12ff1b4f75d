"""The transform's launch shape belongs to the storage precision (host logic, CPU).

The two precisions have kernels of their own and ranges of their own (4 to 16 CTAs
per tile by size in FP32, 8 to 128 in FP64), so a choice that the autotuner made
in one must not hold after the context is converted to the other.
"""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "sscf_internal.h"
int main() {
    sscf::Ctx c;
    c.n_sm = 152;
    c.n_occ_tiles = 16;
    c.prec = SSCF_MIXED;
    const int mixed = sscf::transform_split(&c);
    c.tf_split[c.prec] = 2;   // tuned
    const int tuned = sscf::transform_split(&c);
    c.prec = SSCF_FP64;       // converted
    const int fp64 = sscf::transform_split(&c);
    c.tf_split[c.prec] = 4;
    c.prec = SSCF_MIXED;
    std::printf("%d %d %d %d\n", mixed, tuned, fp64, sscf::transform_split(&c));
}
"""


def test_a_tuned_split_does_not_outlive_its_precision(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1402_2880_gb300", "csrc"), "-I", include,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    # by size: 8 (FP32) or 32 (FP64) CTAs per SM over 16 tiles, at most 16 or 128 per tile
    assert [int(x) for x in out] == [16, 2, 128, 2]
