"""Which values of tail_items let the same rounds into the cluster kernel of a single
query's small rounds (the autotuner times one of them)."""
import os
import subprocess

from paper_1812_10499_gb300 import build as libbuild

PROGRAM = r"""
#include <cstdio>
#include "sssp_engine.h"
using namespace sssp;
int main() {
    // 12288 vertices are 384 tiles; 16 chunks from a hub degree of 256 up, 4096 / degree below.
    const bool ok = same_small_rounds(512, 1024, 256) && same_small_rounds(400, 2048, 256) &&
                    !same_small_rounds(399, 400, 256) && !same_small_rounds(0, 128, 256) &&
                    same_small_rounds(256, 256, 256) && same_small_rounds(1000000, 400, 1u << 20) &&
                    same_small_rounds(416, 512, 128) && !same_small_rounds(415, 512, 128) &&
                    !same_small_rounds(1024, 2048, 4) && same_small_rounds(4480, 4481, 1);
    std::printf("%d\n", ok ? 1 : 0);
    return 0;
}
"""


def test_limits_that_are_one_limit(tmp_path):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), *libbuild.ARCH, "-std=c++17", "-I", libbuild.INCLUDE,
                           "-I", libbuild.CSRC, "-o", str(exe), str(src)])
    assert subprocess.check_output([str(exe)], text=True).strip() == "1"
