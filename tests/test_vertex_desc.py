"""A vertex's description (sssp_dev.cuh) on the CPU: the prefix of its in-edges that
a lower-bound scan reads holds every edge up to the limit, and degrees that 32 bits
do not hold (parallel edges) are marked as such, with whole rows."""
import os
import subprocess

from paper_1812_10499_gb300 import build as libbuild

PROGRAM = r"""
#include <cstdio>
#include "sssp_dev.cuh"
using namespace sssp;
int main() {
    int bad = 0;
    const u64 big = 1ull << 32;
    const u64 degs[] = {0, 1, 7, 255, 256, 257, 4000, 1ull << 31, big - 2, big - 1, big, big + 5, 3 * big + 1};
    const u32 shift = 4;   // weights to 255
    for (u64 deg : degs)
        for (u64 odeg : degs)
            for (int rows = 0; rows < 4; ++rows) {
                u32 sums[kClasses];
                for (u32 k = 0; k < kClasses; ++k)
                    sums[k] = k + 1 == kClasses ? (u32)deg
                              : rows == 1       ? (u32)(deg * (k + 1) / kClasses)
                              : rows == 2       ? (u32)(deg ? 1 : 0)
                                                : 0u;
                const VDesc d = make_vdesc(9, deg, odeg, 3, 2, rows ? sums : nullptr);
                const bool whole = deg >= kDegreeMax;
                if (d.deg != (whole ? kDegreeMax : (u32)deg)) ++bad;
                if (d.odeg != (odeg >= kDegreeMax ? kDegreeMax : (u32)odeg)) ++bad;
                for (u32 w = 1; w <= 255; ++w) {
                    const u32 p = light_prefix(d, w, shift);
                    if (whole || !rows) {
                        if (p != d.deg) ++bad;
                    } else if (p < sums[wclass(w, shift)] || p > d.deg) {
                        ++bad;
                    }
                }
            }
    std::printf("%d\n", bad);
    return 0;
}
"""


def test_descriptions(tmp_path):
    src, exe = tmp_path / "d.cu", tmp_path / "d"
    src.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), *libbuild.ARCH, "-std=c++17", "-I", libbuild.INCLUDE,
                           "-I", libbuild.CSRC, "-o", str(exe), str(src)])
    assert subprocess.check_output([str(exe)], text=True).strip() == "0"
