"""The rules that cut the FFT passes into blocks, compiled for the host."""
import subprocess

from paper_2105_06055_gb300 import build

SRC = """
#include <cstdio>
#include "pd_plan.cuh"
int main()
{
    using namespace pd;
    // rows of a tile: FP64, packed values, fields
    const int rows[][3] = {{1, 512, 2}, {1, 1024, 2}, {0, 512, 2}, {0, 1024, 2}, {1, 1024, 1}, {0, 1024, 3}};
    for (auto &r : rows)
        std::printf("%d %d\\n", row_tile_rows(r[0], r[1], 3, r[2]), row_warps(r[0], r[1], 3, r[2]));
    return 0;
}
"""


def _run(tmp_path):
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(SRC)
    subprocess.check_call([build._nvcc()] + build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                          "-I", build.INCLUDE, "-o", str(exe), str(src), build.build(),
                          "-Xlinker", "-rpath", "-Xlinker", build.BUILD])
    return [tuple(map(int, r.split())) for r in subprocess.check_output([str(exe)], text=True).splitlines()]


def test_long_rows_of_two_fields_take_a_block_each(tmp_path):
    """Two fields in FP64, and rows of 1024 packed values in either precision: one row
    per block (a warp or a pair of warps per field), so that a grid of 16 rows runs on
    16 SMs; shorter FP32 rows go in twos."""
    assert _run(tmp_path) == [(1, 2), (1, 4), (2, 4), (1, 4), (4, 8), (1, 6)]
