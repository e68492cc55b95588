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
    // columns of a special tile: log2 of the axis, tile width, other tiles (148 SMs)
    const int cols[][3] = {{10, 8, 32}, {10, 8, 148}, {10, 8, 149}, {9, 8, 128}, {9, 2, 1000}, {8, 16, 16}, {4, 2, 1}};
    for (auto &c : cols) std::printf("%d 0\\n", special_cols(c[0], c[1], c[2], 148));
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
    assert _run(tmp_path)[:6] == [(1, 2), (1, 4), (2, 4), (1, 4), (4, 8), (1, 6)]


def test_special_tiles_of_long_axes_take_one_pair(tmp_path):
    """Axes of 512 nodes and more whose other tiles fit the SMs at once: a pair of kx = 0
    columns per block; else two pairs, or the tile's width where that is one."""
    assert [c for c, _ in _run(tmp_path)[6:]] == [2, 2, 4, 2, 2, 4, 2]
