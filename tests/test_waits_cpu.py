"""The rule by which a block leaves after a wait that ran out (wait_for_copies), compiled
for the host: one thread of a block, with a wait that answers as told and a vote that
also holds another thread's answer. When any thread's wait has run out, the first
thread, which issues the copies, drains them before the block's last vote; the others
do not, and nothing is drained when all waits succeed."""
import subprocess

from paper_2105_06055_gb300 import build

SRC = """
#include <cstdio>
#include "pd_tma.cuh"
int main()
{
    for (int first = 0; first < 2; ++first)
        for (int other = 0; other < 2; ++other)
            for (int mine = 0; mine < 2; ++mine) {
                int votes = 0;
                const bool ok = pd::wait_for_copies(
                    first != 0, [&]() { return std::printf("w"), mine != 0; },
                    [&](bool x) { return std::printf("v"), x || (votes++ == 0 && other != 0); },
                    []() { std::printf("d"); });
                std::printf(" %d\\n", ok ? 1 : 0);
            }
    return 0;
}
"""


def test_a_block_that_gives_up_drains_its_copies(tmp_path):
    src, exe = tmp_path / "waits.cu", tmp_path / "waits"
    src.write_text(SRC)
    subprocess.check_call([build._nvcc()] + build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                          "-I", build.INCLUDE, "-o", str(exe), str(src)])
    got = subprocess.check_output([str(exe)], text=True).splitlines()
    # by (first thread, another thread's wait ran out, this thread's wait succeeded)
    assert got[:4] == ["wvv 0", "wv 1", "wvv 0", "wvv 0"]
    assert got[4:] == ["wvdv 0", "wv 1", "wvdv 0", "wvdv 0"]
