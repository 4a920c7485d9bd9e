"""The conservation record of a step has one writer per launch: the blocks that
combine the record of the step before, or the block that combines this step's."""
import subprocess

from paper_2106_01557_gb300 import build

PROGRAM = """
#include <cstdio>
#include "lbm_internal.h"
int main() {
    lbm::MarchGrid m{};
    m.groups = 3, m.warps = 4, m.chunks = 5, m.combine_prev = 2;
    for (int first = 0; first < 2; ++first)
        for (int last = 0; last < 2; ++last) {
            const lbm::MarchGrid s = lbm::step_grid(m, first, last);
            std::printf("%d %d %d %d %d %d %d\\n", first, last, s.groups, s.warps, s.chunks, s.combine_prev, s.combine_here);
        }
}
"""


def test_one_writer_of_the_record_per_launch(tmp_path):
    src, exe = tmp_path / "grid.cu", tmp_path / "grid"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    rows = [tuple(map(int, r.split())) for r in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 4
    for first, last, groups, warps, chunks, prev, here in rows:
        assert (groups, warps, chunks) == (3, 4, 5)
        assert not (prev and here)
        assert here == last  # a call's last step combines its own record
        assert prev == (0 if first or last else 2)  # one between two others that of the step before
