"""The height of the items of a batch's second work split: small batches are
spread over all warps, large ones in items of 32 rows."""
import subprocess

import pytest

from paper_2106_01557_gb300 import build

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "lbm_batch.h"
int main(int, char** v) {
    std::printf("%d\\n", lbm::batch_item_rows(std::atoll(v[1]), std::atoi(v[2])));
}
"""


@pytest.fixture(scope="module")
def item_rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "rows.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.CSRC, "-o", str(d / "rows"), str(d / "rows.cu")], check=True)
    return lambda rows, warps: int(subprocess.run([str(d / "rows"), str(rows), str(warps)], check=True, capture_output=True, text=True).stdout)


@pytest.mark.parametrize("rows,warps,want", [(1, 1, 1), (128, 128, 1), (1216, 1216, 1), (1217, 1216, 2), (2432 * 31, 2432, 31),
                                             (2432 * 32 + 1, 2432, 32), (1 << 33, 1216, 32)])
def test_item_rows(item_rows, rows, warps, want):
    assert item_rows(rows, warps) == want
