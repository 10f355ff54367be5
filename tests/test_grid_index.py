"""Record indices of grids whose 16-bit records, with their padding, pass
2^31 in one channel: the functions the kernels index with, compiled for the
host and compared with Python's integers."""
import os
import subprocess

import pytest

from paper_2303_06150_gb300 import build

# (nx, ny, nz, nc): the largest and a thin grid of each kind that check_grid accepts (cells * nc <= 2e9)
GRIDS = [(2, 5000, 240000, 1), (240000, 5000, 2, 1), (2, 240000, 5000, 1), (2, 2, 1000000000, 1), (96, 96, 96, 8),
         (1000000001, 2, 2, 2), (1200, 1200, 1300, 1), (2, 2, 2, 64)]

MAIN = r"""
#include <cstdio>
#include "internal.h"
using namespace ligen;
int main() {
  int n[4];
  while (scanf("%d %d %d %d", n, n + 1, n + 2, n + 3) == 4)
    for (int fmt : {(int)kRecF32, (int)kRecF16}) {
      const int cx = rec_cells(n[0], fmt), cy = rec_cells(n[1], fmt), cz = rec_cells(n[2], fmt), c = n[3] - 1;
      const size_t last = rec_index(cx, cy, cz, c, cx - 1, cy - 1, cz - 1);
      printf("%zu %zu %zu\n", last, rec_index(cx, cy, cz, c, 0, 0, cz - 1),
             fmt == kRecF32 ? rec_index_f32(cx, cy, cz, c, cx - 1, cy - 1, cz - 1) : last);
    }
}
"""


@pytest.fixture(scope="module")
def indices(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid_index")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([build.NVCC, "-std=c++17", *build.ARCH, "-I", build.CSRC, str(d / "main.cu"), "-o", str(d / "main")],
                   check=True, capture_output=True)
    text = "\n".join(" ".join(map(str, g)) for g in GRIDS)
    out = subprocess.run([str(d / "main")], input=text, check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


@pytest.mark.parametrize("k", range(2 * len(GRIDS)))
def test_record_index(indices, k):
    (nx, ny, nz, nc), pad = GRIDS[k // 2], k % 2   # FP32 records: n - 1 cells per axis, 16-bit ones n
    cx, cy, cz = nx - 1 + pad, ny - 1 + pad, nz - 1 + pad
    last = cx * cy * cz * nc - 1
    assert indices[k] == (last, last - cx * cy + 1, last)
