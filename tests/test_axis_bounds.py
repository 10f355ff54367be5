"""The box bound and last cell that the samplers compare and clamp with, for
axes up to the longest accepted one: no FP32 coordinate inside the bound is
past the last point, no clamped cell past the last cell, and short axes are
exact. Compiled for the host from the kernels' header."""
import subprocess

import numpy as np
import pytest

from paper_2303_06150_gb300 import build

POINTS = [2, 3, 96, 2 ** 23, 2 ** 24 - 1, 2 ** 24, 2 ** 24 + 1, 2 ** 24 + 2, 2 ** 24 + 3, 2 ** 24 + 4, 2 ** 24 + 5,
          2 ** 25, 2 ** 25 + 1, 2 ** 25 + 3, 2 ** 27 + 63, 10 ** 9, 10 ** 9 + 1, 2 * 10 ** 9 + 1]

MAIN = r"""
#include <cstdio>
#include "internal.h"
int main() {
  int n;
  while (scanf("%d", &n) == 1) {
    float top, last;
    ligen::axis_bounds(n, &top, &last);
    printf("%.1f %.1f\n", top, last);
  }
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("axis_bounds")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([build.NVCC, "-std=c++17", *build.ARCH, "-I", build.CSRC, str(d / "main.cu"), "-o", str(d / "main")],
                   check=True, capture_output=True)
    out = subprocess.run([str(d / "main")], input="\n".join(map(str, POINTS)), check=True, capture_output=True,
                         text=True).stdout
    return {n: tuple(int(float(v)) for v in line.split()) for n, line in zip(POINTS, out.splitlines())}


@pytest.mark.parametrize("n", POINTS)
def test_axis_bounds(bounds, n):
    top, last = bounds[n]
    assert top <= n - 1 and last <= n - 2
    assert int(np.nextafter(np.float32(top), np.float32(np.inf))) > n - 1 or n <= 2 ** 24   # the largest such float
    if n <= 2 ** 24 + 1:
        assert (top, last) == (n - 1, n - 2)
