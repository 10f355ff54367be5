"""When a workspace may be asked to grow: the decision that keeps a call which
could use more memory from giving up what it has (the overlapped sites' second
set of buffers). Compiled for the host from the library's header."""
import subprocess

import pytest

from paper_2303_06150_gb300 import build

MB, GB = 1 << 20, 1 << 30
# bytes, cap, free, limit, fits
CASES = [
    (100 * MB, 100 * MB, 0, 0, 1),             # already there: nothing is asked of the device
    (100 * MB + 1, 100 * MB, 0, 0, 0),
    (10 * GB, 0, 12 * GB, 0, 1),               # 11.25 GB + 1 MB
    (10 * GB, 0, 11 * GB, 0, 0),
    (10 * GB, 5 * GB, 7 * GB, 0, 1),           # the old one is given back first
    (10 * GB, 5 * GB, 6 * GB, 0, 0),
    (140 * GB, 150 * GB, 0, 0, 1),
    (280 * GB, 140 * GB, 100 * GB, 0, 0),      # two sets on a device that holds one
    (10 * GB, 0, 100 * GB, 10 * GB - 1, 0),    # over the limit
    (10 * GB, 0, int(10.5 * GB), 10 * GB, 1),  # the limit caps the head room
    (10 * GB, 20 * GB, 0, 9 * GB, 0),          # over a limit set after it had grown
    (8 * MB, 0, 10 * MB, 0, 1),                # exactly the pages
    (8 * MB + 8, 0, 10 * MB, 0, 0),            # one byte past the pages
]

MAIN = r"""
#include <cstdio>
#include "internal.h"
int main() {
  size_t bytes, cap, free, limit;
  while (scanf("%zu %zu %zu %zu", &bytes, &cap, &free, &limit) == 4)
    printf("%d\n", (int)ligen::workspace_fits(bytes, cap, free, limit));
}
"""


@pytest.fixture(scope="module")
def answers(tmp_path_factory):
    d = tmp_path_factory.mktemp("workspace_room")
    (d / "main.cu").write_text(MAIN)
    subprocess.run([build.NVCC, "-std=c++17", *build.ARCH, "-I", build.CSRC, str(d / "main.cu"), "-o", str(d / "main")],
                   check=True, capture_output=True)
    text = "\n".join(" ".join(map(str, c[:4])) for c in CASES)
    out = subprocess.run([str(d / "main")], input=text, check=True, capture_output=True, text=True).stdout
    return [int(v) for v in out.split()]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_workspace_fits(answers, k):
    assert answers[k] == CASES[k][4]
