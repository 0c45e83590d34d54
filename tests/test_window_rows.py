"""The windows of a read, row by row (window_rows.h, as the kernels compile
it): every window once and no other, in as many rows as there are, up to the
largest read that a 32-bit length can state."""
from __future__ import annotations

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_1940_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "window_rows.h"
using namespace dbg;

static int rows_of(uint32_t cnt) {  // the loop of the kernels, by the lanes that take part
  const uint32_t rows = window_rows(cnt);
  if ((uint64_t)rows * 32 < cnt || (rows && (uint64_t)(rows - 1) * 32 >= cnt)) return 1;
  uint64_t seen = 0;
  for (uint32_t row = 0; row < rows; row++)
    for (uint32_t lane = row + 1 < rows ? 31 : 0; lane < 32; lane++) {
      const bool there = in_row(cnt, row, lane);
      if (there != ((uint64_t)row * 32 + lane < cnt)) return 2;
      seen += row + 1 < rows ? 32 : there;
    }
  return seen == cnt ? 0 : 3;
}

int main(int argc, char **argv) {
  for (int i = 1; i < argc; i++)
    if (int bad = rows_of((uint32_t)strtoull(argv[i], nullptr, 0))) {
      printf("%s: %d\n", argv[i], bad);
      return 1;
    }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    where = tmp_path_factory.mktemp("rows")
    src = where / "rows.cpp"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-O2", "-std=c++17", f"-I{CSRC}", str(src), "-o", str(where / "rows")])
    return str(where / "rows")


def test_windows_of_a_read(program):
    top = 1 << 32
    counts = [*range(0, 130), 1 << 31, *(top - d for d in (1, 2, 30, 31, 32, 33, 64, 65))]
    assert subprocess.run([program, *map(str, counts)], timeout=120).returncode == 0
