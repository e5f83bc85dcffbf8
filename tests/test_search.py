"""The reduction's search in a sorted row and its check of a row's offsets
(csrc/cg_search.h), compiled for the host: every column of rows at the first,
middle and last entries that the call accepts (2^31 - 1 of them), with a column
reader that refuses any index outside the row, and offsets at the same bounds. No
graph of that size is made."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_04350_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "cg_search.h"
// Columns 3, 5, 7, ... of the row [a, b); any other index ends the program.
struct Row {
  int32_t a, b;
  int32_t operator[](int32_t i) const {
    if (i < a || i >= b) {
      std::printf("read of entry %d outside [%d, %d)\n", (int)i, (int)a, (int)b);
      std::exit(1);
    }
    return 2 * (i - a) + 3;
  }
};
int main(int argc, char** argv) {
  if (argc == 6)
    return cg::row_ok(std::atoll(argv[1]), std::atoll(argv[2]), std::atoll(argv[3]), std::atoll(argv[4]),
                      (int32_t)std::atoll(argv[5])) ? 0 : 1;
  const Row r{(int32_t)std::atoll(argv[1]), (int32_t)std::atoll(argv[2])};
  for (int32_t w = 0; w <= 2 * (r.b - r.a) + 4; ++w) {
    const bool in = w >= 3 && (w & 1) && (w - 3) / 2 < r.b - r.a;
    const int32_t want = in ? r.a + (w - 3) / 2 : -1, got = cg::find_col(r, r.a, r.b, w);
    if (got != want) {
      std::printf("column %d: %d, not %d\n", (int)w, (int)got, (int)want);
      return 1;
    }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("search")
    (d / "search.cpp").write_text(PROGRAM)
    exe = str(d / "search")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, str(d / "search.cpp")], check=True)
    return exe


@pytest.mark.parametrize("a,length", [
    (0, 0), (0, 1), (0, 9), (5, 1000), ((1 << 30) - 4, 8), (1 << 30, 1), (1_200_000_000, 8), (1_200_000_000, 4097),
    ((1 << 31) - 1 - 8, 8), ((1 << 31) - 1 - 5000, 5000), ((1 << 31) - 1, 0)])
def test_every_column_of_a_row(program, a, length):
    r = subprocess.run([program, str(a), str(a + length)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("a,b,m,n,length,ok", [
    (0, 0, 0, 1, 1, True), (0, 3, 8, 4, 1, True), (5, 8, 8, 4, 9, True), (0, 3, 8, 4, 0, False),
    (-1, 2, 8, 4, 1, False), (4, 3, 8, 4, 1, False), (6, 9, 8, 4, 1, False),
    (0, 4, 8, 4, 1, False), (0, 1, 8, 1, 1, False),                     # as many entries as reads
    (0, (1 << 31) - 1, (1 << 31) - 1, 1, 1, False), (0, (1 << 31) - 1, (1 << 31) - 1, (1 << 30) - 1, 1, False),
    (1 << 30, (1 << 31) - 2, (1 << 31) - 1, (1 << 30) - 1, 1, True)])
def test_rows_a_read_can_have(program, a, b, m, n, length, ok):
    r = subprocess.run([program, str(a), str(b), str(m), str(n), str(length)])
    assert (r.returncode == 0) == ok
