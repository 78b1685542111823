"""The row of a matrix element by a multiplication (row_index.h) against the division, on the host.

The element-wise kernels of both amplitude solvers read the transposed element with it, so a row one too large is a
read outside the matrix.  Orders 1 to 300, all from 1600 to 2400 (the plain product first fails at 1649), and
a few up to the largest whose square is an int; every element of the matrix up to order 2400, the ones around row
ends above.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_16575_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "row_index.h"
static long long check(unsigned r, bool ends) {
  const unsigned magic = osv::row_magic(r);
  long long bad = 0;
  for (unsigned a = 0; a < r; a++)
    for (unsigned b = 0; b < r; b += ends && b + 1 < r ? r - 1 : 1) bad += osv::row_of(a * r + b, r, magic) != a;
  return bad;
}
int main() {
  long long bad = 0;
  for (unsigned r = 1; r <= 300; r++) bad += check(r, false);
  for (unsigned r = 1600; r <= 2400; r++) bad += check(r, false);
  for (unsigned r = 2401; r <= 5000; r++) bad += check(r, true);
  const unsigned large[] = {8191, 8192, 10007, 16384, 30011, 46337, 46340};
  for (unsigned r : large) bad += check(r, true);
  std::printf("%lld\n", bad);
}
"""


def test_row_of_equals_the_division(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "row.cpp", tmp_path / "row"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) == 0
