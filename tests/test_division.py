"""The index divisions by reciprocal (csrc/ptt_div.h, host arithmetic, no GPU): fdiv
is exact where index times divisor stays below 2^32, fdiv_any for every index of the
3D energy sum (Me nx/2 nz values, divisor nx/2 nz) of every admitted shape."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_09468_gb300", "csrc")

# A quotient by reciprocal is never low and grows with the index, so it is exact
# on a row [j d, (j + 1) d) when it is at the row's first and last index.
DRIVER = r"""
#include <cstdio>
#include <set>
#include "ptt_div.h"
using namespace ptt;
static bool smooth(unsigned n) {
  for (unsigned p : {2u, 3u, 5u, 7u, 11u, 13u}) while (n % p == 0) n /= p;
  return n == 1;
}
int main() {
  const unsigned rows = 1080;   // the longest energy grid
  std::set<unsigned> ds;
  for (unsigned nx = 8; nx <= 512; nx += 2)
    for (unsigned nz = 4; nz <= 512; nz += 2)
      if (smooth(nx) && smooth(nz)) ds.insert(nx / 2 * nz);
  unsigned any = 0, plain = 0, checked = 0, over = 0;
  for (unsigned d : ds) {
    const FastDiv f = fast_div(d);
    for (unsigned j = 0; j < rows; ++j)
      for (unsigned i : {j * d, j * d + d - 1}) {
        ++checked;
        if (fdiv_any(i, f, d) != j) ++any;
        if (fdiv(i, f) != j) { ++plain; if ((unsigned long long)i * d < (1ull << 32)) ++over; }
      }
  }
  for (unsigned d = 1; d <= 2048; ++d) {   // fdiv within its bound, at every row's ends
    const FastDiv f = fast_div(d);
    for (unsigned long long j = 0; j * d * d < (1ull << 32) && j < (1u << 21); ++j) {
      const unsigned long long e = j * d + d - 1;
      ++checked;
      if (fdiv((unsigned)(j * d), f) != j || (e * d < (1ull << 32) && fdiv((unsigned)e, f) != j)) ++over;
    }
  }
  std::printf("%u %u %u %u\n", any, plain, over, checked);
}
"""


def test_index_divisions(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "div.cpp", tmp_path / "div"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    wrong_any, wrong_plain, wrong_within, checked = [
        int(v) for v in subprocess.run([str(exe)], text=True, capture_output=True, check=True).stdout.split()]
    assert checked > 10 ** 6
    assert wrong_any == 0 and wrong_within == 0
    assert wrong_plain > 0      # the plain quotient does fail there: the sum needs the other one
