"""Every transform length of every admitted shape has a plan: the radices of the
factorisation multiply to the length, and each fixed-point pass's butterflies
fit the threads that run them (256, two of radix 2 or 3 each).  The library's
plan functions are host code (csrc/ptt_plan.h): compiled here, no GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_09468_gb300", "csrc")

# reads "fixed-point three-first n" per line, writes the library's verdict and the radices
DRIVER = r"""
#include <cstdio>
#include "ptt_plan.h"
int main() {
  int fx, three, n;
  while (std::scanf("%d %d %d", &fx, &three, &n) == 3) {
    const ptt::HostPlan p = fx ? ptt::make_plan_fx(n, three != 0) : ptt::make_plan(n, three != 0);
    std::printf("%d", ptt::plan_ok(p, fx != 0) ? 1 : 0);
    for (int r : p.radix) std::printf(" %d", r);
    std::printf("\n");
  }
}
"""


def _smooth(n, primes):
    for p in primes:
        while n % p == 0:
            n //= p
    return n == 1


def _next(n, even):
    while (even and n % 2) or not _smooth(n, (2, 3, 5)):
        n += 1
    return n


def _lengths():
    """(fixed point, three first, n) of every admitted nx, ny, nz (include/ptt.h)."""
    out = set()
    for n in range(4, 513, 2):        # nx (from 8) and nz (from 4): n and its padded length
        if _smooth(n, (2, 3, 5, 7, 11, 13)):
            pad = _next(3 * n // 2 - 2, False)
            out |= {(1, 0, n), (1, 1, pad), (0, 1, pad)}
    for ny in range(9, 514):
        if _smooth(ny - 1, (2, 3, 5, 7, 11, 13)):
            M, Me = _next((3 * ny - 1) // 2, True), _next(2 * ny - 1, True)
            out |= {(1, 0, 2 * (ny - 1)), (1, 0, M), (0, 0, M), (1, 0, Me), (0, 0, Me)}
    return sorted(out)


def test_every_admitted_length_has_a_plan(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "plans.cpp", tmp_path / "plans"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    lengths = _lengths()
    assert {810, 882, 972, 990} <= {n for _, _, n in lengths} and max(lengths)[2] <= 1080
    res = subprocess.run([str(exe)], input="\n".join("%d %d %d" % q for q in lengths), text=True,
                         capture_output=True, check=True).stdout.splitlines()
    assert len(res) == len(lengths)
    for (fx, three, n), line in zip(lengths, res):
        ok, *radix = [int(v) for v in line.split()]
        prod = 1
        for r in radix:
            prod *= r
        assert ok == 1 and prod == n and len(radix) <= 8, (fx, three, n, radix)
        assert set(radix) <= ({2, 3, 4, 5, 6, 7, 8, 11, 13} if fx else {2, 3, 4, 5, 8}), (fx, n, radix)
        if fx:
            assert all(n // r <= (512 if r <= 3 else 256) for r in radix), (n, radix)
