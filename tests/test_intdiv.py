"""The integer reciprocal and quotient (csrc/intdiv.cuh) against the host's IEEE division, bit for bit.

The same source is compiled for the host; the hardware seed is replaced by the host's single-precision
reciprocal moved by -2..2 units in the last place, twice the device seed's bound on either side, so the check
covers whatever seed the device takes.  Operands: random bits, mantissas at both ends of a binade, exponents at
the ends of the range, and every pair of special values.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_14941_gb300", "csrc")
MAIN = r"""
#include "intdiv.cuh"
#include <random>
using namespace chemgb;
int main() {
  std::mt19937_64 g(1);
  const unsigned long long F = 0xfffffffffffffull;
  auto same = [](double x, double y) { return dbits(x) == dbits(y) || (x != x && y != y); };
  auto bad = [&](double a, double b) { return !same(rcp_rn(b), 1.0 / b) || !same(div_rn(a, b), a / b); };
  const double sp[] = {0.0, 1.0, 3.0, 1e300, 1e-300, 1e-310, INFINITY, NAN, 5e-324, 0x1p-1022, 0x1p1022, 0x1p1023,
                       0x1.fffffffffffffp1021, 0x1.fffffffffffffp1022, 0x1.fffffffffffffp1023, 0x1.fffffffffffffp-1022};
  long wrong = 0;
  for (seed_ulps = -2; seed_ulps <= 2; ++seed_ulps) {
    for (double a : sp) for (double b : sp) wrong += bad(a, b) + bad(-a, b) + bad(a, -b);
    for (int i = 0; i < 600000; ++i) {
      unsigned long long u = g(), v = g();
      if (i % 3 == 1) u = (u & ~F) | (i % 2 ? g() % 64 : F - g() % 64);
      if (i % 5 > 2) v = (v & ~F) | (i % 2 ? g() % 64 : F - g() % 64);
      if (i % 4) u = (u & ~(0x7ffull << 52)) | ((0x3e0ull + g() % 64) << 52);
      if (i % 4) v = (v & ~(0x7ffull << 52)) | ((0x3e0ull + g() % 64) << 52);
      wrong += bad(bitsd(u), bitsd(v)) + bad(bitsd(u), bitsd(u));
    }
  }
  return wrong != 0;
}
"""


def test_reciprocal_and_quotient_are_the_ieee_ones(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
