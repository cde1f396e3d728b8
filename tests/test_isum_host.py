"""Host check of the FP64 arithmetic on integer units (csrc/mg_isum.hpp): compiled with g++, every
sum of six and every product with 1/6 that the integer forms accept equals the host's own binary64
operations bit for bit -- random mantissas, short ones (many ties), exponents together and up to
40 binary orders apart, cancellation, near-equal values, both ends of the exponent range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_2403_12179_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "mg_isum.hpp"
using namespace gbmg;
using namespace gbmg::bits;
static long fails = 0, simple = 0, general = 0, sums = 0, products = 0, taken = 0;
static volatile double sixth = 1.0 / 6.0;
static void check_sum(const double (&v)[6], int mode) {
  volatile double s = v[0];
  for (int i = 1; i < 6; ++i) s = s + v[i];
  const double ref = s;
  ++sums;
  const isum::Six q = isum::six_of(v);
  double o;
  if (isum::six_simple(q)) {
    ++simple;
    o = isum::sum6_simple(v, q);
    if (d2u(o) != d2u(ref) && fails++ < 10) std::printf("simple, mode %d: %a vs %a\n", mode, o, ref);
  }
  if (isum::sum6(v, q, &o)) {
    ++general;
    if (d2u(o) != d2u(ref) && fails++ < 10) std::printf("sum, mode %d: %a vs %a\n", mode, o, ref);
  }
}
static void check_mul(double t) {
  double o;
  ++products;
  if (!isum::mul_sixth(t, &o)) return;
  ++taken;
  const double ref = t * sixth;
  if (d2u(o) != d2u(ref) && fails++ < 10) std::printf("product %a: %a vs %a\n", t, o, ref);
}
int main() {
  std::mt19937_64 g(20260801);
  for (int mode = 0; mode < 9; ++mode)
    for (long it = 0; it < 400000; ++it) {
      double v[6];
      const int e0 = mode == 7 ? (int)(g() % 2047) : 1000;
      for (int i = 0; i < 6; ++i) {
        uint64_t m = g() & 0xFFFFFFFFFFFFFull;
        if (mode & 1) m &= ~0ull << (g() % 53);  // short mantissas: ties
        if ((mode == 2 || mode == 3) && (g() & 1)) m = (g() & 1) ? 0xFFFFFFFFFFFFFull : m >> 50;
        int spread = mode < 3 ? 7 : mode == 3 ? 12 : mode == 4 ? 33 : mode == 7 ? 40 : 20;
        if (mode != 7 && (g() & 3) == 0) spread = 1;
        int e = e0 - (int)(g() % spread);
        e = e < 0 ? 0 : e;
        const uint64_t sign = mode == 0 || mode == 8 ? 0 : g() & 1;
        v[i] = u2d(sign << 63 | (uint64_t)e << 52 | m);
        if (mode == 5 && i && g() % 3 == 0) v[i] = -v[i - 1];
        if (mode == 6 && i) v[i] = u2d(d2u(v[0]) + (int64_t)(g() % 9) - 4) * ((g() & 1) ? 1 : -1);
        if (mode == 8 && g() % 50 == 0) v[i] = g() & 1 ? 0.0 : -0.0;
      }
      check_sum(v, mode);
      check_mul(v[0]);
    }
  for (int e = 0; e < 2048; ++e)
    for (uint64_t m : {0ull, 1ull, 2ull, 3ull, 0x8000000000000ull, 0x7FFFFFFFFFFFFull, 0x8000000000001ull,
                       0xFFFFFFFFFFFFFull, 0xFFFFFFFFFFFFEull, 0xFFFFFFFFull, 0x100000000ull})
      for (uint64_t sign : {0ull, 1ull}) check_mul(u2d(sign << 63 | (uint64_t)e << 52 | m));
  std::printf("fails %ld sums %ld simple %ld general %ld products %ld taken %ld\n", fails, sums, simple,
              general, products, taken);
  return fails ? 1 : 0;
}
"""


def test_integer_forms_equal_host_arithmetic(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "isum_check.cpp", tmp_path / "isum_check"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", HDR, str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    n = dict(zip(out.stdout.split()[::2], map(int, out.stdout.split()[1::2])))
    assert n["simple"] > 200_000 and n["general"] > n["sums"] // 2 and n["taken"] > n["products"] // 2
