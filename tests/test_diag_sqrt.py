"""Correctly rounded square root and reciprocal from integers (diag_fixed.cuh)
against the host's float64 sqrt and division, bit for bit: every exponent, powers
of two and their neighbours, squares and their neighbours (the closest calls),
and random mantissas."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_12928_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "diag_fixed.cuh"
using namespace beor;

static long bad = 0;
static void check(long long bits) {
  if (bits < (1ll << 52) || bits >= (2047ll << 52)) return;
  double d, l, r;
  memcpy(&d, &bits, 8);
  long long lb, rb;
  fx_sqrt_rcp(bits, lb, rb);
  memcpy(&l, &lb, 8);
  memcpy(&r, &rb, 8);
  if (l != std::sqrt(d) || r != 1.0 / std::sqrt(d)) ++bad;
}
int main() {
  std::mt19937_64 g(1);
  const long long one = 1ll << 52;
  for (long long e = 1; e < 2047; ++e)
    for (long long k = -70; k <= 70; ++k) check((e << 52) + k);
  for (int i = 0; i < 3000000; ++i) {
    check((long long)(g() >> 1));
    check((1022 + (long long)(g() & 3)) * one + (long long)(g() & (one - 1)));
    // squares of 27 to 53 bits, rounded, and their neighbours
    const double s = std::ldexp((double)((g() >> 11) | (1ull << 52)), -52 + (int)(g() & 1));
    const double w = i & 1 ? s : std::ldexp(std::floor(std::ldexp(s, 26)), -26);
    const double sq = w * w;
    long long b;
    memcpy(&b, &sq, 8);
    for (long long k = -2; k <= 2; ++k) check(b + k);
    const double rc = 1.0 / w, rs = rc * rc;   // reciprocals near a rounding boundary
    memcpy(&b, &rs, 8);
    for (long long k = -2; k <= 2; ++k) check(b + k);
  }
  printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_square_root_and_reciprocal(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text("#define __host__\n#define __device__\n#define __forceinline__ inline\n" + PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
