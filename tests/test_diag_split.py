"""The three floats of a fixed-point element (diag_fixed.cuh): an exact sum whose parts
do not overlap, for elements of every magnitude."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_12928_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "diag_fixed.cuh"
using namespace beor;

static long bad = 0;
static float ulp(float x) { return std::nextafter(std::fabs(x), INFINITY) - std::fabs(x); }
static void check(long long v) {
  float hi, lo, t;
  fx_split3(v, hi, lo, t);
  // every part is a whole number of 2^-61
  const __int128 sum = (__int128)std::ldexp((double)hi, 61) + (__int128)std::ldexp((double)lo, 61) + (__int128)std::ldexp((double)t, 61);
  if (sum != v || (lo != 0.0f && std::fabs(lo) > 0.5f * ulp(hi)) || (t != 0.0f && std::fabs(t) > 0.5f * ulp(lo))) ++bad;
}
int main() {
  const long long one = 1ll << 61;
  for (long long v : {0ll, one, -one}) check(v);
  for (int e = 0; e <= 61; ++e)
    for (int k = 0; k <= 61; ++k)
      for (long long s : {1ll, -1ll})
        for (long long d : {-1ll, 0ll, 1ll}) {
          const long long v = s * (1ll << e) + (k < e ? 1ll << k : 0) + d;
          if (v >= -one && v <= one) check(v);
        }
  std::mt19937_64 g(1);
  for (int i = 0; i < 2000000; ++i) check(((long long)g() >> 2) >> (g() % 62));
  std::printf("%ld\n", bad);
}
"""


def test_three_floats(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = tmp_path / "split.cpp"
    src.write_text("#define __host__\n#define __device__\n#define __forceinline__ inline\n" + PROGRAM)
    exe = tmp_path / "split"
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip() == "0"
