"""The fixed-point arithmetic of the diagonal blocks (diag_fixed.cuh), checked
on the host against 128-bit integers and long double.

Bounds: the reciprocal and the reciprocal square root form their residuals to
2^-58 and round to 2^-59 and 2^-60 of a result of at least 1, so their
relative errors stay below 2^-56; the products leave out one 31 x 31 bit
product per factor pair, (2^31)^2 in units of 2^(61 - S): 2^(S + 1) units of
2^-61 each, and truncate once; the
digit pairs left out of a 32-term product (s + t >= 7) are at most 4 x 32 x
2^16 x 2^27 = 1 unit of 2^50 at s + t = 7, with 2^-8 of that below, and the
level sum rounds twice (below 1 unit together), so it stays within 3 units for
any number; every level stays below 2^24."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_12928_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "diag_fixed.cuh"
using namespace beor;
typedef __int128 i128;

int main() {
  std::mt19937_64 g(1);
  long bad = 0;
  // reciprocals over every scale, 1 and the powers of two included
  for (int it = 0; it < 400000; ++it) {
    long long d = (long long)((g() >> 2) >> (g() % 61));
    if (it < 62) d = 1ll << it;
    if (d <= 0 || d > FX_ONE) continue;
    int e;
    const long long D = fx_normalise(d, e);
    if (D < FX_ONE / 4 || D >= FX_ONE || (e >= 0 ? d << (2 * e) : d >> 2) != D) ++bad;
    const long long y = fx_rsqrt(D), w = fx_recip(D);
    const long double x = ldexpl((long double)D, -61);
    const long double r = ldexpl((long double)y, -60) * sqrtl(x) - 1.0L, q = ldexpl((long double)w, -59) * x - 1.0L;
    if (fabsl(r) > 0x1p-56L || y < (1ll << 60) || y > (1ll << 61)) ++bad;
    if (fabsl(q) > 0x1p-56L || w < (1ll << 59) || w > (1ll << 61)) ++bad;
    if (it < 62 && (r != 0.0L || q != 0.0L) && it % 2 == 1) ++bad;   // powers of four: exact
  }
  for (int it = 0; it < 400000; ++it) {
    const long double p = 6.2831853L * (g() % 1000003) / 1000003.0L, q = 6.2831853L * (g() % 1000003) / 1000003.0L;
    const long double ra = (g() % 1001) / 1000.0L, rb = ldexpl(1.0L, -(int)(g() % 60));
    const long long a = llrintl(ldexpl(cosl(p) * ra, 61)), c = llrintl(ldexpl(sinl(p) * ra, 61));
    const long long b = llrintl(ldexpl(cosl(q) * rb, 61)), d = llrintl(ldexpl(sinl(q) * rb, 61));
    const i128 want = (i128)a * b + (i128)c * d;
    i128 err = ((i128)fx_dot2(fx_split(a), fx_split(b), fx_split(c), fx_split(d)) << 61) - want;
    if (err > (i128)5 << 61 || -err > (i128)5 << 61) ++bad;
    err = ((i128)fx_dot2<1>(fx_split(a), fx_split(b), fx_split(c), fx_split(d)) << 60) - want;
    if (err > (i128)9 << 60 || -err > (i128)9 << 60) ++bad;
    const long long y = (1ll << 60) + (long long)(g() >> 4), w = (1ll << 59) + (long long)((g() >> 5) * 3);
    err = ((i128)fx_mul<1>(a, fx_split(y)) << 60) - (i128)a * y;
    if (err > (i128)5 << 60 || -err > (i128)5 << 60) ++bad;
    err = ((i128)fx_mul<2>(a, fx_split(w)) << 59) - (i128)a * w;
    if (err > (i128)9 << 59 || -err > (i128)9 << 59) ++bad;
  }
  for (int it = 0; it < 60000; ++it) {
    int acc[FX_LEVELS] = {0};
    i128 want = 0;
    for (int k = 0; k < 32; ++k) {
      long long x = (long long)(g() % ((1ull << 54) + 1)) - (1ll << 53), y = (long long)(g() % ((1ull << 54) + 1)) - (1ll << 53);
      if (it == 0) x = y = 1ll << 53;
      if (it == 1) x = -(1ll << 53), y = -x;
      if (it == 2) x = y = 256ll * (1 + (1ll << 9) + (1ll << 18) + (1ll << 27) + (1ll << 36)) * -1;   // every digit -256
      if (it % 3 == 2 && it > 2) x >>= g() % 53, y >>= g() % 53;
      int dx[FX_ND], dy[FX_ND];
      fx_digits(x, dx);
      fx_digits(y, dy);
      long long rx = 0;
      for (int s = 0; s < FX_ND; ++s) {
        rx = rx * 512 + dx[s];
        if (abs(dx[s]) > 256) ++bad;
      }
      if (rx != x) ++bad;
      want += (i128)x * y;
      for (int s = 0; s < FX_ND; ++s)
        for (int t = 0; t < FX_ND; ++t)
          if (s + t < FX_LEVELS) acc[s + t] += dx[s] * dy[t];
    }
    for (int i = 0; i < FX_LEVELS; ++i) bad += abs(acc[i]) >= (1 << 24);
    const i128 got = (i128)fx_levels(acc) << 50, tol = (i128)3 << 50;
    if (got - want > tol || want - got > tol) ++bad;
  }
  std::printf("mismatches %ld\n", bad);
  return bad != 0;
}
"""


def test_fixed_point_arithmetic_of_the_diagonal_blocks(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "fixed.cu", tmp_path / "fixed"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True,
                   timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
