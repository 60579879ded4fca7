// Fixed-point arithmetic of the diagonal blocks (diag_tc.cu): numbers of at
// most 1 in magnitude as 64-bit integers with 61 fractional bits, their
// products from 32 x 32 -> 64 bit multiplications, a reciprocal square root,
// and the balanced base-512 digits that the tensor cores multiply.  Host and
// device code; no float64 instructions, no conversions on the float64 pipe.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace beor {

constexpr int FX_FRAC = 61;
constexpr long long FX_ONE = 1ll << FX_FRAC;
constexpr int FX_ND = 6;        // base-512 digits of a panel row's 54-bit integers
constexpr int FX_LEVELS = 7;    // digit-pair levels s + t = 0 .. 6

// a = h 2^31 + l, 0 <= l < 2^31 (|a| < 2^62)
struct fxs {
  int h, l;
};
__host__ __device__ __forceinline__ fxs fx_split(long long a) {
  return fxs{(int)(a >> 31), (int)(a & 0x7fffffff)};
}
// a b + c d of numbers with 61 fractional bits (b, d: 61 - S); |a + ic| <= 1,
// |b + id| <= 2^S.  The low halves' products are left out, at most 2^(S + 1)
// units of 2^-61 each.
template <int S = 0>
__host__ __device__ __forceinline__ long long fx_dot2(fxs a, fxs b, fxs c, fxs d) {
  const long long hh = (long long)a.h * b.h + (long long)c.h * d.h;
  const long long m = (long long)a.h * b.l + (long long)a.l * b.h + (long long)c.h * d.l + (long long)c.l * d.h;
  return hh * (2 << S) + (m >> (30 - S));
}
// a y with 61 fractional bits, y <= 2^S with 61 - S
template <int S>
__host__ __device__ __forceinline__ long long fx_mul(long long a, fxs y) {
  const fxs s = fx_split(a);
  const long long m = (long long)s.h * y.l + (long long)s.l * y.h;
  return (long long)s.h * y.h * (2 << S) + (m >> (30 - S));
}
__host__ __device__ __forceinline__ int fx_clz(unsigned long long v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
__host__ __device__ __forceinline__ unsigned long long fx_umulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ long long fx_mulhi(long long a, long long b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (long long)(((__int128)a * b) >> 64);
#endif
}
// v 2^-61 as three floats, |v| <= 2^61: exact, and each at most half an ulp of the
// one before.
__host__ __device__ __forceinline__ void fx_split3(long long v, float& hi, float& lo, float& t) {
  const float a = (float)(int)(v >> 38) * 0x1p-23f, b = (float)(int)((v >> 14) & 0xffffff) * 0x1p-47f;
  const float c = (float)(int)(v & 0x3fff) * 0x1p-61f;
  const float h = a + b;                     // a = 0 or |a| > |b|
  const float r = b - (h - a);
  const float l = r + c;
  const float rr = l - r;
  const float e = (r - (l - rr)) + (c - rr);
  hi = h + l;
  const float m = l - (hi - h);              // may have lost a binade against e
  lo = m + e;
  t = e - (lo - m);
}
// A positive number d <= 1 as D 2^(-2g), D in [1/4, 1) (g >= -1).
__host__ __device__ __forceinline__ long long fx_normalise(long long d, int& g) {
  g = (fx_clz((unsigned long long)d) - 3) >> 1;
  return g < 0 ? d >> 2 : d << (2 * g);
}
// 1 / D for D in [1/4, 1), with 59 fractional bits: a float32 estimate r0 and
// one third-order Newton step r0 (1 + e + e^2) with e = 1 - D r0 (|e| < 2^-21)
// formed to 2^-58.
__host__ __device__ __forceinline__ long long fx_recip(long long D) {
  const float f = (float)(int)(D >> 32) * 0x1p-29f;
#ifdef __CUDA_ARCH__
  float r0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(f));
#else
  const float r0 = 1.0f / f;
#endif
  const int rh = (int)(r0 * 0x1p28f);                        // exact: r0 >= 1 has 23 fractional bits
  const long long e = (1ll << 59) - (long long)fx_umulhi((unsigned long long)D << 2, (unsigned long long)rh << 32);
  const int e50 = (int)(e >> 9);
  const long long c = e + (((long long)e50 * e50) >> 41);    // 59 fractional bits
  return ((long long)rh << 31) + (fx_mulhi((long long)rh << 32, c << 22) >> 18);
}
// 1 / sqrt(D) for D in [1/4, 1), with 60 fractional bits: a float32 estimate y0
// and one third-order Newton step, y0 (1 + r / 2 + 3 r^2 / 8) with r = 1 - D
// y0^2 (|r| < 2^-20) formed to 2^-58.
__host__ __device__ __forceinline__ long long fx_rsqrt(long long D) {
  const float f = (float)(int)(D >> 32) * 0x1p-29f;
#ifdef __CUDA_ARCH__
  const float y0 = rsqrtf(f);
#else
  const float y0 = 1.0f / sqrtf(f);
#endif
  const int yh = (int)(y0 * 0x1p29f);                        // exact: y0 >= 1 has 23 fractional bits
  const unsigned long long y2 = (unsigned long long)yh * (unsigned long long)yh;   // 58 fractional bits
  const long long r = (1ll << 60) - (long long)fx_umulhi((unsigned long long)D << 2, y2 << 3);
  const int r50 = (int)(r >> 10);
  const long long rr = ((long long)r50 * r50) >> 40;
  const long long c = (r >> 1) + ((3 * rr) >> 3);            // 60 fractional bits
  return (((long long)yh << 32) + (fx_mulhi((long long)yh << 32, c << 22) >> 18) + 1) >> 1;
}

// l = sqrt(d) and 1 / l, both correctly rounded, of a normal d > 0, by integer
// operations: 53-bit candidates from the reciprocal square root above, then the
// sign of the exact remainder, whose magnitude leaves the low 64 bits of each
// product to decide it.  Half the latency of float64's square root and division.
__host__ __device__ __forceinline__ void fx_sqrt_rcp(long long bits, long long& l, long long& rinv) {
  const int e = (int)(bits >> 52) - 1023, odd = e & 1, h = (e - odd) / 2;
  const long long one = 1ll << 52;
  const long long m = ((bits & (one - 1)) | one) << odd;       // d = m 2^(2 h - 52), 2^52 <= m < 2^54
  const long long y = fx_rsqrt(m << 7);                        // 1 / sqrt(m 2^-54), 60 fractional bits
  const unsigned long long p = fx_umulhi((unsigned long long)m << 10, (unsigned long long)y << 2);
  long long s = (long long)((p + 256) >> 9);                   // sqrt(m 2^52), within 1 of its rounding
  const long long r = (long long)(((unsigned long long)m << 52) - (unsigned long long)s * (unsigned long long)s);
  s += (r > s) - (r <= -s);                                    // (s - 1/2)^2 < m 2^52 < (s + 1/2)^2
  l = ((long long)(h + 1023) << 52) + (s - one);
  long long t = y >> 8;                                        // 2^105 / s, within 2 of its rounding
  const long long q = 2 * -(long long)((unsigned long long)t * (unsigned long long)s);   // 2 (2^105 - t s)
  t += (q > s) + (q > 3 * s) - (q < -s) - (q < -3 * s);        // no ties: s would have to divide a power of two
  rinv = ((long long)(1022 - h) << 52) + (t - one);
}

// Balanced base-512 digits of X, |X| <= 2^53: X = sum_s d[s] 512^(5 - s),
// d[1..5] in [-256, 255], |d[0]| <= 256: each exact in bf16.
__host__ __device__ __forceinline__ void fx_digits(long long x, int* d) {
  const unsigned long long bias = 256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36));
  const unsigned long long t = (unsigned long long)x + bias;
  d[0] = (int)((long long)t >> 45);
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
  for (int s = 1; s < FX_ND; ++s) d[s] = (int)((t >> (9 * (FX_ND - 1 - s))) & 511) - 256;
}
// Sum of 32 products X X' in units of 2^50 (|.| < 2^62) from its levels s + t =
// 0 .. 6: level l is the integer sum of d[s] d'[t] over its pairs and the 32
// terms, at most 6 x 32 x 2^16 < 2^24 (exact in an fp32 accumulator).
__host__ __device__ __forceinline__ long long fx_levels(const int* a) {
  const int low = (((a[6] + 256) >> 9) + a[5] + 16) >> 5;
  return (long long)(low + a[4] * 16) + (long long)a[3] * 8192 + (long long)a[2] * 4194304 +
         (long long)a[1] * 2147483648ll + (long long)((unsigned long long)(unsigned)(a[0] * 256) << 32);
}

}  // namespace beor
