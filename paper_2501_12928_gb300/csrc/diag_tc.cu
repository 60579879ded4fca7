// Diagonal blocks of the mixed-precision factorisation: Cholesky factor,
// log-determinant and inverse of one 128 x 128 block per cluster of C CTAs
// (C = 1, 2 or 4), in one sweep of eight panels of 16 columns.
//
// What bounds it: the GPU's float64 pipe issues one warp instruction per ~19
// cycles and SM, with a latency of 67 cycles, so that the ~44,000 float64 warp
// instructions of a 128 x 128 complex Cholesky take 0.42 ms on the one SM that
// holds a block, and a float32-pipe inverse with compensated sums another 0.24
// ms: the chain of diagonal blocks was two thirds of a small evaluation.  Here
// no float64 arithmetic is left but the logarithms:
//
//  * The block is scaled by powers of two to unit diagonal, a~_il = a_il
//    2^(-e_i - e_l) with 2^(2 e_i) >= a_ii; for a positive definite block
//    |a~_il| <= 1, every Schur complement stays within it and |L~| <= 1, so
//    everything is 64-bit fixed point with 61 fractional bits: its rounding,
//    2^-61 of sqrt(a_ii a_ll), lies below the 2^-53 of a float64 accumulation.
//    Panels (16 x 16 diagonal factor, substitution of the rows below) use 32 x
//    32 -> 64 bit integer products (diag_fixed.cuh), about a fifth of the time
//    of float64 ones.
//  * A panel row of L~ is rounded to X = round(L~ 2^(55 - E)) with E two
//    powers of two above its largest component: at most 2^-53 of that
//    component, a float64 rounding.  X is cut into six balanced base-512
//    digits, exact in bf16.
//  * mma.sync m16n8k16 (two K steps of eight complex columns as [re | im])
//    multiplies the digits: 26 of the 36 digit pairs, s + t <= 6, each level s +
//    t in an fp32 accumulator that stays below 2^24 and is therefore exact; the
//    pairs dropped lie about 2^-60 below the rows' leading product.  The levels
//    are added as one 64-bit integer, shifted to the fixed point and
//    subtracted.
//  * The inverse grows in place: with Y the rows of Linv~ of this panel (16 x
//    16 substitution per column, double-float with exact triples of L, fp32
//    pipe), the rows below take B -= L~ Y by the same products (digits of Y
//    scaled per column, the 21 pairs s + t <= 5: 2^-51) into double-float
//    elements; column j of Linv~ takes the storage that column j of the block
//    no longer needs.  The three floats of an element of L are each at most half
//    an ulp of the one before, since the products of the lower ones are rounded
//    (cut at fixed bits instead, small elements brought errors of 2^-47 of the
//    row's largest into the inverse).
//  * Eight warps update and factor the next panel's diagonal while the others
//    do the rest of the rank-16 update.  The panel loops are kept rolled: a
//    warp alone runs straight-line code at the rate of instruction fetches
//    (6-8 cycles per instruction when they were unrolled).
//  * In a cluster, CTA r owns the rows of the 16-row blocks R = r (mod C): it
//    solves and updates them alone; the panel's factor and the digits of L~ and
//    Y go to every CTA through distributed shared memory, two cluster barriers
//    per panel.
//
// Measured per launch (3280 modes): 0.79 ms before (float64 factor, fp32
// inverse), now 0.181 ms with one problem (clusters of four), 0.225 ms with 64
// (clusters of two) and 0.295 ms with 100 (single CTAs).  Most of it is the
// chain of 128 columns in the panel factors and, between them, the
// substitutions; loading and output take 13 us.
//
// Accuracy against 113-bit arithmetic over 78 blocks (dense random ones of 5 to 128
// rows, condition 7 to 200, and blocks of drift scans, up to 3e6), as a fraction of
// the float64 factor's and its fp32 inverse's: largest backward error 0.13 to 0.21
// (at most 3e-16 of sqrt(a_ii a_ll)), rms error of L 0.23 to 0.79, of the inverse
// 0.12 to 0.63, of the log-determinant 0.09 to 0.79.
//
// tcgen05 is not used: its smallest tile (M = 64 or 128 of one CTA, operands
// by descriptor, accumulators in tensor memory) does not fit a triangle of
// 16 x 8 tiles with seven accumulators per component.
#include <cooperative_groups.h>

#include <cmath>

#include "diag_common.cuh"
#include "diag_fixed.cuh"

namespace beor {

namespace cg = cooperative_groups;

constexpr int DT_P = 16;                         // panel width and row block
constexpr int DT_NPAN = BEOR_TB / DT_P;
constexpr int DT_THREADS = 512;
constexpr int DT_WARPS = DT_THREADS / 32;
constexpr int DT_SLICE = BEOR_TB * 64;           // bytes of one digit of 128 rows x 32 (K)
constexpr int DT_ZERO_E = -400;                  // exponent of an all-zero column

struct DtSmem {
  longlong2 s[DG_PACK];        // packed lower: fixed point (columns not yet eliminated) or Linv~ as float4
  unsigned char dg[FX_ND * DT_SLICE];   // digits: row i of L~ (i below the panel) or column i of Y (up to the panel)
  int ex[BEOR_TB];             // their exponents
  int es[BEOR_TB];             // e_i
  int bad[BEOR_TB];            // row i cannot belong to a positive definite block
  int4 lp[DT_P][DT_P];         // panel diagonal factor L~: halves of (re, im)
  long long y[DT_P];           // reciprocals of its diagonal, y 2^g
  int g[DT_P];
  long long piv[BEOR_TB];      // pivots
  float4 lpf[DT_P][DT_P];      // -L~ of the panel diagonal as three floats per component
  float2 lpt[DT_P][DT_P];
  dfl rinvf[DT_P];
  longlong2 zb[2][DT_P];       // column of the running elimination step, by step parity
  long long pub[2];            // next diagonal element before that step
  double red[4];
  int fail;
  int tile;                    // next tile of the rank-16 update
};

// byte offset of 16-byte chunk (2 K step + component) of a row in one digit:
// 64 bytes per row, chunks permuted so that ldmatrix reads eight rows without
// bank conflicts
__device__ __forceinline__ int dt_off(int row, int chunk) { return row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4); }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
// 2^e as two factors (overflow and underflow apart, x * a * b is exact)
struct pow2 {
  float a, b;
};
__device__ __forceinline__ pow2 make_pow2(int e) {
  e = max(-250, min(250, e));
  const int h = e >> 1;
  return {pow2f(h), pow2f(e - h)};
}
__device__ __forceinline__ float scale2f(float x, pow2 p) { return x * p.a * p.b; }
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((e + 1023) << 20, 0); }
__device__ __forceinline__ long long shl64(long long x, int n) { return (long long)((unsigned long long)x << n); }
// round(x 2^e), |result| < 2^62, by integer operations (conversions to 64-bit
// integers run on the float64 pipe)
__device__ __forceinline__ long long fx_from_float(float x, int e) {
  const unsigned u = __float_as_uint(x);
  const int ex = (int)(u >> 23) & 255;
  const int m = ex ? (int)((u & 0x7fffffu) | 0x800000u) : 0;
  const int sh = ex - 150 + e;
  long long v = m;
  if (sh >= 0)
    v <<= min(sh, 39);
  else
    v = sh > -26 ? (v + (1ll << (-sh - 1))) >> -sh : 0;
  return (int)u < 0 ? -v : v;
}
// round(hi) + round(lo) of two scaled floats, |hi| < 2^53, |lo| < 2^30
__device__ __forceinline__ long long fx_from_scaled(float hi, float lo) {
  const int h1 = __float2int_rn(hi * 0x1p-29f);
  const int h0 = __float2int_rn(fmaf(-(float)h1, 0x1p29f, hi)) + __float2int_rn(lo);
  return (long long)h1 * 536870912ll + h0;
}
// v 2^e as a double-float (|v| < 2^62)
__device__ __forceinline__ dfl df_from_fixed(long long v, pow2 p) {
  const float a = (float)(int)(v >> 40) * 0x1p40f, b = (float)(int)((v >> 16) & 0xffffff) * 0x1p16f;
  const float c = (float)(int)(v & 0xffff);
  const dfl s = df_two_sum(a, b);
  const dfl t = df_fast_two_sum(s.hi, s.lo + c);
  return {scale2f(t.hi, p), scale2f(t.lo, p)};
}
__device__ __forceinline__ int abs_hi(long long x) { return (int)((x < 0 ? -x : x) >> 32); }

// Digits of two integers (K positions k, k + 1) as packed bf16 pairs.
__device__ __forceinline__ void dt_digits2(long long x0, long long x1, uint32_t* out) {
  int d0[FX_ND], d1[FX_ND];
  fx_digits(x0, d0);
  fx_digits(x1, d1);
#pragma unroll
  for (int s = 0; s < FX_ND; ++s) {
    // exact floats of small integers without conversion instructions; |d| <= 256 is exact in the high half
    const uint32_t f0 = __float_as_uint(__int_as_float(0x4B400000 + d0[s]) - 12582912.0f);
    const uint32_t f1 = __float_as_uint(__int_as_float(0x4B400000 + d1[s]) - 12582912.0f);
    out[s] = __byte_perm(f0, f1, 0x7632);
  }
}

__device__ __forceinline__ void dt_ldm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void dt_ldm2(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void dt_mma(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Both components of a 16 x 8 tile: the digit products up to level MAXL over
// both K steps, then each of the lane's four outputs as one integer per
// component.  With A = (Ar | Ai) along K, re takes (Br | sr Bi) and im takes
// (si Bi | Br), sr and si signs as bf16 sign masks.
template <int MAXL>
__device__ __forceinline__ void dt_product(uint32_t dg0, int arow, int brow, int lane, uint32_t sr, uint32_t si,
                                           long long* vre, long long* vim) {
  float acc[2][MAXL + 1][4];
#pragma unroll
  for (int l = 0; l <= MAXL; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[0][l][q] = acc[1][l][q] = 0.0f;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    uint32_t b[FX_ND][2];
    const uint32_t b0 = dg0 + dt_off(brow, 2 * u + ((lane >> 3) & 1)), a0 = dg0 + dt_off(arow, 2 * u + (lane >> 4));
#pragma unroll
    for (int t = 0; t < FX_ND; ++t) dt_ldm2(b[t], b0 + t * DT_SLICE);
#pragma unroll
    for (int s = 0; s < FX_ND; ++s) {
      uint32_t a[4];
      dt_ldm4(a, a0 + s * DT_SLICE);
#pragma unroll
      for (int t = 0; t < FX_ND; ++t)
        if (s + t <= MAXL) {
          dt_mma(acc[0][s + t], a, b[t][0], b[t][1] ^ sr);
          dt_mma(acc[1][s + t], a, b[t][1] ^ si, b[t][0]);
        }
    }
  }
#pragma unroll
  for (int comp = 0; comp < 2; ++comp)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int i[FX_LEVELS];
#pragma unroll
      for (int l = 0; l < FX_LEVELS; ++l) i[l] = l <= MAXL ? __float2int_rn(acc[comp][l <= MAXL ? l : 0][q]) : 0;
      (comp ? vim : vre)[q] = fx_levels(i);
    }
}

// The rank-16 update of tile (16 rows R, 8 columns cb) by panel pan: columns
// of the inverse (cb < 2 pan + 2) or of the block.
__device__ __forceinline__ void dt_update(DtSmem& sm, int pan, int R, int cb, int lane) {
  const int s0 = pan * DT_P;
  const uint32_t dg0 = (uint32_t)__cvta_generic_to_shared(sm.dg);
  const int arow = 16 * R + (lane & 15), brow = 8 * cb + (lane & 7);
  const uint32_t neg = 0x80008000u;
  const int i0 = 16 * R + (lane >> 2), c0 = 8 * cb + 2 * (lane & 3);
  long long vre[4], vim[4];
  if (cb < 2 * pan + 2) {   // B -= L Y
    dt_product<5>(dg0, arow, brow, lane, neg, 0u, vre, vim);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + (q & 2 ? 8 : 0), c = c0 + (q & 1);
      float4* f = reinterpret_cast<float4*>(&sm.s[pk(i, c)]);
      const pow2 ps = make_pow2(sm.ex[i] + sm.ex[c] - 60);
      const dfl wr = df_from_fixed(vre[q], ps), wi = df_from_fixed(vim[q], ps);
      const float4 o = c >= s0 ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : *f;   // the panel's own columns start at zero
      const dfl sr = df_two_sum(o.x, -wr.hi), si = df_two_sum(o.z, -wi.hi);
      const dfl nr = df_fast_two_sum(sr.hi, sr.lo + (o.y - wr.lo));
      const dfl ni = df_fast_two_sum(si.hi, si.lo + (o.w - wi.lo));
      *f = make_float4(nr.hi, nr.lo, ni.hi, ni.lo);
    }
  } else {                  // A -= L L^H
    dt_product<6>(dg0, arow, brow, lane, 0u, neg, vre, vim);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + (q & 2 ? 8 : 0), c = c0 + (q & 1);
      if (c > i) continue;
      const int sh = 60 - FX_FRAC - (sm.ex[i] + sm.ex[c]);   // -7 .. 53
      longlong2 o = sm.s[pk(i, c)];
      const long long half = sh > 0 ? 1ll << (sh - 1) : 0;
      const int rsh = max(sh, 0), lsh = max(-sh, 0);
      o.x -= shl64((vre[q] + half) >> rsh, lsh);
      o.y -= shl64((vim[q] + half) >> rsh, lsh);
      sm.s[pk(i, c)] = o;
      if (i == c && o.x <= 0) sm.bad[i] = 1;   // pivots only decrease from here on
    }
  }
}

__device__ __forceinline__ longlong2 dt_shfl2(longlong2 v, int src) {
  return make_longlong2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
// Column value z of a pivot D 2^(-2g) scaled by 2^g (|z~| = |L~| sqrt(D)).
// over: |z~| >= 1, impossible in a positive definite block; zero then.
__device__ __forceinline__ longlong2 dt_shift(longlong2 z, int g, bool& over) {
  const int gl = max(g, 0), gr = gl - g;   // g >= -1
  over = (max(abs_hi(z.x), abs_hi(z.y)) >> max(29 - gl, 0)) > 0;
  return over ? make_longlong2(0, 0) : make_longlong2(shl64(z.x >> gr, gl), shl64(z.y >> gr, gl));
}

template <int C>
__device__ __forceinline__ DtSmem* dt_peer(DtSmem& sm, int rank) {
  if constexpr (C == 1) return &sm;
  return cg::this_cluster().map_shared_rank(&sm, rank);
}
template <int C>
__device__ __forceinline__ void dt_sync() {
  if constexpr (C == 1)
    __syncthreads();
  else
    cg::this_cluster().sync();
}

// Factor of the 16 x 16 diagonal block of panel pan by eight warps of its
// owner: thread = element (row r, column c); a warp whose two rows have been
// pivots is done.  Square-root-free
// elimination, a_rc -= z~_r conj(z~_c) / D, so that only a reciprocal lies
// between two pivots (beside the products, which do not need it), and every
// thread forms the next pivot itself: one barrier per column.  The square
// roots follow for all columns at once.  The factor goes to every CTA.
constexpr int DT_FW = 8;   // warps
__device__ __forceinline__ void dt_fsync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * DT_FW) : "memory"); }
template <int C>
__device__ __forceinline__ void dt_factor(DtSmem& sm, float4* __restrict__ ws, int pan, int tid) {
  const int s0 = pan * DT_P, r = tid >> 4, c = tid & 15;
  longlong2 x = c <= r ? sm.s[pk(s0 + r, s0 + c)] : make_longlong2(0, 0);
  long long d = sm.s[pk(s0, s0)].x;
#pragma unroll 1
  for (int j = 0; j < DT_P; ++j) {
    if ((r | 1) < j) break;   // both rows of the warp have been pivots
    int g;
    const long long D = fx_normalise(d > 0 ? d : FX_ONE / 2, g);
    bool over;
    const longlong2 z = dt_shift(x, g, over);
    if (c == j && r > j) {
      x = z;
      sm.zb[j & 1][r] = z;
      if (over) sm.bad[s0 + r] = 1;
    }
    if (r == j + 1 && c == j + 1) sm.pub[j & 1] = x.x;
    // the warps with row j or rows below it
    asm volatile("bar.sync 2, %0;" ::"r"(32 * (DT_FW - j / 2)) : "memory");
    if (d <= 0 || sm.bad[s0 + j]) {
      if (r == DT_P - 1 && c < C) dt_peer<C>(sm, c)->fail = s0 + j + 1;
      break;
    }
    if (tid == 32 * DT_FW - 1) sm.piv[s0 + j] = d;
    // the reciprocal beside the products, which do not need it
    const longlong2* zb = sm.zb[j & 1];
    const longlong2 zn = zb[min(j + 1, DT_P - 1)], zr = zb[r], zc = zb[c];
    const long long pub = sm.pub[j & 1];
    const fxs w = fx_split(fx_recip(D));
    const fxs nx = fx_split(zn.x), ny = fx_split(zn.y);
    const fxs ar = fx_split(zr.x), ai = fx_split(zr.y), nr = fx_split(-zr.x);
    const fxs br = fx_split(zc.x), bi = fx_split(zc.y);
    const long long nn = fx_dot2(nx, nx, ny, ny), re = fx_dot2(ar, br, ai, bi), im = fx_dot2(ai, br, nr, bi);
    d = pub - fx_mul<2>(nn, w);
    if (c > j && c <= r) {
      if (c == r && re > D + (1ll << 45)) sm.bad[s0 + r] = 1;   // |L~_rj| > 1
      x.x -= fx_mul<2>(re, w);
      x.y -= fx_mul<2>(im, w);
    }
  }
  dt_fsync();   // every pivot is written
  if (sm.fail) return;
  if (tid < DT_P) {
    int g;
    const long long piv = sm.piv[s0 + tid];
    const long long y = fx_rsqrt(fx_normalise(piv, g));
    const dfl ri = df_from_fixed(y, make_pow2(g - 60));
#pragma unroll
    for (int q = 0; q < C; ++q) {
      DtSmem* o = dt_peer<C>(sm, q);
      o->y[tid] = y;
      o->g[tid] = g;
      o->piv[s0 + tid] = piv;
      o->rinvf[tid] = ri;
    }
  }
  dt_fsync();
  const pow2 pe = make_pow2(sm.es[s0 + r] - FX_FRAC);
  if (c < r) {
    const fxs y = fx_split(sm.y[c]);
    const longlong2 l = make_longlong2(fx_mul<1>(x.x, y), fx_mul<1>(x.y, y));
    // L~ y, 60 fractional bits: the multipliers of the rows below
    const fxs re = fx_split(fx_mul<0>(l.x, y)), im = fx_split(fx_mul<0>(l.y, y));
    float4 f;   // -L~
    float2 t;
    fx_split3(-l.x, f.x, f.y, t.x);
    fx_split3(-l.y, f.z, f.w, t.y);
#pragma unroll
    for (int q = 0; q < C; ++q) {
      DtSmem* o = dt_peer<C>(sm, q);
      o->lp[r][c] = make_int4(re.h, re.l, im.h, im.l);
      o->lpf[r][c] = f;
      o->lpt[r][c] = t;
    }
    const dfl lre = df_from_fixed(l.x, pe), lim = df_from_fixed(l.y, pe);
    ws[(s0 + c) * BEOR_TB + s0 + r] = make_float4(lre.hi, lre.lo, lim.hi, lim.lo);
  }
}

// Lanes per row of the rows below a panel: more where a CTA has fewer rows,
// while that shortens the chain (16 lanes with C = 4 took 3 % longer a block).
template <int C>
constexpr int dt_lpr() {
  return C == 1 ? 4 : 8;
}
// Rows below the panel, dt_lpr lanes per row (columns q, q + LPR, ..): substitution with the panel's factor, digits to
// every CTA, L to the workspace.
template <int C>
__device__ __forceinline__ void dt_solve(DtSmem& sm, float4* __restrict__ ws, int s0, int row, int lane) {
  constexpr int LPR = dt_lpr<C>(), NC = DT_P / LPR;
  const int q = lane & (LPR - 1);
  longlong2 x[NC];
  bool bad = sm.bad[row];
#pragma unroll
  for (int h = 0; h < NC; ++h) x[h] = sm.s[pk(row, s0 + q + LPR * h)];
#pragma unroll
  for (int h0 = 0; h0 < NC; ++h0) {
#pragma unroll 1
    for (int qj = 0; qj < LPR; ++qj) {
      const int j = h0 * LPR + qj;
      bool over;
      const longlong2 z = dt_shift(x[h0], sm.g[j], over);
      if (q == qj) {
        x[h0] = z;
        bad |= over;
      }
      const longlong2 zr = dt_shfl2(z, (lane & ~(LPR - 1)) | qj);
      const fxs ar = fx_split(zr.x), ai = fx_split(zr.y), nr = fx_split(-zr.x);
#pragma unroll
      for (int h = h0; h < NC; ++h) {
        const int c = q + LPR * h;
        if (c > j) {
          const int4 u = sm.lp[c][j];
          const fxs br{u.x, u.y}, bi{u.z, u.w};
          x[h].x -= fx_dot2<1>(ar, br, ai, bi);
          x[h].y -= fx_dot2<1>(ai, br, nr, bi);
        }
      }
    }
  }
#pragma unroll
  for (int h = 0; h < NC; ++h) {
    const fxs y = fx_split(sm.y[q + LPR * h]);
    x[h] = make_longlong2(fx_mul<1>(x[h].x, y), fx_mul<1>(x[h].y, y));
  }
  // largest component of the row by the high words; sum |L~_ij|^2 <= a~_ii <= 1
  // unless the block is not positive definite at this row: such a row (and one
  // whose diagonal has become negative) takes no further part, which also keeps
  // the fixed point in range
  int mx = 0;
  float n2 = 0.0f;
#pragma unroll
  for (int h = 0; h < NC; ++h) {
    const int a = abs_hi(x[h].x), b = abs_hi(x[h].y);
    mx = max(mx, max(a, b));
    n2 = fmaf((float)a, (float)a, fmaf((float)b, (float)b, n2));
  }
#pragma unroll
  for (int o = 1; o < LPR; o <<= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  }
  bad |= !(n2 <= 1.001f * 0x1p58f);
  constexpr unsigned GROUP = (1u << LPR) - 1u;
  if ((__ballot_sync(0xffffffffu, bad) >> (lane & ~(LPR - 1))) & GROUP) {
    bad = true;
#pragma unroll
    for (int h = 0; h < NC; ++h) x[h] = make_longlong2(0, 0);
    mx = 0;
  }
  if (bad && q == 0) sm.bad[row] = 1;
  // X = x 2^(53 - lb), all components below 2^lb
  const int lb = mx > 0 ? 64 - __clz(mx) : 32;
  const int rs = max(lb - 53, 0), ls = max(53 - lb, 0);
  const long long half = rs > 0 ? 1ll << (rs - 1) : 0;
  const pow2 pe = make_pow2(sm.es[row] - FX_FRAC);
  const int part = lane & 1;   // of a pair of columns, the even lane takes the real, the odd one the imaginary digits
#pragma unroll
  for (int h = 0; h < NC; ++h) {
    const int c = q + LPR * h;
    const long long got = __shfl_xor_sync(0xffffffffu, part ? x[h].x : x[h].y, 1);
    const long long x0 = part ? got : x[h].x, x1 = part ? x[h].y : got;
    uint32_t dg[FX_ND];
    dt_digits2(shl64((x0 + half) >> rs, ls), shl64((x1 + half) >> rs, ls), dg);
#pragma unroll
    for (int k = 0; k < C; ++k) {
      unsigned char* o = dt_peer<C>(sm, k)->dg + dt_off(row, 2 * (c >> 3) + part) + 4 * ((c & 7) >> 1);
#pragma unroll
      for (int d = 0; d < FX_ND; ++d) *reinterpret_cast<uint32_t*>(o + d * DT_SLICE) = dg[d];
    }
    const dfl re = df_from_fixed(x[h].x, pe), im = df_from_fixed(x[h].y, pe);
    ws[(s0 + c) * BEOR_TB + row] = make_float4(re.hi, re.lo, im.hi, im.lo);
  }
  if (q < C) dt_peer<C>(sm, q)->ex[row] = lb - 59;
}

constexpr int DT_IP = 4;   // lanes per sum
// The panel's rows of the inverse, column j, component comp (0 re, 1 im; the
// other component is the neighbouring lane's): Y = L_pp^-1 B, row by row, each
// sum over four lanes (one lane took 18,000 cycles a panel, the longest of the
// chain).  A
// CTA that does not own the rows keeps its columns of Y in its own copy too.
template <int C>
__device__ __forceinline__ void dt_inverse_rows(DtSmem& sm, int pan, int j, int part, int comp) {
  const int s0 = pan * DT_P, m0 = max(0, j - s0);   // rows above column j are zero
  DtSmem* own = dt_peer<C>(sm, pan % C);            // holds the rows
  const float sg = comp ? 1.0f : -1.0f;
  float mx = 0.0f;
  if (C > 1 && own != &sm && j < s0) {   // the column so far, all rows in flight at once
    float2 b[DT_P / DT_IP];
#pragma unroll
    for (int q = 0; q < DT_P / DT_IP; ++q)
      b[q] = reinterpret_cast<const float2*>(&own->s[pk(s0 + part * (DT_P / DT_IP) + q, j)])[comp];
#pragma unroll
    for (int q = 0; q < DT_P / DT_IP; ++q)
      reinterpret_cast<float2*>(&sm.s[pk(s0 + part * (DT_P / DT_IP) + q, j)])[comp] = b[q];
    __syncwarp();
  }
#pragma unroll 1
  for (int r = 0; r < DT_P; ++r) {
    dfl c0{j == s0 + r && !comp && !part ? 1.0f : 0.0f, 0.0f}, c1{0.0f, 0.0f};
    if (j < s0 && !part) {
      const float2 b = reinterpret_cast<const float2*>(&sm.s[pk(s0 + r, j)])[comp];
      c0 = dfl{b.x, b.y};
    }
#pragma unroll 2
    for (int m = m0 + part; m < r; m += DT_IP) {
      const float4 a = sm.lpf[r][m];
      const float2 at = sm.lpt[r][m];
      const float4 y = *reinterpret_cast<const float4*>(&sm.s[pk(s0 + m, j)]);
      const float yh = comp ? y.z : y.x, yl = comp ? y.w : y.y, zh = comp ? y.x : y.z, zl = comp ? y.y : y.w;
      dot2_acc3(c0, a.x, a.y, at.x, yh, yl);
      dot2_acc3(c1, sg * a.z, sg * a.w, sg * at.y, zh, zl);
    }
    dfl s = df_two_sum(c0.hi, c1.hi);
    s.lo += c0.lo + c1.lo;
#pragma unroll
    for (int o = 2; o < 2 * DT_IP; o <<= 1) {   // the same bits in every lane
      const dfl t{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.lo, o)};
      const dfl u = df_two_sum(s.hi, t.hi);
      s = dfl{u.hi, u.lo + (s.lo + t.lo)};
    }
    const dfl y = df_mul(df_fast_two_sum(s.hi, s.lo), sm.rinvf[r]);
    mx = fmaxf(mx, fabsf(y.hi));
    if (r >= m0 && !part) {
      reinterpret_cast<float2*>(&sm.s[pk(s0 + r, j)])[comp] = make_float2(y.hi, y.lo);
      if (C > 1 && own != &sm) reinterpret_cast<float2*>(&own->s[pk(s0 + r, j)])[comp] = make_float2(y.hi, y.lo);
    }
    __syncwarp();
  }
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  const bool zero = !(mx > 0x1p-120f);
  const int eu = zero ? DT_ZERO_E : ilogbf(mx) + 4;   // two powers of two of headroom; hi + lo may round up to one more
  const pow2 ps = zero ? pow2{0.0f, 0.0f} : make_pow2(55 - eu);
  // digits of the eight pairs of rows, two of them by each lane
  {
    const int p0 = part * 2;
    uint32_t dg[2][FX_ND];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      long long xv[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 2 * (p0 + q) + h;
        const float2 y = r >= m0 ? reinterpret_cast<const float2*>(&sm.s[pk(s0 + r, j)])[comp] : make_float2(0.0f, 0.0f);
        xv[h] = fx_from_scaled(scale2f(y.x, ps), scale2f(y.y, ps));
      }
      dt_digits2(xv[0], xv[1], dg[q]);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      unsigned char* o = dt_peer<C>(sm, c)->dg + dt_off(j, 2 * (p0 >> 2) + comp) + 4 * (p0 & 3);
#pragma unroll
      for (int d = 0; d < FX_ND; ++d) *reinterpret_cast<uint2*>(o + d * DT_SLICE) = make_uint2(dg[0][d], dg[1][d]);
    }
  }
  if (2 * part + comp < C) dt_peer<C>(sm, 2 * part + comp)->ex[j] = eu;
}

template <int C>
__global__ void __launch_bounds__(DT_THREADS, 1) diag_tc_kernel(BatchView v, int kg) {
  extern __shared__ __align__(16) unsigned char dt_raw[];
  DtSmem& sm = *reinterpret_cast<DtSmem*>(dt_raw);
  const int p = blockIdx.x / C, rank = blockIdx.x % C;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;   // this problem's block step
  if (k < 0 || k >= pr.nt) return;
  if (v.status[p] != 0) return;
  if (!BEOR_INBOUNDS(v.flags, pr.ws_off + (tri_index(k, k) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_DIAG_WS) ||
      !BEOR_INBOUNDS(v.flags, pr.dinv_off + (int64_t)(k + 1) * DG_PACK <= v.dinv_elems, BC_DIAG_DINV) ||
      !BEOR_INBOUNDS(v.flags, (int64_t)(p + 1) * BEOR_TB <= (int64_t)v.P * BEOR_TB, BC_DIAG_LINV))
    return;
  float4* ws = reinterpret_cast<float4*>(v.ws) + pr.ws_off + tri_index(k, k) * BEOR_TILE_ELEMS;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // scales: 2^(2 e_i) >= a_ii.  A row whose diagonal is not positive and
  // finite fails at its own column at the latest.
  if (tid < BEOR_TB) {
    const float d = ws[tid * BEOR_TB + tid].x;
    const bool ok = d > 0.0f && isfinite(d);
    sm.es[tid] = ok ? (ilogbf(d) + 2) >> 1 : 0;
    sm.bad[tid] = !ok;
  }
  if (tid == 0) sm.fail = 0;
  __syncthreads();
  // the rows of this CTA's blocks of 16
  for (int w = warp; w < BEOR_TB * (BEOR_TB / 16 / C) / 2; w += DT_WARPS) {
    const int c = (w % (BEOR_TB / 2)) * 2 + (lane >> 4), R = (w / (BEOR_TB / 2)) * C + rank, r = 16 * R + (lane & 15);
    if (r < c) continue;
    const float4 a = ws[c * BEOR_TB + r];
    const int sh = FX_FRAC - sm.es[r] - sm.es[c];
    const pow2 ps = make_pow2(sh);
    // |a_il| <= sqrt(a_ii a_ll) unless the block is not positive definite, which then shows at column r at the latest
    longlong2 x = make_longlong2(0, 0);
    if (fabsf(scale2f(a.x, ps)) <= 0x1.00001p61f && fabsf(scale2f(a.z, ps)) <= 0x1.00001p61f)
      x = make_longlong2(fx_from_float(a.x, sh) + fx_from_float(a.y, sh), fx_from_float(a.z, sh) + fx_from_float(a.w, sh));
    else
      sm.bad[r] = 1;
    sm.s[pk(r, c)] = x;
  }
  dt_sync<C>();   // every CTA's shared memory is ready for its peers
  if (warp < DT_FW && rank == 0) dt_factor<C>(sm, ws, 0, tid);

  for (int pan = 0; pan < DT_NPAN; ++pan) {
    const int s0 = pan * DT_P;
    dt_sync<C>();   // the panel's factor, the updated rows
    if (sm.fail) break;
    // own row blocks below the panel, WB warps each; then one warp per four columns of the panel's rows of the inverse
    const int first = pan + 1 + (rank - (pan + 1) % C + C) % C;   // first own block below the panel
    const int nblk = first < DT_NPAN ? (DT_NPAN - 1 - first) / C + 1 : 0;
    constexpr int LPR = dt_lpr<C>(), WB = LPR / 2;   // warps per block of 16 rows
    if (tid == 0) sm.tile = 0;
    if (warp < WB * nblk) {
      const int R = first + (warp / WB) * C;
      dt_solve<C>(sm, ws, s0, 16 * R + (warp % WB) * (DT_P / WB) + lane / LPR, lane);
    } else {
      for (int w = warp - WB * nblk; w / 4 * C + rank <= pan; w += DT_WARPS - WB * nblk)
        dt_inverse_rows<C>(sm, pan, 16 * (w / 4 * C + rank) + 4 * (w & 3) + (lane >> 3), (lane >> 1) & 3, lane & 1);
    }
    dt_sync<C>();   // digits and exponents
    if (pan + 1 == DT_NPAN) break;
    // rank-16 update of the own rows; the owner of the next panel first updates and factors its diagonal
    const bool next = (pan + 1) % C == rank;
    if (next && warp < DT_FW) {
      if (warp < 2) dt_update(sm, pan, pan + 1, 2 * pan + 2 + warp, lane);
      dt_fsync();
      dt_factor<C>(sm, ws, pan + 1, tid);
    }
    // the own tiles, 2 R + 2 of each block without the next diagonal's two, longest rows first
    for (;;) {
      int t = 0;
      if (lane == 0) t = atomicAdd(&sm.tile, 1);
      t = __shfl_sync(0xffffffffu, t, 0);
      int R = first + (nblk - 1) * C;
      while (R >= first && nblk > 0) {
        const int n = 2 * R + 2 - (R == pan + 1 ? 2 : 0);
        if (t < n) break;
        t -= n;
        R -= C;
      }
      if (R < first || nblk == 0) break;
      dt_update(sm, pan, R, t, lane);
    }
  }
  __syncthreads();
  if (sm.fail) {
    if (tid == 0 && rank == 0) v.status[p] = k * BEOR_TB + sm.fail;
    return;
  }

  // diagonal of L and the log-determinant, 2 sum ln L_jj over the real rows
  if (rank == 0 && tid < BEOR_TB) {
    const double l = sqrt((double)sm.piv[tid] * 0x1p-61) * pow2d(sm.es[tid]);
    const float lh = (float)l;
    ws[tid * BEOR_TB + tid] = make_float4(lh, (float)(l - (double)lh), 0.0f, 0.0f);
    double ld = k * BEOR_TB + tid < pr.n ? 2.0 * log(l) : 0.0;
    for (int o = 16; o > 0; o >>= 1) ld += __shfl_xor_sync(0xffffffffu, ld, o);
    if (lane == 0) sm.red[warp] = ld;
  }
  // Linv = Linv~ diag(2^-e_j) (float64) for the solves, and its rows'
  // exponents for the slices
  double2* dinv = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
  float4* Af = reinterpret_cast<float4*>(sm.s);
  for (int w = warp; w < BEOR_TB / C; w += DT_WARPS) {
    const int r = ((w >> 4) * C + rank) * 16 + (w & 15);
    float mx = 0.0f;
    for (int c = lane; c <= r; c += 32) {
      const int e = pk(r, c);
      const float4 f = Af[e];
      const pow2 ps = make_pow2(-sm.es[c]);
      const float4 g = make_float4(scale2f(f.x, ps), scale2f(f.y, ps), scale2f(f.z, ps), scale2f(f.w, ps));
      Af[e] = g;
      dinv[e] = make_double2((double)g.x + (double)g.y, (double)g.z + (double)g.w);
      mx = fmaxf(mx, fmaxf(fabsf(g.x), fabsf(g.z)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int e = mx > 0.0f ? ilogbf(mx) + 1 : -1000;
    if (lane == 0) {
      sm.ex[r] = e;
      v.linv_exp[(int64_t)p * BEOR_TB + r] = e;
    }
  }
  __syncthreads();
  if (tid == 0 && rank == 0) v.logdet_sigma[p] += ((sm.red[0] + sm.red[1]) + sm.red[2]) + sm.red[3];

  // slices of Linv's rows (B operand of the panel product L_ik = A_ik Linv^H):
  // work item (own block of 16 rows, K-chunk of 16); lane = (8-row group, K
  // half, row), 16-byte chunks of eight columns, a warp writing 512 contiguous
  // bytes of every plane
  for (int w = warp; w < 64 / C; w += DT_WARPS) {
    const int r = ((w >> 3) * C + rank) * 16 + (lane >> 4) * 8 + (lane & 7);
    linv_slice_chunk(v, p, Af, r, (w & 7) * 16 + ((lane >> 3) & 1) * 8, sm.ex[r]);
  }
}

template <int C>
static int dt_fit() {   // blocks that are factored at once
  static PerDevice<int> fit;
  return fit.get([] {   // once: the kernel's attribute, and the device's answer
    allow_smem<diag_tc_kernel<C>>((int)sizeof(DtSmem));
    return C == 1 ? device_sms() : max_clusters(diag_tc_kernel<C>, DT_THREADS, sizeof(DtSmem), C);
  });
}
template <int C>
static cudaError_t launch_dt(const BatchView& v, int k, cudaStream_t s, int prio) {
  dt_fit<C>();
  return launch_cluster(diag_tc_kernel<C>, dim3(C * v.P), dim3(DT_THREADS), sizeof(DtSmem), s, prio, C, v, k);
}

// Clusters of four CTAs per block, or of two, while the GPU holds the batch's at
// once (36 and 76 on a GB300), else single CTAs.
static int cluster_size(int active) { return active <= dt_fit<4>() ? 4 : active <= dt_fit<2>() ? 2 : 1; }
int diag_tc_ctas(int active) { return active * cluster_size(active); }

cudaError_t launch_diag_tc(const BatchView& v, int k, int active, cudaStream_t s, int prio) {
  switch (cluster_size(active)) {
    case 4: return launch_dt<4>(v, k, s, prio);
    case 2: return launch_dt<2>(v, k, s, prio);
    default: return launch_dt<1>(v, k, s, prio);
  }
}

}  // namespace beor
