// Diagonal blocks of the float64 path and of the posterior mean: Cholesky
// factor, log-determinant and inverse of one 128 x 128 block on a cluster of C
// CTAs.  Every element sees the operations of the column by column factorisation
// and of the row by row inverse in one fixed order, so that the results do not
// depend on C, bit for bit (a posterior mean moves by 5e-8 with any other
// rounding of its factor).  The posterior mean's inverse is formed on the fp32
// pipe.
//
// What bounds it: one SM issues a float64 warp instruction every 19 cycles, so
// that a block's 44,000 take 0.42 ms there; the chain of 128 pivots takes 0.06 ms
// on any number of SMs (their square roots and reciprocals from integers, 450
// cycles a pair; 1,000 with float64's).  The
// rows are dealt to the CTAs in blocks of eight (zigzag, so that each has short
// and long ones); per panel of 16 columns every CTA factors the 16 x 16
// diagonal (the same operations everywhere, cheaper than an exchange per
// column), solves its rows and sends them to every CTA, and updates its rows.
// The inverse goes by columns, which do not depend on each other, from the copy
// of L that every CTA then has.  One point of 3280 modes, one CTA with barriers
// per column -> eight: float64 1.16 ms -> 0.39 per block, posterior mean 0.79 ->
// 0.33; with the pivots' square roots and reciprocals from integers 0.35 and
// 0.30; with the posterior mean's 32 x 32 inverses dealt by columns 0.28.
#include <cooperative_groups.h>

#include <cmath>
#include <type_traits>

#include "diag_common.cuh"
#include "diag_fixed.cuh"

namespace beor {

namespace cg = cooperative_groups;

constexpr int DC_P = 16;                     // panel width
constexpr int DC_THREADS = 512;
constexpr int DC_WARPS = DC_THREADS / 32;
constexpr int DC_NB = BEOR_TB / 8;           // blocks of eight rows

struct DcCommon {
  double rinv[DC_P];             // reciprocals of the panel's diagonal
  double pub;                    // next diagonal element before the running step
  double red[4];
  dfl invs[BEOR_TB];             // mixed: 1 / L_ii
  double dinvs[BEOR_TB];         // float64: 1 / L_ii
  float rmax[8][BEOR_TB];        // mixed: row maxima of each CTA's columns
  int ex[BEOR_TB];
  int fail;
};
template <bool MIXED>
constexpr size_t dc_smem() {
  return sizeof(double2) * DG_PACK + (MIXED ? sizeof(float2) * DG_PACK : 0) + sizeof(DcCommon);
}

__device__ __forceinline__ double2 dc_load(const double2* p) { return *p; }
__device__ __forceinline__ double2 dc_load(const float4* p) {
  const float4 v = *p;
  return make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
}
__device__ __forceinline__ void dc_store(double2* p, double2 v) { *p = v; }
__device__ __forceinline__ void dc_store(float4* p, double2 v) {
  const float rh = (float)v.x, ih = (float)v.y;
  *p = make_float4(rh, (float)(v.x - (double)rh), ih, (float)(v.y - (double)ih));
}
// x -= a conj(b); the order of the four products is part of the result
__device__ __forceinline__ void dc_mac(double2& x, double2 a, double2 b) {
  x.x = fma(-a.x, b.x, fma(-a.y, b.y, x.x));
  x.y = fma(-a.y, b.x, fma(a.x, b.y, x.y));
}
template <int C>
__device__ __forceinline__ int dc_owner(int b) {
  const int m = b % (2 * C);
  return m < C ? m : 2 * C - 1 - m;
}
// block q of CTA `rank`, ascending
template <int C>
__device__ __forceinline__ int dc_block(int rank, int q) {
  return q / 2 * 2 * C + (q & 1 ? 2 * C - 1 - rank : rank);
}
template <typename T>
__device__ __forceinline__ T* dc_peer(T* p, int rank) {
  return cg::this_cluster().map_shared_rank(p, rank);
}
// Complex Dot2 accumulation of a b into c (c[0] + c[1] the real part,
// c[2] + c[3] the imaginary part): a an element of L as double-float with
// its third terms at, b a double-float element.
__device__ __forceinline__ void cmac_l(dfl* c, float4 a, float2 at, float4 b) {
  dot2_acc3(c[0], a.x, a.y, at.x, b.x, b.y);
  dot2_acc3(c[1], -a.z, -a.w, -at.y, b.z, b.w);
  dot2_acc3(c[2], a.x, a.y, at.x, b.z, b.w);
  dot2_acc3(c[3], a.z, a.w, at.y, b.x, b.y);
}
__device__ __forceinline__ dfl df_add_quick(dfl x, dfl y) {
  const dfl t = df_two_sum(x.hi, y.hi);
  return dfl{t.hi, t.lo + (x.lo + y.lo)};
}

// Columns c0 .. c0 + 7 (c0 a multiple of 8) of the inverse of their 32 x 32
// diagonal block of L (packed, double-float Af with third terms Lt), in place,
// row by row, by one warp, four lanes per column.  invs: reciprocals of L's
// diagonal.
__device__ __forceinline__ void invert_diag_columns(float4* Af, const float2* Lt, const dfl* invs, int c0, int lane) {
  const int jj = c0 + (lane >> 2), part = lane & 3;
#pragma unroll 1
  for (int i = c0; i < (c0 | 31) + 1; ++i) {
    dfl c[4] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
    for (int m = jj + part; m < i; m += 4) cmac_l(c, Af[pk(i, m)], Lt[pk(i, m)], Af[pk(m, jj)]);
    dfl sr = df_add_quick(c[0], c[1]), si = df_add_quick(c[2], c[3]);
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      sr = df_add_quick(sr, dfl{__shfl_xor_sync(0xffffffffu, sr.hi, o), __shfl_xor_sync(0xffffffffu, sr.lo, o)});
      si = df_add_quick(si, dfl{__shfl_xor_sync(0xffffffffu, si.hi, o), __shfl_xor_sync(0xffffffffu, si.lo, o)});
    }
    __syncwarp();   // every read of row i (as L) is done
    if (jj <= i && part == 0) {
      const dfl inv = invs[i];
      const dfl qr = df_mul(df_fast_two_sum(sr.hi, sr.lo), inv);
      const dfl qi = df_mul(df_fast_two_sum(si.hi, si.lo), inv);
      Af[pk(i, jj)] = jj < i ? make_float4(-qr.hi, -qr.lo, -qi.hi, -qi.lo) : make_float4(inv.hi, inv.lo, 0.0f, 0.0f);
    }
    __syncwarp();   // row i of these columns is complete
  }
}

// 16 x 16 diagonal block of the panel at s0, in place: threads 0 .. 127 hold the
// elements (row r, columns c0 and c0 + 8), warp 4 the chain of pivots.
__device__ __forceinline__ void dc_factor(double2* A, DcCommon& sm, int s0, int col0, int tid) {
  auto sync = [] { asm volatile("bar.sync 1, 160;" ::: "memory"); };
  const bool chain = tid >= 128;
  const int r = tid >> 3, c0 = tid & 7;
  double2 x[2];
  if (!chain)
#pragma unroll
    for (int h = 0; h < 2; ++h) x[h] = c0 + 8 * h <= r ? A[pk(s0 + r, s0 + c0 + 8 * h)] : make_double2(0.0, 0.0);
  double d = A[pk(s0, s0)].x;   // (chain)
#pragma unroll 1
  for (int j = 0; j < DC_P; ++j) {
    if (chain) {
      const bool ok = d > 0.0 && isfinite(d);
      double l, rinv;
      const int ef = __double2hiint(d) >> 20;
      if (ef >= 1 && ef < 2047) {
        long long lb, rb;
        fx_sqrt_rcp(__double_as_longlong(d), lb, rb);
        l = __longlong_as_double(lb);
        rinv = __longlong_as_double(rb);
      } else {
        l = sqrt(d);
        rinv = 1.0 / l;
      }
      if (tid == 128) {
        if (!ok) sm.fail = col0 + s0 + j + 1;
        A[pk(s0 + j, s0 + j)] = make_double2(l, 0.0);
        sm.rinv[j] = rinv;
      }
    }
    sync();
    if (sm.fail || j == DC_P - 1) break;
    if (!chain) {
      if (c0 == (j & 7) && r > j) {
        const double rinv = sm.rinv[j];
        double2& a = j < 8 ? x[0] : x[1];
        a.x *= rinv;
        a.y *= rinv;
        A[pk(s0 + r, s0 + j)] = a;
      }
      if (r == j + 1 && c0 == ((j + 1) & 7)) sm.pub = j + 1 < 8 ? x[0].x : x[1].x;
    }
    sync();
    if (chain) {
      const double2 a = A[pk(s0 + j + 1, s0 + j)];
      d = fma(-a.x, a.x, fma(-a.y, a.y, sm.pub));
    } else {
      const double2 a = A[pk(s0 + max(r, j + 1), s0 + j)];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = c0 + 8 * h;
        if (8 * h + 7 > j && c > j && c <= r) dc_mac(x[h], a, A[pk(s0 + c, s0 + j)]);
      }
    }
  }
}

template <typename WS, int C>
__global__ void __launch_bounds__(DC_THREADS, 1) diag_cluster_kernel(BatchView v, int kg) {
  constexpr bool MIXED = std::is_same<WS, float4>::value;
  constexpr int NBLK = DC_NB / C;   // row blocks of eight per CTA
  extern __shared__ __align__(16) unsigned char dc_raw[];
  double2* A = reinterpret_cast<double2*>(dc_raw);   // packed lower 128 x 128
  float2* Lt = reinterpret_cast<float2*>(A + DG_PACK);
  DcCommon& sm = *reinterpret_cast<DcCommon*>(dc_raw + dc_smem<MIXED>() - sizeof(DcCommon));
  const int p = blockIdx.x / C, rank = blockIdx.x % C;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;   // this problem's block step
  if (k < 0 || k >= pr.nt) return;
  if (v.status[p] != 0) return;
  if (!BEOR_INBOUNDS(v.flags, pr.ws_off + (tri_index(k, k) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_DIAG_WS) ||
      !BEOR_INBOUNDS(v.flags, pr.dinv_off + (int64_t)(k + 1) * DG_PACK <= v.dinv_elems, BC_DIAG_DINV) ||
      !BEOR_INBOUNDS(v.flags, !MIXED || (int64_t)(p + 1) * BEOR_TB <= (int64_t)v.P * BEOR_TB, BC_DIAG_LINV))
    return;
  WS* ws = reinterpret_cast<WS*>(v.ws) + pr.ws_off + tri_index(k, k) * BEOR_TILE_ELEMS;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) sm.fail = 0;
  // own rows (a warp per block and four columns), and the first panel's diagonal block
  for (int w = warp; w < NBLK * (BEOR_TB / 4); w += DC_WARPS) {
    const int r = 8 * dc_block<C>(rank, w / (BEOR_TB / 4)) + (lane & 7), c = w % (BEOR_TB / 4) * 4 + (lane >> 3);
    if (c <= r) A[pk(r, c)] = dc_load(ws + c * BEOR_TB + r);
  }
  if (tid < DC_P * DC_P && tid % DC_P >= tid / DC_P)
    A[pk(tid % DC_P, tid / DC_P)] = dc_load(ws + tid / DC_P * BEOR_TB + tid % DC_P);
  cg::this_cluster().sync();

  for (int s0 = 0; s0 < BEOR_TB; s0 += DC_P) {
    const int s1 = s0 + DC_P;
    if (tid < 160) dc_factor(A, sm, s0, k * BEOR_TB, tid);
    __syncthreads();
    if (sm.fail) break;   // the same in every CTA of the cluster
    if (s1 == BEOR_TB) break;
    const int b1 = s1 / 8;                                   // first block of eight rows below the panel
    const int q0 = [&] { int q = 0; while (q < NBLK && dc_block<C>(rank, q) < b1) ++q; return q; }();
    // own rows below the panel: eight lanes per row (columns q, q + 8), results to every CTA
    for (int w = warp; w < 2 * (NBLK - q0); w += DC_WARPS) {
      const int row = 8 * dc_block<C>(rank, q0 + w / 2) + (w & 1) * 4 + (lane >> 3), q = lane & 7;
      double2 x[2] = {A[pk(row, s0 + q)], A[pk(row, s0 + q + 8)]};
#pragma unroll
      for (int h0 = 0; h0 < 2; ++h0) {
#pragma unroll 1
        for (int qj = 0; qj < 8; ++qj) {
          const int j = 8 * h0 + qj;
          const double rinv = sm.rinv[j];
          const double2 l = make_double2(x[h0].x * rinv, x[h0].y * rinv);
          if (q == qj) x[h0] = l;
          const double2 lr = make_double2(__shfl_sync(0xffffffffu, l.x, (lane & ~7) | qj),
                                          __shfl_sync(0xffffffffu, l.y, (lane & ~7) | qj));
          if (q > qj) dc_mac(x[h0], lr, A[pk(s0 + q + 8 * h0, s0 + j)]);
          if (h0 == 0) dc_mac(x[1], lr, A[pk(s0 + q + 8, s0 + j)]);
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        double2* o = dc_peer(A, c);
        o[pk(row, s0 + q)] = x[0];
        o[pk(row, s0 + q + 8)] = x[1];
      }
    }
    cg::this_cluster().sync();
    // rank-16 update of the own rows, 8 x 8 tiles; the next panel's diagonal block goes to every CTA
    int t = warp;
    for (int q = q0; q < NBLK; ++q) {
      const int b = dc_block<C>(rank, q);
      for (; t < b - b1 + 1; t += DC_WARPS) {
        const int cb = b1 + t, i = 8 * b + (lane >> 2), c = 8 * cb + (lane & 3);
        const bool on0 = c <= i, on1 = c + 4 <= i;
        double2 x0 = A[pk(i, min(c, i))], x1 = A[pk(i, min(c + 4, i))];
#pragma unroll 4
        for (int m = s0; m < s1; ++m) {
          const double2 a = A[pk(i, m)];
          dc_mac(x0, a, A[pk(c, m)]);
          dc_mac(x1, a, A[pk(c + 4, m)]);
        }
        if (on0) A[pk(i, c)] = x0;
        if (on1) A[pk(i, c + 4)] = x1;
        if (b <= b1 + 1)
#pragma unroll
          for (int o = 0; o < C; ++o) {
            if (o == rank) continue;
            double2* B = dc_peer(A, o);
            if (on0) B[pk(i, c)] = x0;
            if (on1) B[pk(i, c + 4)] = x1;
          }
      }
      t -= b - b1 + 1;
    }
    cg::this_cluster().sync();
  }
  if (sm.fail) {
    if (tid == 0 && rank == 0) v.status[p] = sm.fail;
    cg::this_cluster().sync();
    return;
  }

  // log-determinant contribution, 2 sum ln L_jj over the real rows
  if (rank == 0) {
    double ldp = 0.0;
    if (tid < BEOR_TB && k * BEOR_TB + tid < pr.n) ldp = 2.0 * log(A[pk(tid, tid)].x);
    for (int o = 16; o > 0; o >>= 1) ldp += __shfl_xor_sync(0xffffffffu, ldp, o);
    if (lane == 0 && warp < 4) sm.red[warp] = ldp;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < 4; ++w) s += sm.red[w];
      v.logdet_sigma[p] += s;
    }
  }
  // L_kk back to the workspace tile (own rows; upper part zero)
  for (int w = warp; w < NBLK * (BEOR_TB / 4); w += DC_WARPS) {
    const int r = 8 * dc_block<C>(rank, w / (BEOR_TB / 4)) + (lane & 7), c = w % (BEOR_TB / 4) * 4 + (lane >> 3);
    dc_store(ws + c * BEOR_TB + r, c <= r ? A[pk(r, c)] : make_double2(0.0, 0.0));
  }

  if constexpr (!MIXED) {
    // Linv[i][j] = -(sum_{m=j}^{i-1} L[i][m] Linv[m][j]) / L[i][i]: four partial
    // sums over m = j + part, j + part + 4, .., added up in pairs.  A warp takes
    // two columns, lane = (column, row of a block of 16); the rows of a block
    // follow each other through shuffles, the blocks through the CTA's copy.
    if (tid < BEOR_TB) sm.dinvs[tid] = 1.0 / A[pk(tid, tid)].x;
    __syncthreads();
    constexpr int NPAIR = BEOR_TB / 2 / C, NPW = NPAIR > DC_WARPS ? NPAIR / DC_WARPS : 1;   // pairs of this CTA, per warp
    const int r = lane & 15;
    const bool on = warp < NPAIR;
    auto column = [&](int q) { return 2 * dc_block<C>(rank, warp + DC_WARPS * q) + (lane >> 4); };   // dealt like the rows
    for (int I = 0; I < BEOR_TB / 16; ++I) {
      const int i = 16 * I + r, m1 = 16 * I;
      double2 out[NPW];
#pragma unroll
      for (int q = 0; q < NPW; ++q) {
        const int jj = column(q);
        out[q] = make_double2(0.0, 0.0);
        if (!on || m1 + 15 < (jj & ~1)) continue;
        double sr[4] = {0.0, 0.0, 0.0, 0.0}, si[4] = {0.0, 0.0, 0.0, 0.0};
        for (int m = jj; m < m1; m += 4) {
#pragma unroll
          for (int part = 0; part < 4; ++part)
            if (m + part < m1) {
              const double2 a = A[pk(i, m + part)], b = A[pk(m + part, jj)];
              sr[part] = fma(a.x, b.x, fma(-a.y, b.y, sr[part]));
              si[part] = fma(a.x, b.y, fma(a.y, b.x, si[part]));
            }
        }
#pragma unroll 1
        for (int t = 0; t < 16; ++t) {
          const int m = m1 + t;
          if (r == t && m >= jj) {
            const double inv = sm.dinvs[m];
            if (m == jj)
              out[q] = make_double2(inv, 0.0);
            else
              out[q] = make_double2(-((sr[0] + sr[1]) + (sr[2] + sr[3])) * inv, -((si[0] + si[1]) + (si[2] + si[3])) * inv);
          }
          const double2 b = make_double2(__shfl_sync(0xffffffffu, out[q].x, (lane & 16) | t),
                                         __shfl_sync(0xffffffffu, out[q].y, (lane & 16) | t));
          if (r > t && m >= jj) {
            const int part = (m - jj) & 3;
            const double2 a = A[pk(i, m)];
            double cr = part == 0 ? sr[0] : part == 1 ? sr[1] : part == 2 ? sr[2] : sr[3];
            double ci = part == 0 ? si[0] : part == 1 ? si[1] : part == 2 ? si[2] : si[3];
            cr = fma(a.x, b.x, fma(-a.y, b.y, cr));
            ci = fma(a.x, b.y, fma(a.y, b.x, ci));
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (u == part) {
                sr[u] = cr;
                si[u] = ci;
              }
          }
        }
      }
      __syncthreads();   // every read of block row I of L is done
      if (on)
#pragma unroll
        for (int q = 0; q < NPW; ++q)
          if (i >= column(q)) A[pk(i, column(q))] = out[q];
      __syncwarp();
    }
    double2* dinv = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
    if (on)
#pragma unroll
      for (int q = 0; q < NPW; ++q)
        for (int i = r; i < BEOR_TB; i += 16)
          if (i >= column(q)) dinv[pk(i, column(q))] = A[pk(i, column(q))];
  } else {
    // On the fp32 pipe (float64's rate is 1/64 of it): the inverse feeds the
    // 40-bit panel slices and the solves only.  Exact float triples of L (each
    // CTA splits its share for all), so that each product keeps its terms down
    // to 2^-48 of the leading part (Dot2 accumulation); Linv is held as
    // double-float.  Blocked by 32: the own columns of the diagonal blocks row by
    // row, sent to every CTA (all columns in every CTA: 83,000 of 590,000 cycles),
    // then X_IJ = sum_{M=J}^{I-1} L_IM Linv_MJ and Linv_IJ = -Linv_II X_IJ for
    // the own columns (blocks of eight, dealt like the rows).
    float4* Af = reinterpret_cast<float4*>(A);
    cg::this_cluster().sync();   // L is written out everywhere
    for (int e = tid + rank * DC_THREADS; e < DG_PACK; e += C * DC_THREADS) {
      const double2 a = A[e];
      const float rh = (float)a.x, ih = (float)a.y;
      const double rd = a.x - (double)rh, id = a.y - (double)ih;
      const float rl = (float)rd, il = (float)id;
      const float4 f = make_float4(rh, rl, ih, il);
      const float2 l3 = make_float2((float)(rd - (double)rl), (float)(id - (double)il));
#pragma unroll
      for (int c = 0; c < C; ++c) {
        dc_peer(Af, c)[e] = f;
        dc_peer(Lt, c)[e] = l3;
      }
    }
    cg::this_cluster().sync();
    if (tid < BEOR_TB) {
      const float4 d = Af[pk(tid, tid)];
      sm.invs[tid] = df_from_double(1.0 / ((double)d.x + (double)d.y + (double)Lt[pk(tid, tid)].x));
    }
    __syncthreads();
    if (warp < NBLK) invert_diag_columns(Af, Lt, sm.invs, 8 * dc_block<C>(rank, warp), lane);
    cg::this_cluster().sync();   // L's diagonal blocks are read everywhere
    for (int e = tid; e < NBLK * 256; e += DC_THREADS) {
      const int c0 = 8 * dc_block<C>(rank, e >> 8), i = (c0 & ~31) + ((e >> 3) & 31), jj = c0 + (e & 7);
      if (i < jj) continue;
      const float4 f = Af[pk(i, jj)];
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (c != rank) dc_peer(Af, c)[pk(i, jj)] = f;
    }
    cg::this_cluster().sync();
    // block row I: X_IJ = sum_{m=jj}^{32 I - 1} L[i][m] Linv[m][jj], then Linv_IJ = -Linv_II X_IJ
    constexpr int NQ = NBLK / 2;   // outputs per thread: two blocks of eight columns x 32 rows at a time
    const int cr = (tid >> 3) & 31, cc = tid & 7;
    for (int I = 1; I < BEOR_TB / 32; ++I) {
      const int i = 32 * I + cr;
      dfl xr[NQ], xi[NQ];
#pragma unroll
      for (int step = 0; step < 2; ++step) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const int jj = 8 * dc_block<C>(rank, 2 * q + (tid >> 8)) + cc;
          if (jj >= 32 * I) continue;
          dfl a[4] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
          if (step == 0) {
#pragma unroll 1
            for (int m = jj; m < 32 * I; ++m) cmac_l(a, Af[pk(i, m)], Lt[pk(i, m)], Af[pk(m, jj)]);
          } else {
            const float2 zero = make_float2(0.0f, 0.0f);
#pragma unroll 1
            for (int m = 32 * I; m <= i; ++m) cmac_l(a, Af[pk(i, m)], zero, Af[pk(m, jj)]);
          }
          xr[q] = df_add_quick(a[0], a[1]);
          xi[q] = df_add_quick(a[2], a[3]);
        }
        __syncthreads();   // every read of block row I (of L, then of X) is done
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const int jj = 8 * dc_block<C>(rank, 2 * q + (tid >> 8)) + cc;
          if (jj >= 32 * I) continue;
          const dfl ur = df_fast_two_sum(xr[q].hi, xr[q].lo), ui = df_fast_two_sum(xi[q].hi, xi[q].lo);
          Af[pk(i, jj)] = step == 0 ? make_float4(ur.hi, ur.lo, ui.hi, ui.lo) : make_float4(-ur.hi, -ur.lo, -ui.hi, -ui.lo);
        }
        __syncthreads();
      }
    }
    // own columns out: float64 inverse, row maxima to every CTA, then the slices
    double2* dinv = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
    if (tid < BEOR_TB) {
      float mx = 0.0f;
      for (int q = 0; q < NBLK; ++q) {
        const int c0 = 8 * dc_block<C>(rank, q);
        for (int c = c0; c < min(c0 + 8, tid + 1); ++c) {
          const float4 f = Af[pk(tid, c)];
          mx = fmaxf(mx, fmaxf(fabsf(f.x), fabsf(f.z)));
          dinv[pk(tid, c)] = make_double2((double)f.x + (double)f.y, (double)f.z + (double)f.w);
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) dc_peer(&sm, c)->rmax[rank][tid] = mx;
    }
    cg::this_cluster().sync();
    if (tid < BEOR_TB) {
      float mx = 0.0f;
#pragma unroll
      for (int c = 0; c < C; ++c) mx = fmaxf(mx, sm.rmax[c][tid]);
      const int e = mx > 0.0f ? ilogbf(mx) + 1 : -1000;
      sm.ex[tid] = e;
      if (rank == 0) v.linv_exp[(int64_t)p * BEOR_TB + tid] = e;
    }
    __syncthreads();
    for (int w = warp; w < NBLK * (BEOR_TB / 32); w += DC_WARPS) {
      const int r = w / NBLK * 32 + lane, c0 = 8 * dc_block<C>(rank, w % NBLK);
      linv_slice_chunk(v, p, Af, r, c0, sm.ex[r]);
    }
  }
}

// One CTA per block, for batches that have more blocks than the GPU holds
// clusters of two: the float64 pipe (0.87 ms of it per block and SM) bounds it,
// and the finer steps of the cluster's kernel cost more of its instructions
// (1.33 ms a block with C = 1, 1.17 here).
__global__ void __launch_bounds__(512) diag_f64_kernel(BatchView v, int kg) {
  extern __shared__ double2 dsm[];
  double2* A = dsm;                    // packed lower 128x128
  double2* col = dsm + DG_PACK;        // 128
  __shared__ int s_fail;
  __shared__ double s_rinv;            // 1 / L_jj of the current column
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;   // this problem's block step
  if (k < 0 || k >= pr.nt) return;
  if (v.status[p] != 0) return;
  if (!BEOR_INBOUNDS(v.flags, pr.ws_off + (tri_index(k, k) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_DIAG_WS) ||
      !BEOR_INBOUNDS(v.flags, pr.dinv_off + (int64_t)(k + 1) * DG_PACK <= v.dinv_elems, BC_DIAG_DINV))
    return;
  double2* ws = reinterpret_cast<double2*>(v.ws) + pr.ws_off + tri_index(k, k) * BEOR_TILE_ELEMS;
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int e = tid; e < BEOR_TILE_ELEMS; e += nthr) {
    int r = e % BEOR_TB, c = e / BEOR_TB;
    if (r >= c) A[pk(r, c)] = ws[e];
  }
  if (tid == 0) s_fail = 0;
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31, nwarp = nthr >> 5;
  // Right-looking Cholesky, two columns per pass (rank-2 updates): half the
  // barriers and shared-memory round trips of one column per pass, with the
  // same operations in the same order as the rank-1 sequence (identical
  // results).  Thread 0 takes both pivots: L_jj, column j's element in row
  // j+1 and its update of a_{j+1,j+1}, then L_{j+1,j+1}.
  double2* col2 = col + BEOR_TB;   // column j+1
  __shared__ double s_rinv2;
  for (int j = 0; j < BEOR_TB; j += 2) {
    if (tid == 0) {
      const double d = A[pk(j, j)].x;
      if (!(d > 0.0) || !isfinite(d)) {
        s_fail = k * BEOR_TB + j + 1;
      } else {
        const double l = sqrt(d);
        A[pk(j, j)] = make_double2(l, 0.0);
        const double rinv = 1.0 / l;
        s_rinv = rinv;
        double2 a = A[pk(j + 1, j)];
        a.x *= rinv;
        a.y *= rinv;
        A[pk(j + 1, j)] = a;
        col[j + 1] = a;
        double2 x = A[pk(j + 1, j + 1)];
        x.x = fma(-a.x, a.x, fma(-a.y, a.y, x.x));
        x.y = fma(-a.y, a.x, fma(a.x, a.y, x.y));
        const double d2 = x.x;
        if (!(d2 > 0.0) || !isfinite(d2)) {
          s_fail = k * BEOR_TB + j + 2;
        } else {
          const double l2 = sqrt(d2);
          A[pk(j + 1, j + 1)] = make_double2(l2, 0.0);
          s_rinv2 = 1.0 / l2;
        }
      }
    }
    __syncthreads();
    if (s_fail) break;
    const double inv = s_rinv, inv2 = s_rinv2;
    const double2 lj1 = col[j + 1];   // L_{j+1,j}
    // columns j and j+1 below the pair: scale column j, apply it to column
    // j+1 (the rank-1 step's update of those elements), scale column j+1
    for (int i = j + 2 + tid; i < BEOR_TB; i += nthr) {
      double2 a = A[pk(i, j)];
      a.x *= inv;
      a.y *= inv;
      A[pk(i, j)] = a;
      col[i] = a;
      double2 b = A[pk(i, j + 1)];
      b.x = fma(-a.x, lj1.x, fma(-a.y, lj1.y, b.x));
      b.y = fma(-a.y, lj1.x, fma(a.x, lj1.y, b.y));
      b.x *= inv2;
      b.y *= inv2;
      A[pk(i, j + 1)] = b;
      col2[i] = b;
    }
    __syncthreads();
    // rank-2 update of the trailing lower triangle (rows and columns >= j+2):
    // A_il -= L_ij conj(L_lj), then -= L_i,j+1 conj(L_l,j+1); the triangle's
    // elements are dealt out in order, so every lane has work
    {
      const int nt2 = BEOR_TB - 2 - j;
      const int total = nt2 * (nt2 + 1) / 2;
      for (int e = tid; e < total; e += nthr) {
        int a = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        while (a * (a + 1) / 2 > e) --a;
        while ((a + 1) * (a + 2) / 2 <= e) ++a;
        const int i = j + 2 + a, l = j + 2 + (e - a * (a + 1) / 2);
        const double2 ai = col[i], al = col[l], bi = col2[i], bl = col2[l];
        double2 x = A[pk(i, l)];
        x.x = fma(-ai.x, al.x, fma(-ai.y, al.y, x.x));
        x.y = fma(-ai.y, al.x, fma(ai.x, al.y, x.y));
        x.x = fma(-bi.x, bl.x, fma(-bi.y, bl.y, x.x));
        x.y = fma(-bi.y, bl.x, fma(bi.x, bl.y, x.y));
        A[pk(i, l)] = x;
      }
    }
    __syncthreads();
  }
  if (s_fail) {
    if (tid == 0) v.status[p] = s_fail;
    return;
  }
  // log-determinant contribution, 2 sum ln L_jj over the real rows, in parallel
  {
    __shared__ double red[32];
    double ldp = 0.0;
    if (tid < BEOR_TB && k * BEOR_TB + tid < pr.n) ldp = 2.0 * log(A[pk(tid, tid)].x);
    for (int o = 16; o > 0; o >>= 1) ldp += __shfl_xor_sync(0xffffffffu, ldp, o);
    if (lane == 0) red[warp] = ldp;
    __syncthreads();
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < nwarp; ++w) s += red[w];
      v.logdet_sigma[p] += s;
    }
  }
  // L_kk back to the workspace tile (upper part zero)
  for (int e = tid; e < BEOR_TILE_ELEMS; e += nthr) {
    int r = e % BEOR_TB, c = e / BEOR_TB;
    ws[e] = r >= c ? A[pk(r, c)] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  // in-place inverse, row by row: Linv[i][j] = -(sum_{m=j}^{i-1} L[i][m] Linv[m][j]) / L[i][i];
  // four threads share each dot product (thread = 4 j + part)
  const int jj = tid >> 2, part = tid & 3;
  for (int i = 0; i < BEOR_TB; ++i) {
    if (tid == 0) s_rinv = 1.0 / A[pk(i, i)].x;
    double sr = 0.0, si = 0.0;
    if (jj < i) {
      for (int m = jj + part; m < i; m += 4) {
        const double2 a = A[pk(i, m)], b = A[pk(m, jj)];
        sr = fma(a.x, b.x, fma(-a.y, b.y, sr));
        si = fma(a.x, b.y, fma(a.y, b.x, si));
      }
    }
    sr += __shfl_xor_sync(0xffffffffu, sr, 1);
    si += __shfl_xor_sync(0xffffffffu, si, 1);
    sr += __shfl_xor_sync(0xffffffffu, sr, 2);
    si += __shfl_xor_sync(0xffffffffu, si, 2);
    __syncthreads();
    if (jj < i && part == 0) {
      const double inv = s_rinv;
      A[pk(i, jj)] = make_double2(-sr * inv, -si * inv);
    }
    if (tid == 0) A[pk(i, i)] = make_double2(s_rinv, 0.0);
    __syncthreads();
  }
  double2* dinv = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
  for (int e = tid; e < DG_PACK; e += nthr) dinv[e] = A[e];
}

template <typename WS, int C>
static int dc_fit() {   // blocks that are factored at once
  constexpr size_t smem = dc_smem<std::is_same<WS, float4>::value>();
  static PerDevice<int> fit;
  return fit.get([] {   // once: the kernel's attribute, and the device's answer
    allow_smem<diag_cluster_kernel<WS, C>>((int)smem);
    return max_clusters(diag_cluster_kernel<WS, C>, DC_THREADS, smem, C);
  });
}
template <typename WS, int C>
static cudaError_t launch_dc(const BatchView& v, int k, cudaStream_t s, int prio) {
  dc_fit<WS, C>();
  return launch_cluster(diag_cluster_kernel<WS, C>, dim3(C * v.P), dim3(DC_THREADS),
                        dc_smem<std::is_same<WS, float4>::value>(), s, prio, C, v, k);
}

// Float64: the largest cluster, of up to eight CTAs, of which the GPU holds the
// whole batch at once (15 clusters of eight, 36 of four and 76 of two on a GB300:
// 0.35, 0.46 and 0.73 ms a block), else one CTA per block (1.17 ms).  The
// posterior mean is of one point, and always takes eight.
cudaError_t launch_diag_cluster(const BatchView& v, int k, bool mixed, int active, cudaStream_t s, int prio) {
  if (mixed) return launch_dc<float4, DIAG_MEAN_CTAS>(v, k, s, prio);
  if (active <= dc_fit<double2, 8>()) return launch_dc<double2, 8>(v, k, s, prio);
  if (active <= dc_fit<double2, 4>()) return launch_dc<double2, 4>(v, k, s, prio);
  if (active <= dc_fit<double2, 2>()) return launch_dc<double2, 2>(v, k, s, prio);
  constexpr size_t smem = sizeof(double2) * (DG_PACK + 2 * BEOR_TB);   // packed block and two columns
  const cudaError_t attr = allow_smem<diag_f64_kernel>((int)smem);
  if (attr != cudaSuccess) return attr;
  return launch_prio(diag_f64_kernel, dim3(v.P), dim3(512), smem, s, prio, v, k);
}

}  // namespace beor
