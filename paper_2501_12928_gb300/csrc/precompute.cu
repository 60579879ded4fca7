// One-off precompute of M = T^H N^-1 T and dbar = T^H N^-1 d in float64.
//
// Sec. "Running BayesEoR": the instrument model forward-models the data; the
// likelihood needs the data-space products T^H N^-1 T and T^H N^-1 d once
// per instrument, after which every prior point only changes a diagonal.
// Two routes:
//  * dense:    M = T^H diag(w) T directly from T (n_vis x n row-major): on
//              the FP64 pipe (float64 contexts) or as seven-digit bf16 slice
//              products on the tensor cores (mixed contexts, herk_tc.cu),
//  * factored: T[(f,tb),(c,x)] = A_f[tb,c] W[f,x] gives
//              G_f = A_f^H diag(w_f) A_f and
//              M[(c,x),(c',x')] = sum_f conj(W[f,x]) W[f,x'] G_f[c,c'],
//    which never forms T.
// Both are float64 throughout (the refinement of the solve and the
// log-determinant need an M accurate far beyond float32).
#include <algorithm>

#include "beor_common.cuh"
#include "beor_internal.h"

namespace beor {

// ---------------------------------------------------------------------------
// C = X^H diag(w) X, X: K x n complex (row-major, leading dimension ldx).  Each
// CTA computes one 64 x 64 sub-tile of a lower 128-tile of C, in packed tiles
// (the factorisation layout).
// ---------------------------------------------------------------------------
constexpr int HK_T = 64;   // sub-tile edge
constexpr int HK_K = 16;   // K rows per smem stage

__global__ void __launch_bounds__(256) herk_f64_kernel(const double2* __restrict__ X, int64_t ldx,
                                                       const double* __restrict__ w, int64_t K, int n,
                                                       double2* __restrict__ C) {
  __shared__ double2 sa[HK_K][HK_T];
  __shared__ double2 sb[HK_K][HK_T];
  // which 128-tile (I, J), I >= J, and which 64 sub-tile
  int t = blockIdx.x >> 2, sub = blockIdx.x & 3;
  int I = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
  while ((int64_t)I * (I + 1) / 2 > t) --I;
  while ((int64_t)(I + 1) * (I + 2) / 2 <= t) ++I;
  int J = t - I * (I + 1) / 2;
  const int si = sub >> 1, sj = sub & 1;
  const int r0 = I * BEOR_TB + si * HK_T;     // rows of C  <- columns of X (conj side)
  const int c0 = J * BEOR_TB + sj * HK_T;     // cols of C  <- columns of X
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double ar[4][4], ai[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) ar[a][b] = ai[a][b] = 0.0;
  const bool skip = (r0 >= n) || (c0 >= n);
  if (!skip) {
    for (int64_t k0 = 0; k0 < K; k0 += HK_K) {
      for (int e = threadIdx.x; e < HK_K * HK_T; e += 256) {
        int kk = e / HK_T, cc = e % HK_T;
        int64_t k = k0 + kk;
        double2 va = make_double2(0.0, 0.0), vb = make_double2(0.0, 0.0);
        if (k < K) {
          if (r0 + cc < n) va = X[k * ldx + r0 + cc];
          if (c0 + cc < n) {
            vb = X[k * ldx + c0 + cc];
            double ww = w[k];
            vb.x *= ww;
            vb.y *= ww;
          }
        }
        sa[kk][cc] = va;
        sb[kk][cc] = vb;
      }
      __syncthreads();
#pragma unroll 4
      for (int kk = 0; kk < HK_K; ++kk) {
        double2 a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          a[q] = sa[kk][ty * 4 + q];
          b[q] = sb[kk][tx * 4 + q];
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // conj(a) * b
            ar[p][q] = fma(a[p].x, b[q].x, fma(a[p].y, b[q].y, ar[p][q]));
            ai[p][q] = fma(a[p].x, b[q].y, fma(-a[p].y, b[q].x, ai[p][q]));
          }
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int r = r0 + ty * 4 + p, c = c0 + tx * 4 + q;
      double vr = ar[p][q], vi = ai[p][q];
      if (r >= n || c >= n) { vr = 0.0; vi = 0.0; }
      if (r == c) vi = 0.0;
      C[tri_index(I, J) * BEOR_TILE_ELEMS + (int64_t)(c - J * BEOR_TB) * BEOR_TB + (r - I * BEOR_TB)] =
          make_double2(vr, vi);
    }
}

// G_f = A_f^H diag(w_f) A_f of a factored instrument, f = blockIdx.y, lower
// triangle of a row-major n x n matrix (n uv cells): one 16 x 16 tile per warp,
// lane = (row, eight columns).  Bound by the float64 pipe (64 cycles per warp
// instruction and sub-partition, so that the operands' way through shared
// memory, eight rows at a time, costs nothing).  64 x 64 tiles left three
// quarters of the work in padding and above the diagonal at 80 cells: 38
// channels of 2394 rows 9.9 ms -> 2.85 (its floor is 2.7).  Each element sums the rows in
// order, w on the column's side.
constexpr int GK = 8;   // rows per step
__global__ void __launch_bounds__(128) gram_cells_kernel(const double2* __restrict__ X, const double* __restrict__ w,
                                                         int64_t K, int n, int ntiles, double2* __restrict__ G) {
  __shared__ double2 sa[4][GK][16], sb[4][GK][16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = blockIdx.x * 4 + warp;
  if (t >= ntiles) return;
  X += blockIdx.y * K * n;
  w += blockIdx.y * K;
  G += (int64_t)blockIdx.y * n * n;
  int I = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (I * (I + 1) / 2 > t) --I;
  while ((I + 1) * (I + 2) / 2 <= t) ++I;
  const int J = t - I * (I + 1) / 2;
  const int r = lane >> 1, c0 = (lane & 1) * 8;
  const int ca = min(16 * I + (lane & 15), n - 1), cb = min(16 * J + (lane & 15), n - 1), kl = lane >> 4;
  double2 a[GK / 2], b[GK / 2];
  auto load = [&](int64_t k0) {   // rows k0 + kl, + 2, ..; zeros beyond the last
#pragma unroll
    for (int i = 0; i < GK / 2; ++i) {
      const int64_t k = k0 + kl + 2 * i, kc = min(k, K - 1);
      a[i] = X[kc * n + ca];
      b[i] = X[kc * n + cb];
      const double ww = k < K ? w[kc] : 0.0;
      b[i].x *= ww;
      b[i].y *= ww;
    }
  };
  double ar[8], ai[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) ar[q] = ai[q] = 0.0;
  load(0);
  for (int64_t k0 = 0; k0 < K; k0 += GK) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < GK / 2; ++i) {
      sa[warp][kl + 2 * i][lane & 15] = a[i];
      sb[warp][kl + 2 * i][lane & 15] = b[i];
    }
    __syncwarp();
    if (k0 + GK < K) load(k0 + GK);
    const int nk = (int)min((int64_t)GK, K - k0);
#pragma unroll 2
    for (int kk = 0; kk < nk; ++kk) {
      const double2 x = sa[warp][kk][r];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double2 y = sb[warp][kk][c0 + q];
        // conj(x) * y
        ar[q] = fma(x.x, y.x, fma(x.y, y.y, ar[q]));
        ai[q] = fma(x.x, y.y, fma(-x.y, y.x, ai[q]));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = 16 * I + r, j = 16 * J + c0 + q;
    if (i < n && j <= i) G[(int64_t)i * n + j] = make_double2(ar[q], i == j ? 0.0 : ai[q]);
  }
}

// u[b][j] = sum_k conj(X_b[k, j]) w_b[k] d_b[k]  (atomic accumulation over K chunks)
__global__ void __launch_bounds__(256) xh_w_d_kernel(const double2* __restrict__ X, int64_t ldx, int64_t x_batch_stride,
                              const double* __restrict__ w, const double2* __restrict__ d,
                              int64_t vec_batch_stride, int64_t K, int n, int64_t kchunk,
                              double2* __restrict__ u, int64_t u_batch_stride) {
  const int bz = blockIdx.z;
  X += bz * x_batch_stride;
  w += bz * vec_batch_stride;
  d += bz * vec_batch_stride;
  u += bz * u_batch_stride;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t k0 = blockIdx.y * kchunk, k1 = min(K, k0 + kchunk);
  // w d of 256 rows at a time, formed once per CTA (two of six float64 products
  // per element, on the pipe that bounds this kernel)
  __shared__ double2 dw[256];
  double sr = 0.0, si = 0.0;
  for (int64_t kb = k0; kb < k1; kb += 256) {
    __syncthreads();
    if (kb + threadIdx.x < k1) {
      const double2 dd = d[kb + threadIdx.x];
      const double ww = w[kb + threadIdx.x];
      dw[threadIdx.x] = make_double2(dd.x * ww, dd.y * ww);
    }
    __syncthreads();
    const int nk = (int)min((int64_t)256, k1 - kb);
    const double2* __restrict__ x0 = X + kb * ldx + min(j, n - 1);
#pragma unroll 8
    for (int k = 0; k < nk; ++k) {
      const double2 x = x0[k * ldx], q = dw[k];
      sr = fma(x.x, q.x, fma(x.y, q.y, sr));
      si = fma(x.x, q.y, fma(-x.y, q.x, si));
    }
  }
  if (j >= n) return;
  atomicAdd(&u[j].x, sr);
  atomicAdd(&u[j].y, si);
}

// The same, same bits, where that has few CTAs.
// A chunk's sum is one chain of dependent float64 products per component (134
// cycles a row).  32 columns per CTA and a warp per component keep each chain on a
// quarter of an SM, with two chunks of 16 rows in flight: the data of a 3280-mode
// instrument (38 channels of 2394 rows, 80 cells) 0.98 -> 0.32 ms.
constexpr int XH_COLS = 32, XH_U = 16, XH_ROWS = 256;
__global__ void __launch_bounds__(2 * XH_COLS) xh_w_d_split_kernel(const double2* __restrict__ X, int64_t ldx, int64_t x_batch_stride,
                              const double* __restrict__ w, const double2* __restrict__ d,
                              int64_t vec_batch_stride, int64_t K, int n, int64_t kchunk,
                              double2* __restrict__ u, int64_t u_batch_stride) {
  const int bz = blockIdx.z, comp = threadIdx.x / XH_COLS;
  X += bz * x_batch_stride;
  w += bz * vec_batch_stride;
  d += bz * vec_batch_stride;
  u += bz * u_batch_stride;
  const int j = blockIdx.x * XH_COLS + threadIdx.x % XH_COLS;
  const int64_t k0 = blockIdx.y * kchunk, k1 = min(K, k0 + kchunk);
  // w d of 256 rows at a time, formed once per CTA, by component
  __shared__ double dw[2][XH_ROWS];
  const double2* __restrict__ x0 = X + min(j, n - 1);
  double2 a[XH_U], b[XH_U];
  auto load = [&](double2* o, int64_t k) {
#pragma unroll
    for (int q = 0; q < XH_U; ++q) o[q] = x0[min(k + q, k1 - 1) * ldx];
  };
  double acc = 0.0;
  auto mac = [&](const double2* x, int64_t k) {   // re: x d, im: x d with the parts of d exchanged and one sign
    const int r = (int)((k - k0) % XH_ROWS);
#pragma unroll
    for (int q = 0; q < XH_U; ++q)
      if (k + q < k1) acc = fma(x[q].x, dw[comp][r + q], fma(comp ? -x[q].y : x[q].y, dw[1 - comp][r + q], acc));
  };
  load(a, k0);
  for (int64_t kb = k0; kb < k1; kb += 2 * XH_U) {
    if ((kb - k0) % XH_ROWS == 0) {
      __syncthreads();
      for (int r = threadIdx.x; r < XH_ROWS && kb + r < k1; r += 2 * XH_COLS) {
        const double2 dd = d[kb + r];
        const double ww = w[kb + r];
        dw[0][r] = dd.x * ww;
        dw[1][r] = dd.y * ww;
      }
      __syncthreads();
    }
    load(b, kb + XH_U);
    mac(a, kb);
    load(a, kb + 2 * XH_U);
    mac(b, kb + XH_U);
  }
  if (j >= n) return;
  atomicAdd(comp ? &u[j].y : &u[j].x, acc);
}

static void launch_xh_w_d(const double2* X, int64_t ldx, int64_t x_batch_stride, const double* w, const double2* d,
                          int64_t vec_batch_stride, int64_t K, int n, int64_t kchunk, double2* u, int64_t u_batch_stride,
                          int nbatch, cudaStream_t s) {
  const unsigned chunks = (unsigned)((K + kchunk - 1) / kchunk);
  // two waves of the wide kernel's CTAs: beyond, fewer reads of X count for more than the chains (a dense 3280-mode
  // instrument of 90,972 visibilities, 1157 CTAs: 2.15 ms, 3.46 in the split kernel)
  if ((int64_t)((n + 255) / 256) * chunks * nbatch >= 2 * device_sms())
    xh_w_d_kernel<<<dim3((n + 255) / 256, chunks, nbatch), 256, 0, s>>>(X, ldx, x_batch_stride, w, d, vec_batch_stride, K, n,
                                                                       kchunk, u, u_batch_stride);
  else
    xh_w_d_split_kernel<<<dim3((n + XH_COLS - 1) / XH_COLS, chunks, nbatch), 2 * XH_COLS, 0, s>>>(
        X, ldx, x_batch_stride, w, d, vec_batch_stride, K, n, kchunk, u, u_batch_stride);
}

// Structured M: M[(c,x),(c',x')] = sum_f conj(W[f,x]) W[f,x'] G[f][c][c'] into
// packed tiles.
//
// Bound by the float64 pipe.  The products of two weights depend on (f, x, x')
// only; formed once, they leave four of eight instructions per element and f.  A
// CTA takes units of 16 columns of a tile, four elements per thread.  3280 modes
// (38 channels, nx = 41): 3.01 -> 1.44 ms.
__device__ __forceinline__ double2 weight_product(double2 wa, double2 wb) {   // conj(wa) wb
  return make_double2(wa.x * wb.x + wa.y * wb.y, wa.x * wb.y - wa.y * wb.x);
}
__global__ void weight_products_kernel(const double2* __restrict__ W, int nf, int nx, double2* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // [f][x'][x]
  if (i >= (int64_t)nf * nx * nx) return;
  const int64_t f = i / ((int64_t)nx * nx);
  out[i] = weight_product(W[f * nx + i % nx], W[f * nx + i / nx % nx]);
}
constexpr int AM_THREADS = 512, AM_COLS = 16, AM_Q = AM_COLS * BEOR_TB / AM_THREADS;
template <bool TABLE>   // tab: the products, else unused
__global__ void __launch_bounds__(AM_THREADS)
    assemble_M_kernel(const double2* __restrict__ G, const double2* __restrict__ W, const double2* __restrict__ tab, int nf,
                      int ncells, int nx, int n, int nt, double2* __restrict__ Mt) {
  const int64_t units = tri_count(nt) * (BEOR_TB / AM_COLS);
  const int row = threadIdx.x & (BEOR_TB - 1);
  for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
    const int64_t t = u / (BEOR_TB / AM_COLS);
    int I = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((int64_t)I * (I + 1) / 2 > t) --I;
    while ((int64_t)(I + 1) * (I + 2) / 2 <= t) ++I;
    const int J = (int)(t - (int64_t)I * (I + 1) / 2);
    const int c0 = (int)(u % (BEOR_TB / AM_COLS)) * AM_COLS + threadIdx.x / BEOR_TB;
    const int r = I * BEOR_TB + row;
    const int cr = r / nx, xr = r % nx;
    int cc[AM_Q], xc[AM_Q];
    double vr[AM_Q], vi[AM_Q];
    bool on[AM_Q];
#pragma unroll
    for (int q = 0; q < AM_Q; ++q) {
      const int c = J * BEOR_TB + c0 + q * (AM_THREADS / BEOR_TB);
      on[q] = r < n && c <= r;   // G's lower triangle; the diagonal tiles' upper halves are zero
      cc[q] = on[q] ? c / nx : 0;
      xc[q] = on[q] ? c % nx : 0;
      vr[q] = vi[q] = 0.0;
    }
    if (on[0]) {   // else all four lie above the diagonal or beyond n
#pragma unroll 2
      for (int f = 0; f < nf; ++f) {
        const double2* __restrict__ g0 = G + ((int64_t)f * ncells + cr) * ncells;
        const double2 wa = TABLE ? make_double2(0.0, 0.0) : W[f * nx + xr];
#pragma unroll
        for (int q = 0; q < AM_Q; ++q) {
          const double2 p = TABLE ? tab[((int64_t)f * nx + xc[q]) * nx + xr] : weight_product(wa, W[f * nx + xc[q]]);
          const double2 g = g0[cc[q]];
          vr[q] = fma(p.x, g.x, fma(-p.y, g.y, vr[q]));
          vi[q] = fma(p.x, g.y, fma(p.y, g.x, vi[q]));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < AM_Q; ++q) {
      const int cw = c0 + q * (AM_THREADS / BEOR_TB);
      Mt[t * BEOR_TILE_ELEMS + cw * BEOR_TB + row] =
          on[q] ? make_double2(vr[q], r == J * BEOR_TB + cw ? 0.0 : vi[q]) : make_double2(0.0, 0.0);
    }
  }
}

// dbar[(c,x)] = sum_f conj(W[f,x]) u[f][c]
__global__ void assemble_dbar_kernel(const double2* __restrict__ u, const double2* __restrict__ W, int nf,
                                     int ncells, int nx, int n, int np, double2* __restrict__ dbar) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= np) return;
  double vr = 0.0, vi = 0.0;
  if (j < n) {
    int c = j / nx, x = j % nx;
    for (int f = 0; f < nf; ++f) {
      double2 ww = W[f * nx + x], uu = u[(int64_t)f * ncells + c];
      vr = fma(ww.x, uu.x, fma(ww.y, uu.y, vr));
      vi = fma(ww.x, uu.y, fma(-ww.y, uu.x, vi));
    }
  }
  dbar[j] = make_double2(vr, vi);
}

// x -> (hi, lo) float pairs with hi + lo = x to ~48 bits (once per precompute)
__global__ void split_df_kernel(const double2* __restrict__ M, int64_t n, float4* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = M[e];
    const float rh = (float)v.x, ih = (float)v.y;
    out[e] = make_float4(rh, (float)(v.x - (double)rh), ih, (float)(v.y - (double)ih));
  }
}

// ---------------------------------------------------------------------------
// host launchers
// Tile (I, J) of the full square, element (r, c) column-major: M_IJ for
// I > J, conj(M_JI)^T for I < J, the Hermitian mirror of the stored lower
// part inside diagonal tiles; entries beyond n are zero.  Each component
// is split m = hi + lo + t exactly (hi = fl(m), lo = fl(m - hi), and the
// remainder has at most 53 - 48 bits).
__global__ void split_full_kernel(const double2* __restrict__ M, int n, int nt, float4* __restrict__ hl,
                                  float2* __restrict__ tt) {
  const int I = blockIdx.x / nt, J = blockIdx.x % nt;
  const int64_t out0 = (int64_t)blockIdx.x * BEOR_TILE_ELEMS;
  for (int e = threadIdx.x; e < BEOR_TILE_ELEMS; e += blockDim.x) {
    const int c = e / BEOR_TB, r = e % BEOR_TB;
    const int gr = I * BEOR_TB + r, gc = J * BEOR_TB + c;
    double2 m = make_double2(0.0, 0.0);
    if (gr < n && gc < n) {
      if (gr >= gc) {
        m = M[tri_index(I, J) * BEOR_TILE_ELEMS + (int64_t)c * BEOR_TB + r];
      } else {
        const double2 u = M[tri_index(J, I) * BEOR_TILE_ELEMS + (int64_t)r * BEOR_TB + c];
        m = make_double2(u.x, -u.y);
      }
    }
    const float rh = (float)m.x, ih = (float)m.y;
    const double rd = m.x - (double)rh, id = m.y - (double)ih;
    const float rl = (float)rd, il = (float)id;
    hl[out0 + e] = make_float4(rh, rl, ih, il);
    tt[out0 + e] = make_float2((float)(rd - (double)rl), (float)(id - (double)il));
  }
}

// Packed lower tiles -> rows of the full matrix, through 32 x 32 blocks in shared
// memory (the tiles are column-major, the output row-major; blocks above the
// diagonal are read from their mirror image).  86 MB read and 172 MB written at
// 3280 modes; the host loop that did this took 60 ms.
__global__ void __launch_bounds__(256) unpack_hermitian_kernel(const double2* __restrict__ M, int n, int64_t r0,
                                                               int64_t rows, double2* __restrict__ out) {
  __shared__ double2 s[32][33];
  const int64_t rb = r0 + (int64_t)blockIdx.y * 32;   // the block's first row and column
  const int cb = blockIdx.x * 32;
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5;
  // source block: rows rs.., columns cs.. of the lower triangle
  const bool mirror = rb + 31 < cb;
  const int64_t rs = mirror ? cb : rb, cs = mirror ? rb : cb;
  for (int y = y0; y < 32; y += 8) {   // x: row of the source (contiguous), y: column
    int64_t i = rs + x, j = cs + y;
    const bool flip = i < j;           // only in blocks that cross the diagonal
    if (flip) {
      const int64_t t = i;
      i = j;
      j = t;
    }
    double2 v = make_double2(0.0, 0.0);
    if (i < n && j < n)
      v = M[tri_index((int)(i / BEOR_TB), (int)(j / BEOR_TB)) * BEOR_TILE_ELEMS + (j % BEOR_TB) * BEOR_TB + i % BEOR_TB];
    if (flip != mirror) v.y = -v.y;
    s[y][x] = v;
  }
  __syncthreads();
  for (int y = y0; y < 32; y += 8) {   // row y, column x of the output block
    const int64_t r = rb + y;
    if (r < r0 + rows && cb + x < n) out[(r - r0) * n + cb + x] = mirror ? s[y][x] : s[x][y];
  }
}

cudaError_t unpack_hermitian(const double2* M, int n, int64_t r0, int64_t rows, double2* out, cudaStream_t s) {
  const int nb = (n + 31) / 32;
  unpack_hermitian_kernel<<<dim3(nb, (unsigned)((rows + 31) / 32)), 256, 0, s>>>(M, n, r0, rows, out);
  return cudaGetLastError();
}

cudaError_t split_full_triple(const double2* M, int n, int nt, float4* hl, float2* t, cudaStream_t s) {
  split_full_kernel<<<nt * nt, 256, 0, s>>>(M, n, nt, hl, t);
  return cudaGetLastError();
}

cudaError_t split_double_float(const double2* M, int64_t n, float4* out, cudaStream_t s) {
  split_df_kernel<<<1024, 256, 0, s>>>(M, n, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
cudaError_t precompute_dense(const double2* T, int64_t n_vis, int n, int64_t ld, const double* w,
                             const double2* d, int nt, double2* Mt, double2* dbar, cudaStream_t s, bool tc) {
  cudaError_t e;
  if (tc) {
    e = herk_dense_tc(T, n_vis, n, ld, w, nt, Mt, s);   // seven-digit slice products (herk_tc.cu)
  } else {
    dim3 grid((unsigned)(tri_count(nt) * 4), 1, 1);
    herk_f64_kernel<<<grid, 256, 0, s>>>(T, ld, w, n_vis, n, Mt);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  cudaMemsetAsync(dbar, 0, sizeof(double2) * (size_t)nt * BEOR_TB, s);
  // chunks of 1024 visibilities of a large T, so that its rows stream from memory on every SM
  int64_t kchunk = n_vis <= 4096 ? 4096 : 1024;
  while ((n_vis + kchunk - 1) / kchunk > 65535) kchunk *= 2;
  launch_xh_w_d(T, ld, 0, w, d, 0, n_vis, n, kchunk, dbar, 0, 1, s);
  return cudaGetLastError();
}

cudaError_t precompute_factored(const double2* A, const double2* W, int nf, int64_t ntb, int ncells,
                                int nx, const double* w, const double2* d, int n, int nt,
                                double2* G_scratch, double2* u_scratch, double2* P_scratch, double2* Mt, double2* dbar,
                                cudaStream_t s) {
  const int nb = (ncells + 15) / 16, tiles = nb * (nb + 1) / 2;
  gram_cells_kernel<<<dim3((tiles + 3) / 4, nf), 128, 0, s>>>(A, w, ntb, ncells, tiles, G_scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned units = (unsigned)std::min<int64_t>(tri_count(nt) * (BEOR_TB / AM_COLS), 65535);
  if (P_scratch) {
    weight_products_kernel<<<(unsigned)(((int64_t)nf * nx * nx + 255) / 256), 256, 0, s>>>(W, nf, nx, P_scratch);
    assemble_M_kernel<true><<<units, AM_THREADS, 0, s>>>(G_scratch, W, P_scratch, nf, ncells, nx, n, nt, Mt);
  } else {
    assemble_M_kernel<false><<<units, AM_THREADS, 0, s>>>(G_scratch, W, nullptr, nf, ncells, nx, n, nt, Mt);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  cudaMemsetAsync(u_scratch, 0, sizeof(double2) * (size_t)nf * ncells, s);
  int64_t kchunk = 2048;
  launch_xh_w_d(A, ncells, ntb * ncells, w, d, ntb, ntb, ncells, kchunk, u_scratch, ncells, nf, s);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int np = nt * BEOR_TB;
  assemble_dbar_kernel<<<(np + 255) / 256, 256, 0, s>>>(u_scratch, W, nf, ncells, nx, n, np, dbar);
  return cudaGetLastError();
}

}  // namespace beor
