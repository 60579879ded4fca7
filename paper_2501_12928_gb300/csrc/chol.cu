// Blocked right-looking complex Cholesky of Sigma = M + Phi^-1 for a batch of
// problems, the triangular solves for abar = Sigma^-1 dbar, and the lnL
// assembly (lnL = -1/2 log|Phi| - 1/2 log|Sigma| + 1/2 dbar^H abar).
//
// Kernels here serve both precisions:
//  * prior / init:  Phi^-1 from phi (one amplitude per k bin, Eq. for P(k_i)),
//                   log|Phi|, and the working matrix W = M + diag(Phi^-1);
//  * diag:          float64 factorisation of the 128 x 128 diagonal block,
//                   log|Sigma| accumulation, status, and its inverse (float64;
//                   on the fp32 pipe, with bf16 slices, on the mixed path);
//  * panel/trail:   float64 tile GEMMs (the float64 comparator path);
//  * solve:         blocked forward / backward substitution;
//  * lnl:           q = Re(dbar^H abar), or its residual-corrected form, and lnL.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "beor_common.cuh"
#include "beor_internal.h"
#include "diag_common.cuh"

namespace beor {

// --------------------------------------------------------------------------
// workspace element access
// --------------------------------------------------------------------------

__device__ __forceinline__ void tile_of(int64_t t, int& I, int& J) {
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((int64_t)i * (i + 1) / 2 > t) --i;
  while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
  I = i;
  J = (int)(t - (int64_t)i * (i + 1) / 2);
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}

// --------------------------------------------------------------------------
// prior: Phi^-1 per row, log|Phi| per problem, reset of the per-problem sums
// --------------------------------------------------------------------------
__global__ void prior_kernel(BatchView v) {
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const SetDesc sd = v.sets[pr.set];
  const double* phi = sd.phi + (int64_t)pr.b * sd.n_k;
  const double ln10 = 2.302585092994045684;
  __shared__ double red[33];
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  // a non-finite phi (possible only for device-memory input, which the host
  // does not read) marks the point; every later kernel skips it
  for (int i = threadIdx.x; i < sd.n_k; i += blockDim.x)
    if (!isfinite(phi[i])) s_bad = 1;
  // the float64 powers and logarithm (about a thousand cycles each) once per
  // k bin, not once per mode (44 us -> 9 us at 3280 modes)
  constexpr int KB = 256;
  __shared__ double s_inv[KB], s_log[2];
  const bool cached = sd.n_k <= KB;
  for (int i = threadIdx.x; cached && i < sd.n_k; i += blockDim.x) s_inv[i] = exp10(-phi[i]);
  if (threadIdx.x == 0) s_log[0] = log(sd.lssm_prior_var);
  if (threadIdx.x == 32) s_log[1] = 1.0 / sd.lssm_prior_var;
  __syncthreads();
  double acc = 0.0;
  const int np = pr.nt * BEOR_TB;
  for (int j = threadIdx.x; j < np; j += blockDim.x) {
    double inv = 1.0;
    if (j < pr.n) {
      int kb = sd.kbin[j];
      if (kb >= 0) {
        double ph = phi[kb];
        inv = cached ? s_inv[kb] : exp10(-ph);
        acc += ph * ln10;
      } else {
        inv = s_log[1];
        acc += s_log[0];
      }
    }
    v.phi_inv[pr.row_off + j] = inv;
  }
  double tot = block_sum(acc, red);   // its barriers also order the writes of s_bad
  if (threadIdx.x == 0) {
    v.logdet_phi[p] = tot;
    v.logdet_sigma[p] = 0.0;
    v.status[p] = s_bad ? STATUS_BAD_PHI : 0;
    v.resid[p] = 0.0;
  }
}

// grid (problem, tile): problems fastest, so the problems of one instrument
// read each tile of M from L2 rather than from HBM.  Float64 path: M as is.
__global__ void __launch_bounds__(256) init_ws_f64_kernel(BatchView v) {
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const SetDesc sd = v.sets[pr.set];
  const int64_t ntiles = tri_count(pr.nt);
  for (int64_t t = blockIdx.y; t < ntiles; t += gridDim.y) {
    int I, J;
    tile_of(t, I, J);
    if (!BEOR_INBOUNDS(v.flags, pr.ws_off + (t + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_INIT_WS)) return;
    const double2* __restrict__ src = sd.M + t * BEOR_TILE_ELEMS;
    double2* __restrict__ dst = reinterpret_cast<double2*>(v.ws) + pr.ws_off + t * BEOR_TILE_ELEMS;
    const double* pinv = v.phi_inv + pr.row_off + (int64_t)I * BEOR_TB;
    for (int e = threadIdx.x; e < BEOR_TILE_ELEMS; e += blockDim.x) {
      double2 m = src[e];
      if (I == J && (e % BEOR_TB) == (e / BEOR_TB)) {
        m.x += pinv[e % BEOR_TB];
        m.y = 0.0;
      }
      dst[e] = m;
    }
  }
}

// Mixed path: copy the double-float M; the diagonal gets Phi^-1 in
// double-float arithmetic (no float64 instruction per element).
__global__ void __launch_bounds__(256) init_ws_df_kernel(BatchView v) {
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const SetDesc sd = v.sets[pr.set];
  const int64_t ntiles = tri_count(pr.nt);
  for (int64_t t = blockIdx.y; t < ntiles; t += gridDim.y) {
    int I, J;
    tile_of(t, I, J);
    if (!BEOR_INBOUNDS(v.flags, pr.ws_off + (t + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_INIT_WS)) return;
    const float4* __restrict__ src = sd.Mdf + t * BEOR_TILE_ELEMS;
    float4* __restrict__ dst = reinterpret_cast<float4*>(v.ws) + pr.ws_off + t * BEOR_TILE_ELEMS;
    for (int e = threadIdx.x; e < BEOR_TILE_ELEMS; e += blockDim.x) dst[e] = src[e];
    if (I != J) continue;                 // uniform per CTA
    __syncthreads();                      // the copy of every diagonal element has landed
    if (threadIdx.x < BEOR_TB) {
      const int r = threadIdx.x;
      const int e = r * BEOR_TB + r;
      const float4 m = src[e];
      const dfl w = df_add(dfl{m.x, m.y}, df_from_double(v.phi_inv[pr.row_off + (int64_t)I * BEOR_TB + r]));
      dst[e] = make_float4(w.hi, w.lo, 0.0f, 0.0f);
    }
  }
}

cudaError_t launch_prior_init(const BatchView& v, bool mixed, cudaStream_t s) {
  prior_kernel<<<v.P, 256, 0, s>>>(v);
  dim3 g(v.P, (unsigned)std::min<int64_t>(tri_count(v.max_nt), 65535));
  if (mixed)
    init_ws_df_kernel<<<g, 256, 0, s>>>(v);
  else
    init_ws_f64_kernel<<<g, 256, 0, s>>>(v);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// diagonal blocks: Cholesky factor, log-det, status, and the inverse of the
// block, with, on the mixed path, the bf16 slices of its rows
//
// lnL on the mixed path factors them in fixed point (diag_tc.cu).  The posterior
// mean stays with float64: its amplitudes are Sigma^-1 times the
// float64-accurate residual's rounding (relative 5e-8 at kappa ~ 1e8, 3280
// modes), so that any other rounding of the factor moves them by as much,
// while the quadratic form of lnL does not see it (1e-10).
// --------------------------------------------------------------------------
cudaError_t launch_diag(const BatchView& v, int k, bool mixed, int active, cudaStream_t s, int prio) {
  if (mixed && !v.mean) return launch_diag_tc(v, k, active, s, prio);
  return launch_diag_cluster(v, k, mixed, active, s, prio);
}

// --------------------------------------------------------------------------
// float64 panel: L_ik = A_ik Linv_kk^H for i > k, R rows per CTA
//
// Bound by the float64 pipe.  Column c needs the terms m <= c only (Linv is
// lower triangular; the terms left out are exact zeros): warp w takes the
// eight-column groups w and 15 - w, which together have the same number of
// terms for every w; lane = (row, part of the group's columns).  Few rows per
// CTA where the batch is small, so that the work reaches every SM: one point of
// 3280 modes took 26 ms in at most 50 CTAs of 64 rows (with the zeros) and takes
// 3.3 ms with R = 8.
// --------------------------------------------------------------------------
template <int R>
__global__ void __launch_bounds__(256) panel_f64_kernel(BatchView v, int kg) {
  __shared__ double2 xs[BEOR_TB][R];
  constexpr int NC = R / 4;             // columns per thread and group
  const int p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;
  const int i = k + 1 + blockIdx.x / (BEOR_TB / R);
  if (k < 0 || i >= pr.nt || v.status[p] != 0) return;
  const int r0 = (blockIdx.x % (BEOR_TB / R)) * R;
  double2* tile = reinterpret_cast<double2*>(v.ws) + pr.ws_off + tri_index(i, k) * BEOR_TILE_ELEMS + r0;
  const double2* __restrict__ linv = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
  for (int e = threadIdx.x; e < BEOR_TB * R; e += 256) xs[e / R][e % R] = tile[(e / R) * BEOR_TB + e % R];
  __syncthreads();   // every element of these rows is read
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane % R, q = lane / R;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int g = h ? 15 - warp : warp, c0 = 8 * g + q * NC;
    double ar[NC], ai[NC];
#pragma unroll
    for (int b = 0; b < NC; ++b) ar[b] = ai[b] = 0.0;
#pragma unroll 4
    for (int m = 0; m < 8 * g + 8; ++m) {
      const double2 x = xs[m][r];
#pragma unroll
      for (int b = 0; b < NC; ++b) {
        const int c = c0 + b;
        const double2 y = m <= c ? linv[pk(c, m)] : make_double2(0.0, 0.0);
        // x * conj(y)
        ar[b] = fma(x.x, y.x, fma(x.y, y.y, ar[b]));
        ai[b] = fma(x.y, y.x, fma(-x.x, y.y, ai[b]));
      }
    }
#pragma unroll
    for (int b = 0; b < NC; ++b) tile[(c0 + b) * BEOR_TB + r] = make_double2(ar[b], ai[b]);
  }
}

cudaError_t launch_panel_f64(const BatchView& v, int k, cudaStream_t s) {
  const int rows = v.max_nt - 1 - k;   // block rows
  if (rows <= 0) return cudaSuccess;
  // 32 rows per CTA read the inverse block (132 KB) a quarter as often; from
  // four such CTAs per SM on
  if ((int64_t)rows * 4 * v.P >= 4 * device_sms())
    panel_f64_kernel<32><<<dim3(rows * 4, v.P), 256, 0, s>>>(v, k);
  else
    panel_f64_kernel<8><<<dim3(rows * 16, v.P), 256, 0, s>>>(v, k);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// float64 trailing update: A_ij -= L_ik L_jk^H, k < j <= i, 64 x 64 sub-tiles
// --------------------------------------------------------------------------
__global__ void __launch_bounds__(256) trail_f64_kernel(BatchView v, int kg) {
  __shared__ double2 xs[16][64];
  __shared__ double2 ys[16][64];
  const int p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;
  const int T = k < 0 ? 0 : pr.nt - k - 1;
  const int64_t t = blockIdx.x >> 2;
  if (T <= 0 || t >= tri_count(T) || v.status[p] != 0) return;
  const int si = (blockIdx.x >> 1) & 1, sj = blockIdx.x & 1;
  int a, b;
  tile_of(t, a, b);
  const int i = k + 1 + a, j = k + 1 + b;
  if (i == j && si < sj) return;   // upper part of a diagonal tile is never read
  double2* ws = reinterpret_cast<double2*>(v.ws) + pr.ws_off;
  const double2* X = ws + tri_index(i, k) * BEOR_TILE_ELEMS + si * 64;
  const double2* Y = ws + tri_index(j, k) * BEOR_TILE_ELEMS + sj * 64;
  double2* C = ws + tri_index(i, j) * BEOR_TILE_ELEMS;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double ar[4][4], ai[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int w = 0; w < 4; ++w) ar[q][w] = ai[q][w] = 0.0;
  for (int m0 = 0; m0 < BEOR_TB; m0 += 16) {
    for (int e = threadIdx.x; e < 16 * 64; e += 256) {
      int mm = e / 64, r = e % 64;
      xs[mm][r] = X[(m0 + mm) * BEOR_TB + r];
      ys[mm][r] = Y[(m0 + mm) * BEOR_TB + r];
    }
    __syncthreads();
#pragma unroll 4
    for (int mm = 0; mm < 16; ++mm) {
      double2 x[4], y[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        x[q] = xs[mm][ty * 4 + q];
        y[q] = ys[mm][tx * 4 + q];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          ar[q][w] = fma(x[q].x, y[w].x, fma(x[q].y, y[w].y, ar[q][w]));
          ai[q][w] = fma(x[q].y, y[w].x, fma(-x[q].x, y[w].y, ai[q][w]));
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      int r = si * 64 + ty * 4 + q, c = sj * 64 + tx * 4 + w;
      double2 cv = C[c * BEOR_TB + r];
      cv.x -= ar[q][w];
      cv.y -= ai[q][w];
      C[c * BEOR_TB + r] = cv;
    }
}

cudaError_t launch_trail_f64(const BatchView& v, int k, cudaStream_t s) {
  int T = v.max_nt - k - 1;
  if (T <= 0) return cudaSuccess;
  int64_t nblk = tri_count(T) * 4;
  trail_f64_kernel<<<dim3((unsigned)nblk, v.P), 256, 0, s>>>(v, k);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// Triangular solves with the factor: out = L^-H L^-1 rhs, blocked by 128.
// One launch per block step covers every problem: CTA (i, p) applies the
// update of block row i with the block just solved; the CTA that completes
// the next block row also applies that block's float64 inverse, so a step's
// critical path is one tile update plus one 128 x 128 float64 matvec.
// Off-diagonal products: float64 for the float64 path, double-float (fp32
// pairs) for the mixed path's double-float factor.
// --------------------------------------------------------------------------
struct CAcc {          // complex accumulator
  double2 d;           // float64 path
  dfl re, im;          // double-float path: hi = error-free running sum, lo = its accumulated errors
};

__device__ __forceinline__ void cacc_zero(CAcc& a) {
  a.d = make_double2(0.0, 0.0);
  a.re = dfl{0.0f, 0.0f};
  a.im = dfl{0.0f, 0.0f};
}
// a += L * y (conj_l: a += conj(L) * y); y given as double2 and as double-float pairs
__device__ __forceinline__ void cacc_mac(CAcc& a, const double2* L, double2 y, dfl, dfl, bool conj_l) {
  const double2 l = *L;
  const double li = conj_l ? -l.y : l.y;
  a.d.x = fma(l.x, y.x, fma(-li, y.y, a.d.x));
  a.d.y = fma(l.x, y.y, fma(li, y.x, a.d.y));
}
__device__ __forceinline__ void cacc_mac(CAcc& a, const float4* L, double2, dfl yr, dfl yi, bool conj_l) {
  const float4 l = *L;
  const float lih = conj_l ? -l.z : l.z, lil = conj_l ? -l.w : l.w;
  // re += lr yr - li yi, im += lr yi + li yr
  dot2_acc(a.re, l.x, l.y, yr.hi, yr.lo);
  dot2_acc(a.re, -lih, -lil, yi.hi, yi.lo);
  dot2_acc(a.im, l.x, l.y, yi.hi, yi.lo);
  dot2_acc(a.im, lih, lil, yr.hi, yr.lo);
}
__device__ __forceinline__ double2 cacc_get(const CAcc& a, const double2*) { return a.d; }
__device__ __forceinline__ double2 cacc_get(const CAcc& a, const float4*) {
  return make_double2((double)a.re.hi + (double)a.re.lo, (double)a.im.hi + (double)a.im.lo);
}
__device__ __forceinline__ void cacc_add(CAcc& a, const CAcc& b) {
  a.d.x += b.d.x;
  a.d.y += b.d.y;
  dfl s = df_two_sum(a.re.hi, b.re.hi);
  a.re = dfl{s.hi, s.lo + (a.re.lo + b.re.lo)};
  s = df_two_sum(a.im.hi, b.im.hi);
  a.im = dfl{s.hi, s.lo + (a.im.lo + b.im.lo)};
}

// sum over the 8 lanes of an aligned lane octet (xor 1, 2, 4)
__device__ __forceinline__ void cacc_reduce8(CAcc& a, const double2*) {
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    a.d.x += __shfl_xor_sync(0xffffffffu, a.d.x, o);
    a.d.y += __shfl_xor_sync(0xffffffffu, a.d.y, o);
  }
}
__device__ __forceinline__ void cacc_reduce8(CAcc& a, const float4*) {
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    CAcc b;
    b.d = make_double2(0.0, 0.0);
    b.re.hi = __shfl_xor_sync(0xffffffffu, a.re.hi, o);
    b.re.lo = __shfl_xor_sync(0xffffffffu, a.re.lo, o);
    b.im.hi = __shfl_xor_sync(0xffffffffu, a.im.hi, o);
    b.im.lo = __shfl_xor_sync(0xffffffffu, a.im.lo, o);
    cacc_add(a, b);
  }
}

// The inverse diagonal block times a block of the right-hand side, y = Linv rk
// or (herm) Linv^H rk, into out; 256 threads.  Float64 blocks (the float64 path
// and the posterior mean): one thread per row, the loads unrolled ahead of the
// chain of float64 products.
__device__ __forceinline__ void diag_apply(const double2* __restrict__ li, const double2* rk, const dfl*, const dfl*,
                                           CAcc*, double2* out, bool herm) {
  const int t = threadIdx.x;
  if (t >= BEOR_TB) return;
  double sr = 0.0, si = 0.0;
  const int m0 = herm ? t : 0, m1 = herm ? BEOR_TB - 1 : t;
  constexpr int U = 8;
  double2 a[U];
#pragma unroll
  for (int u = 0; u < U; ++u) a[u] = li[herm ? pk(min(m0 + u, m1), t) : pk(t, min(m0 + u, m1))];
  for (int m = m0; m <= m1; m += U) {
    double2 n[U];
#pragma unroll
    for (int u = 0; u < U; ++u) n[u] = li[herm ? pk(min(m + U + u, m1), t) : pk(t, min(m + U + u, m1))];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (m + u > m1) break;
      const double2 q = rk[m + u];
      const double ai = herm ? -a[u].y : a[u].y;
      sr = fma(a[u].x, q.x, fma(-ai, q.y, sr));
      si = fma(a[u].x, q.y, fma(ai, q.x, si));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] = n[u];
  }
  out[t] = make_double2(sr, si);
}
// Double-float blocks (lnL on the mixed path): compensated products on the fp32
// pipe, as for the off-diagonal tiles.  33,000 float64 products of one block
// take 10 us on one SM, and as a chain per row with uncoalesced loads they took
// 40 us of a step; eight lanes per row (forward) or two threads per column
// (backward) read the block coalesced.
__device__ __forceinline__ void diag_apply(const float4* __restrict__ li, const double2*, const dfl* rkr,
                                           const dfl* rki, CAcc* part, double2* out, bool herm) {
  const int tid = threadIdx.x;
  if (!herm) {
    const int lane8 = tid & 7;
    for (int t = tid >> 3; t < BEOR_TB; t += 32) {
      CAcc a;
      cacc_zero(a);
#pragma unroll 4
      for (int m = lane8; m <= t; m += 8)
        cacc_mac(a, li + pk(t, m), make_double2(0.0, 0.0), rkr[m], rki[m], false);
      cacc_reduce8(a, li);
      if (lane8 == 0) out[t] = cacc_get(a, li);
    }
  } else {
    const int t = tid & 127, half = tid >> 7;
    CAcc a;
    cacc_zero(a);
#pragma unroll 4
    for (int m = t + half; m < BEOR_TB; m += 2)
      cacc_mac(a, li + pk(m, t), make_double2(0.0, 0.0), rkr[m], rki[m], true);
    if (half) part[t] = a;
    __syncthreads();
    if (!half) {
      cacc_add(a, part[t]);
      out[t] = cacc_get(a, li);
    }
  }
}

// Forward step k (k = -1: only y_0).  CTA (i, p), i = k+1 .. nt-1:
// r_i -= L_ik y_k; the CTA with i == k+1 then sets y_{k+1} = Linv r_{k+1}.
// DV: element type of the inverse diagonal blocks.
template <typename WS, typename DV>
__global__ void __launch_bounds__(256) fwd_step_kernel(BatchView v, int kg, const double2* __restrict__ rhs) {
  __shared__ double2 yk[BEOR_TB];
  __shared__ dfl ykr[BEOR_TB], yki[BEOR_TB];
  __shared__ CAcc part[BEOR_TB];
  __shared__ double2 rk[BEOR_TB];
  __shared__ dfl rkr[BEOR_TB], rki[BEOR_TB];
  auto set_rk = [&](int t, double2 q) {
    rk[t] = q;
    if (std::is_same<DV, float4>::value) {
      rkr[t] = df_from_double(q.x);
      rki[t] = df_from_double(q.y);
    }
  };
  const int p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;   // this problem's step (-1: start)
  if (k < -1) return;
  const int i = k + 1 + blockIdx.x;
  if (i >= pr.nt || prob_skipped(v.status[p])) return;
  if (!BEOR_INBOUNDS(v.flags, pr.row_off + (int64_t)pr.nt * BEOR_TB <= v.rows, BC_SOLVE_VEC) ||
      !BEOR_INBOUNDS(v.flags, k < 0 || pr.ws_off + (tri_index(i, k) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_SOLVE_VEC))
    return;
  const int tid = threadIdx.x;
  double2* r = v.vec_t + pr.row_off;
  double2* y = v.vec_y + pr.row_off;
  if (k < 0) {
    // initial step: r = rhs for all rows of block 0 handled here, other rows by their own CTAs
    if (tid < BEOR_TB) r[i * BEOR_TB + tid] = rhs[pr.row_off + i * BEOR_TB + tid];
    if (i != 0) return;
    __syncthreads();
    if (tid < BEOR_TB) set_rk(tid, r[tid]);
    __syncthreads();
    diag_apply(reinterpret_cast<const DV*>(v.dinv) + pr.dinv_off, rk, rkr, rki, part, yk, false);
    __syncthreads();
    if (tid < BEOR_TB) y[tid] = yk[tid];
    return;
  }
  if (tid < BEOR_TB) {
    const double2 q = y[k * BEOR_TB + tid];
    yk[tid] = q;
    ykr[tid] = df_from_double(q.x);
    yki[tid] = df_from_double(q.y);
  }
  __syncthreads();
  const WS* t = reinterpret_cast<const WS*>(v.ws) + pr.ws_off + tri_index(i, k) * BEOR_TILE_ELEMS;
  const int row = tid & 127, half = tid >> 7;
  CAcc a;
  cacc_zero(a);
#pragma unroll 4
  for (int m = half * 64; m < half * 64 + 64; ++m)
    cacc_mac(a, t + m * BEOR_TB + row, yk[m], ykr[m], yki[m], false);
  if (half) part[row] = a;
  __syncthreads();
  if (!half) {
    cacc_add(a, part[row]);
    const double2 s = cacc_get(a, t);
    double2 cur = r[i * BEOR_TB + row];
    cur.x -= s.x;
    cur.y -= s.y;
    r[i * BEOR_TB + row] = cur;
    if (i == k + 1) set_rk(row, cur);
  }
  if (i != k + 1) return;
  __syncthreads();
  diag_apply(reinterpret_cast<const DV*>(v.dinv) + pr.dinv_off + (int64_t)i * DG_PACK, rk, rkr, rki, part, yk, false);
  __syncthreads();
  if (tid < BEOR_TB) y[i * BEOR_TB + tid] = yk[tid];
}

// Backward step k (k = nt: only x_{nt-1} for each problem).  CTA (i, p),
// i = 0 .. k-1: r_i -= L_ki^H x_k; the CTA with i == k-1 then sets
// x_{k-1} = Linv^H r_{k-1}.  Steps run from the largest nt down; problems
// with fewer tiles join when k < their nt.
template <typename WS, typename DV>
__global__ void __launch_bounds__(256) bwd_step_kernel(BatchView v, int k, double2* __restrict__ out) {
  __shared__ double2 xk[BEOR_TB];
  __shared__ dfl xkr[BEOR_TB], xki[BEOR_TB];
  __shared__ double2 rk[BEOR_TB];
  __shared__ dfl rkr[BEOR_TB], rki[BEOR_TB];
  __shared__ CAcc part[BEOR_TB];
  auto set_rk = [&](int t, double2 q) {
    rk[t] = q;
    if (std::is_same<DV, float4>::value) {
      rkr[t] = df_from_double(q.x);
      rki[t] = df_from_double(q.y);
    }
  };
  const int p = blockIdx.y;
  const Prob pr = v.prob[p];
  if (prob_skipped(v.status[p])) return;
  if (!BEOR_INBOUNDS(v.flags, pr.row_off + (int64_t)pr.nt * BEOR_TB <= v.rows, BC_SOLVE_VEC)) return;
  const int tid = threadIdx.x;
  double2* r = v.vec_t + pr.row_off;
  double2* x = out + pr.row_off;
  const double2* y = v.vec_y + pr.row_off;
  if (k >= pr.nt) {
    // start: r = y; the CTA for the last block applies Linv^H
    const int i = blockIdx.x;
    if (i >= pr.nt) return;
    if (tid < BEOR_TB) r[i * BEOR_TB + tid] = y[i * BEOR_TB + tid];
    if (k != pr.nt || i != pr.nt - 1) return;
    __syncthreads();
    if (tid < BEOR_TB) set_rk(tid, r[i * BEOR_TB + tid]);
    __syncthreads();
    diag_apply(reinterpret_cast<const DV*>(v.dinv) + pr.dinv_off + (int64_t)i * DG_PACK, rk, rkr, rki, part, xk, true);
    __syncthreads();
    if (tid < BEOR_TB) x[i * BEOR_TB + tid] = xk[tid];
    return;
  }
  const int i = blockIdx.x;
  if (i >= k) return;
  if (tid < BEOR_TB) {
    const double2 q = x[k * BEOR_TB + tid];
    xk[tid] = q;
    xkr[tid] = df_from_double(q.x);
    xki[tid] = df_from_double(q.y);
  }
  __syncthreads();
  // r_i[c] -= sum_m conj(L_ki[m][c]) x_k[m]: tile (k, i) is column-major, so
  // column c is 128 contiguous elements.  A warp takes 4 columns at a time,
  // 8 lanes per column on interleaved m (each load instruction reads four
  // 128-byte segments), and sums the 8 partials by shuffles.
  const WS* t = reinterpret_cast<const WS*>(v.ws) + pr.ws_off + tri_index(k, i) * BEOR_TILE_ELEMS;
  const int warp = tid >> 5, lane = tid & 31, cl = lane >> 3, mo = lane & 7;
#pragma unroll 1
  for (int it = 0; it < 4; ++it) {
    const int c = warp * 16 + it * 4 + cl;
    CAcc a;
    cacc_zero(a);
#pragma unroll 4
    for (int u = 0; u < 16; ++u) {
      const int m = mo + 8 * u;
      cacc_mac(a, t + c * BEOR_TB + m, xk[m], xkr[m], xki[m], true);
    }
    cacc_reduce8(a, t);
    if (mo == 0) {
      const double2 sv = cacc_get(a, t);
      double2 cur = r[i * BEOR_TB + c];
      cur.x -= sv.x;
      cur.y -= sv.y;
      r[i * BEOR_TB + c] = cur;
      if (i == k - 1) set_rk(c, cur);
    }
  }
  if (i != k - 1) return;
  __syncthreads();
  diag_apply(reinterpret_cast<const DV*>(v.dinv) + pr.dinv_off + (int64_t)i * DG_PACK, rk, rkr, rki, part, xk, true);
  __syncthreads();
  if (tid < BEOR_TB) x[i * BEOR_TB + tid] = xk[tid];
}


// Forward step k of y = L^-1 rhs (k = -1: r = rhs and y_0), every problem.
cudaError_t launch_fwd_step(const BatchView& v, bool mixed, const double2* rhs, int k, cudaStream_t s, int prio) {
  const int nb = k < 0 ? v.max_nt : v.max_nt - k - 1;
  if (nb <= 0) return cudaSuccess;
  auto kern = !mixed ? fwd_step_kernel<double2, double2>
                     : v.mean ? fwd_step_kernel<float4, double2> : fwd_step_kernel<float4, float4>;
  return launch_prio(kern, dim3(nb, v.P), dim3(256), 0, s, prio, v, k, rhs);
}

// out = L^-H y (y in vec_y), every problem.
template <typename WS, typename DV>
static cudaError_t bwd_impl(const BatchView& v, double2* out, cudaStream_t s) {
  const int nt = v.max_nt;
  bwd_step_kernel<WS, DV><<<dim3(nt, v.P), 256, 0, s>>>(v, nt, out);
  for (int k = nt - 1; k >= 1; --k) {
    // problems whose last block is k-1 (nt_p == k) start here
    bwd_step_kernel<WS, DV><<<dim3(k, v.P), 256, 0, s>>>(v, k, out);
  }
  return cudaGetLastError();
}

cudaError_t launch_bwd(const BatchView& v, bool mixed, double2* out, cudaStream_t s) {
  if (!mixed) return bwd_impl<double2, double2>(v, out, s);
  return v.mean ? bwd_impl<float4, double2>(v, out, s) : bwd_impl<float4, float4>(v, out, s);
}

cudaError_t launch_solve_fwd(const BatchView& v, bool mixed, const double2* rhs, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int k = -1; k + 1 < v.max_nt && e == cudaSuccess; ++k) e = launch_fwd_step(v, mixed, rhs, k, s, 0);
  return e;
}

cudaError_t launch_solve(const BatchView& v, bool mixed, const double2* rhs, double2* out, cudaStream_t s) {
  cudaError_t e = launch_solve_fwd(v, mixed, rhs, s);
  return e == cudaSuccess ? launch_bwd(v, mixed, out, s) : e;
}

int solve_launch_count(int max_nt) { return 2 * max_nt; }

// --------------------------------------------------------------------------
// dbar of each problem's set into the right-hand-side vector
// --------------------------------------------------------------------------
__global__ void copy_dbar_kernel(BatchView v) {
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const SetDesc sd = v.sets[pr.set];
  const int np = pr.nt * BEOR_TB;
  for (int j = threadIdx.x; j < np; j += blockDim.x) v.vec_b[pr.row_off + j] = sd.dbar[j];
}

cudaError_t launch_copy_dbar(const BatchView& v, cudaStream_t s) {
  copy_dbar_kernel<<<v.P, 256, 0, s>>>(v);
  return cudaGetLastError();
}

// --------------------------------------------------------------------------
// lnL = -1/2 log|Phi| - 1/2 log|Sigma| + 1/2 Re(dbar^H x)
// --------------------------------------------------------------------------
// lnL = -1/2 log|Phi| - 1/2 log|Sigma| + 1/2 q (Eq. for the marginal
// likelihood of the power spectrum).  corr = 0: q = Re(dbar^H x), x the
// (refined) solution.  corr = 1: q from the first solution x~ of the
// approximate factor, corrected with the float64 residual r = dbar - Sigma x~
// (vec_r) and y = L~^-1 r (vec_y):
//   q = dbar^H x~ + x~^H r + r^H Sigma^-1 r,  r^H Sigma^-1 r ~ |y|^2,
// exact but for the last term's factor error, about eta |y|^2 with
// eta ~ sqrt(|y|^2 / q) the relative error of x~ in the Sigma norm.
__global__ void lnl_kernel(BatchView v, int corr) {
  const int p = blockIdx.x;
  const Prob pr = v.prob[p];
  const SetDesc sd = v.sets[pr.set];
  __shared__ double red[33];
  double acc = 0.0, t = 0.0;
  for (int j = threadIdx.x; j < pr.n; j += blockDim.x) {
    double2 d = sd.dbar[j], x = v.vec_x[pr.row_off + j];
    acc += d.x * x.x + d.y * x.y;
    if (corr) {
      const double2 r = v.vec_r[pr.row_off + j], y = v.vec_y[pr.row_off + j];
      acc += x.x * r.x + x.y * r.y;
      t += y.x * y.x + y.y * y.y;
    }
  }
  double q = block_sum(acc, red);
  __syncthreads();
  if (corr) t = block_sum(t, red);
  if (threadIdx.x == 0) {
    if (corr) {
      q += t;
      const double eta = q > 0.0 ? sqrt(t / q) : INFINITY;
      v.resid[p] = eta;
      // estimated remaining error of q above 1e-2 (5e-3 in lnL): flag
      if (v.status[p] == 0 && !(eta * t <= 1e-2)) v.status[p] = -1;
    }
    v.q[p] = q;
    if (v.status[p] == STATUS_BAD_PHI)
      v.lnl[p] = __longlong_as_double(0x7ff8000000000000ll);   // NaN: no likelihood for a non-finite phi
    else if (v.status[p] > 0)
      v.lnl[p] = -INFINITY;
    else
      v.lnl[p] = -0.5 * v.logdet_phi[p] - 0.5 * v.logdet_sigma[p] + 0.5 * q;
  }
}

cudaError_t launch_lnl(const BatchView& v, cudaStream_t s, int corr) {
  lnl_kernel<<<v.P, 256, 0, s>>>(v, corr);
  return cudaGetLastError();
}

}  // namespace beor
