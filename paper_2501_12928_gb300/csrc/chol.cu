// Blocked right-looking complex Cholesky of Sigma = M + Phi^-1 for a batch of
// problems, and the lnL assembly (lnL = -1/2 log|Phi| - 1/2 log|Sigma| + 1/2
// dbar^H abar).
//
//  * prior / init:  Phi^-1 from phi (one amplitude per k bin, Eq. for P(k_i)),
//                   log|Phi|, and the working matrix W = M + diag(Phi^-1);
//  * diag:          choice of the diagonal blocks' kernel (diag_tc.cu,
//                   diag_cluster.cu);
//  * panel/trail:   float64 tile GEMMs (the float64 comparator path);
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
// float64 trailing update: A_ij -= L_ik L_jk^H, k < j <= i, 32 x 32 sub-tiles
//
// Bound by the float64 pipe: a sub-tile takes 0.13 ms of one SM.  With 64 x 64
// sub-tiles (0.5 ms) the late steps of a small batch, of fewer sub-tiles than a
// few per SM, left SMs idle for up to that long: one point of 3280 modes 45.2 ms,
// now 39.9, with the pipe busy throughout.
// --------------------------------------------------------------------------
constexpr int TF_S = 32, TF_N = BEOR_TB / TF_S, TF_K = 32, TF_Q = TF_S / 16;   // sub-tile, per side, terms at once, per thread
__global__ void __launch_bounds__(256) trail_f64_kernel(BatchView v, int kg) {
  __shared__ double2 xs[TF_K][TF_S];
  __shared__ double2 ys[TF_K][TF_S];
  const int p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = kg - pr.k_off;
  const int T = k < 0 ? 0 : pr.nt - k - 1;
  const int64_t t = blockIdx.x / (TF_N * TF_N);
  if (T <= 0 || t >= tri_count(T) || v.status[p] != 0) return;
  const int si = blockIdx.x / TF_N % TF_N, sj = blockIdx.x % TF_N;
  int a, b;
  tile_of(t, a, b);
  const int i = k + 1 + a, j = k + 1 + b;
  if (i == j && si < sj) return;   // upper part of a diagonal tile is never read
  double2* ws = reinterpret_cast<double2*>(v.ws) + pr.ws_off;
  const double2* X = ws + tri_index(i, k) * BEOR_TILE_ELEMS + si * TF_S;
  const double2* Y = ws + tri_index(j, k) * BEOR_TILE_ELEMS + sj * TF_S;
  double2* C = ws + tri_index(i, j) * BEOR_TILE_ELEMS;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double ar[TF_Q][TF_Q], ai[TF_Q][TF_Q];
#pragma unroll
  for (int q = 0; q < TF_Q; ++q)
#pragma unroll
    for (int w = 0; w < TF_Q; ++w) ar[q][w] = ai[q][w] = 0.0;
  for (int m0 = 0; m0 < BEOR_TB; m0 += TF_K) {
#pragma unroll
    for (int e = threadIdx.x; e < TF_K * TF_S; e += 256) {
      const int mm = e / TF_S, r = e % TF_S;
      xs[mm][r] = X[(m0 + mm) * BEOR_TB + r];
      ys[mm][r] = Y[(m0 + mm) * BEOR_TB + r];
    }
    __syncthreads();
#pragma unroll 4
    for (int mm = 0; mm < TF_K; ++mm) {
      double2 x[TF_Q], y[TF_Q];
#pragma unroll
      for (int q = 0; q < TF_Q; ++q) {
        x[q] = xs[mm][ty * TF_Q + q];
        y[q] = ys[mm][tx * TF_Q + q];
      }
#pragma unroll
      for (int q = 0; q < TF_Q; ++q)
#pragma unroll
        for (int w = 0; w < TF_Q; ++w) {
          ar[q][w] = fma(x[q].x, y[w].x, fma(x[q].y, y[w].y, ar[q][w]));
          ai[q][w] = fma(x[q].y, y[w].x, fma(-x[q].x, y[w].y, ai[q][w]));
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < TF_Q; ++q)
#pragma unroll
    for (int w = 0; w < TF_Q; ++w) {
      const int r = si * TF_S + ty * TF_Q + q, c = sj * TF_S + tx * TF_Q + w;
      double2 cv = C[c * BEOR_TB + r];
      cv.x -= ar[q][w];
      cv.y -= ai[q][w];
      C[c * BEOR_TB + r] = cv;
    }
}

cudaError_t launch_trail_f64(const BatchView& v, int k, cudaStream_t s) {
  int T = v.max_nt - k - 1;
  if (T <= 0) return cudaSuccess;
  int64_t nblk = tri_count(T) * TF_N * TF_N;
  trail_f64_kernel<<<dim3((unsigned)nblk, v.P), 256, 0, s>>>(v, k);
  return cudaGetLastError();
}

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
