// Triangular solves with the factor (both precisions).
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "diag_common.cuh"

namespace beor {

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

// --------------------------------------------------------------------------
// The same steps for small batches.  A step above takes 35 to 45 us, all of it
// latency: 16 rounds of loads per tile, then the inverse diagonal block in one
// CTA while the others are idle.  Here
//   - step k forms its block of the solution, y_k = Linv_k r_k, in every CTA
//     (33,000 products, cheaper than a launch that waits for one CTA) and
//     then updates the other blocks, 32 rows (or columns) of a tile per CTA;
//   - tile and inverse block are copied to shared memory by cp.async, all in
//     flight at once, before the step waits for the one before
//     (programmatic dependent launch): the factor is final by then;
//   - real and imaginary part of a sum go to two threads.
// Each sum has the operations and the order it has in the kernels above (same
// bits).  Bound by the launch and by the chains: one point of 3280 modes takes
// 5 us a step (35 above), of 2000 modes in float64 30 us (38), whose chains of
// 128 dependent pairs of products alone are 9 us.
// --------------------------------------------------------------------------
constexpr int SOLVE_SPLIT = 4;                       // CTAs per tile
constexpr int SOLVE_ROWS = BEOR_TB / SOLVE_SPLIT;
constexpr int SOLVE_THREADS = 512;
template <typename V>   // V: the factor's real type, double or dfl
struct SolveSmem {
  double2 li[DG_PACK];                 // Linv_k, packed (double2 or float4 elements)
  double2 tile[BEOR_TB * SOLVE_ROWS];  // forward: [column][own row]; backward: [own column][row]
  double2 yk[BEOR_TB];
  double rd[2][BEOR_TB];               // r_k by component
  dfl rf[2][BEOR_TB];
  V yv[2][BEOR_TB];                    // y_k by component
  V part[2][SOLVE_ROWS];
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void to_real(double& o, double x) { o = x; }
__device__ __forceinline__ void to_real(dfl& o, double x) { o = df_from_double(x); }
// one component of acc += l (u + i v) [or conj(l)]: u is y's part of that
// component, v its other part
__device__ __forceinline__ void mac_part(double& acc, const double2* L, bool conj_l, int comp, double u, double v) {
  const double2 l = *L;
  acc = fma(l.x, u, fma((comp == 0) != conj_l ? -l.y : l.y, v, acc));
}
__device__ __forceinline__ void mac_part(dfl& acc, const float4* L, bool conj_l, int comp, dfl u, dfl v) {
  const float4 l = *L;
  const bool neg = (comp == 0) != conj_l;
  dot2_acc(acc, l.x, l.y, u.hi, u.lo);
  dot2_acc(acc, neg ? -l.z : l.z, neg ? -l.w : l.w, v.hi, v.lo);
}
__device__ __forceinline__ void add_part(double& a, double b) { a += b; }
__device__ __forceinline__ void add_part(dfl& a, dfl b) {
  const dfl s = df_two_sum(a.hi, b.hi);
  a = dfl{s.hi, s.lo + (a.lo + b.lo)};
}
__device__ __forceinline__ double shfl_part(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ dfl shfl_part(dfl a, int o) {
  return dfl{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double get_part(double a) { return a; }
__device__ __forceinline__ double get_part(dfl a) { return (double)a.hi + (double)a.lo; }

// yk = Linv rk or (HERM) Linv^H rk.  Float64: 256 threads, one per row and
// component; the two warps of an SM quarter get rows of 160 terms together.
template <bool HERM>
__device__ __forceinline__ void solve_diag(const double2* li, const double (*rd)[BEOR_TB], const dfl (*)[BEOR_TB], dfl*,
                                           double2* yk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= 8) return;
  const int comp = warp & 1, gl = warp < 4 ? 3 - (warp >> 1) : (warp - 4) >> 1;   // group by length, 3 the longest
  const int t = 32 * (HERM ? 3 - gl : gl) + lane;
  double acc = 0.0;
#pragma unroll 4
  for (int m = HERM ? t : 0; m < (HERM ? BEOR_TB : t + 1); ++m)
    mac_part(acc, li + (HERM ? pk(m, t) : pk(t, m)), HERM, comp, rd[comp][m], rd[1 - comp][m]);
  (comp ? yk[t].y : yk[t].x) = acc;
}
// Double-float: forward eight lanes per row, backward two threads per column
// and component; warps of an SM quarter get columns of all lengths.
template <bool HERM>
__device__ __forceinline__ void solve_diag(const float4* li, const double (*)[BEOR_TB], const dfl (*rf)[BEOR_TB], dfl* part,
                                           double2* yk) {
  const int tid = threadIdx.x;
  if (!HERM) {
    const int lane8 = tid & 7;
    for (int t = tid >> 3; t < BEOR_TB; t += SOLVE_THREADS / 8) {
      dfl a[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 2
      for (int m = lane8; m <= t; m += 8)
#pragma unroll
        for (int comp = 0; comp < 2; ++comp) mac_part(a[comp], li + pk(t, m), false, comp, rf[comp][m], rf[1 - comp][m]);
#pragma unroll
      for (int comp = 0; comp < 2; ++comp)
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) add_part(a[comp], shfl_part(a[comp], o));
      if (lane8 == 0) yk[t] = make_double2(get_part(a[0]), get_part(a[1]));
    }
  } else {
    const int warp = tid >> 5, comp = warp >> 3, half = (warp >> 2) & 1;
    const int t = 32 * ((warp + (warp >> 2)) & 3) + (tid & 31);
    dfl a{0.0f, 0.0f};
#pragma unroll 2
    for (int m = t + half; m < BEOR_TB; m += 2) mac_part(a, li + pk(m, t), true, comp, rf[comp][m], rf[1 - comp][m]);
    if (half) part[comp * BEOR_TB + t] = a;
    __syncthreads();
    if (!half) {
      add_part(a, part[comp * BEOR_TB + t]);
      (comp ? yk[t].y : yk[t].x) = get_part(a);
    }
  }
}

// Step k of y = L^-1 src (CTA (SOLVE_SPLIT (i - k - 1) + quarter, p)) or, HERM, of
// out = L^-H src (CTA (SOLVE_SPLIT i + quarter, p), problems join when k < their
// nt).  src: the right-hand side; the running one is vec_t.
template <typename WS, typename DV, bool HERM>
__global__ void __launch_bounds__(SOLVE_THREADS, 1)
    solve_step_kernel(BatchView v, int kg, const double2* __restrict__ src, double2* __restrict__ out) {
  using V = typename std::conditional<std::is_same<WS, float4>::value, dfl, double>::type;
  extern __shared__ __align__(16) unsigned char ss_raw[];
  SolveSmem<V>& sm = *reinterpret_cast<SolveSmem<V>*>(ss_raw);
  dfl* const dpart = reinterpret_cast<dfl*>(sm.yv);   // HERM, DV float4: halves of yk (yv is filled after)
  const int tid = threadIdx.x, p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = HERM ? kg : kg - pr.k_off;   // this problem's step
  const int i = (HERM ? 0 : k + 1) + blockIdx.x / SOLVE_SPLIT, c0 = blockIdx.x % SOLVE_SPLIT * SOLVE_ROWS;
  const bool upd = HERM ? i < k : i < pr.nt;   // has a block to update
  const int ti = HERM ? k : i, tj = HERM ? i : k;
  bool on = k >= 0 && k < pr.nt && (upd || blockIdx.x == 0) && !prob_skipped(v.status[p]);
  on = on && BEOR_INBOUNDS(v.flags, pr.row_off + (int64_t)pr.nt * BEOR_TB <= v.rows, BC_SOLVE_VEC) &&
       BEOR_INBOUNDS(v.flags, !upd || pr.ws_off + (tri_index(ti, tj) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_SOLVE_VEC) &&
       BEOR_INBOUNDS(v.flags, pr.dinv_off + (int64_t)(k + 1) * DG_PACK <= v.dinv_elems, BC_DIAG_DINV);
  if (on) {
    const double2* li = reinterpret_cast<const double2*>(v.dinv) + pr.dinv_off + (int64_t)k * DG_PACK;
    for (int e = tid; e < DG_PACK; e += SOLVE_THREADS) cp_async16(&sm.li[e], li + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (upd) {
      const double2* t = reinterpret_cast<const double2*>(v.ws) + pr.ws_off + tri_index(ti, tj) * BEOR_TILE_ELEMS;
#pragma unroll
      for (int q = 0; q < BEOR_TB * SOLVE_ROWS / SOLVE_THREADS; ++q) {
        const int e = tid + q * SOLVE_THREADS;
        cp_async16(&sm.tile[e], HERM ? t + c0 * BEOR_TB + e : t + e / SOLVE_ROWS * BEOR_TB + c0 + e % SOLVE_ROWS);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // every CTA waits, those without work too: the grid after this one must not
  // run past the one before
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!on) return;
  const bool first = k == (HERM ? pr.nt - 1 : 0);
  const double2* r = (first ? src : v.vec_t) + pr.row_off;
  const int comp = HERM ? tid >> 8 : (tid >> 6) & 1;               // update: component,
  const int own = HERM ? (tid >> 3) & 31 : tid & 31;               // row (column),
  const int ms = HERM ? tid & 7 : (tid >> 5) & 1;                  // part of the sum
  const bool last = upd && (HERM ? ms == 0 : ms == 0 && tid < 128);   // takes the sum
  double cur = 0.0;
  if (tid < BEOR_TB) {
    const double2 q = r[k * BEOR_TB + tid];
    if constexpr (std::is_same<DV, double2>::value) {
      sm.rd[0][tid] = q.x;
      sm.rd[1][tid] = q.y;
    } else {
      sm.rf[0][tid] = df_from_double(q.x);
      sm.rf[1][tid] = df_from_double(q.y);
    }
  }
  if (last) cur = reinterpret_cast<const double*>(r + i * BEOR_TB + c0 + own)[comp];
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();
  solve_diag<HERM>(reinterpret_cast<const DV*>(sm.li), sm.rd, sm.rf, dpart, sm.yk);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if (tid < BEOR_TB) {
    const double2 q = sm.yk[tid];
    if (blockIdx.x == 0) out[pr.row_off + k * BEOR_TB + tid] = q;
    to_real(sm.yv[0][tid], q.x);
    to_real(sm.yv[1][tid], q.y);
  }
  if (!upd) return;
  __syncthreads();
  const WS* t = reinterpret_cast<const WS*>(sm.tile);
  V a{};
  if (HERM) {
    // column own of tile (k, i): eight lanes, interleaved rows
#pragma unroll 4
    for (int u = 0; u < 16; ++u) {
      const int m = ms + 8 * u;
      mac_part(a, t + own * BEOR_TB + m, true, comp, sm.yv[comp][m], sm.yv[1 - comp][m]);
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) add_part(a, shfl_part(a, o));
  } else {
    // row own of tile (i, k): two threads, 64 columns each
    if (tid < 128)
#pragma unroll 4
      for (int m = ms * 64; m < ms * 64 + 64; ++m)
        mac_part(a, t + m * SOLVE_ROWS + own, false, comp, sm.yv[comp][m], sm.yv[1 - comp][m]);
    if (tid < 128 && ms) sm.part[comp][own] = a;
    __syncthreads();
    if (last) add_part(a, sm.part[comp][own]);
  }
  if (last) reinterpret_cast<double*>(v.vec_t + pr.row_off + i * BEOR_TB + c0 + own)[comp] = cur - get_part(a);
}

template <typename WS, typename DV, bool HERM>
static cudaError_t solve_steps(const BatchView& v, const double2* src, double2* out, cudaStream_t s) {
  using V = typename std::conditional<std::is_same<WS, float4>::value, dfl, double>::type;
  auto kern = solve_step_kernel<WS, DV, HERM>;
  static bool init = false;
  if (!init) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SolveSmem<V>));
    init = true;
  }
  cudaError_t e = cudaSuccess;
  for (int j = 0; j < v.max_nt && e == cudaSuccess; ++j) {
    const int k = HERM ? v.max_nt - 1 - j : j, blocks = v.max_nt - 1 - j;   // blocks left to update
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(std::max(1, SOLVE_SPLIT * blocks), v.P);
    cfg.blockDim = dim3(SOLVE_THREADS);
    cfg.dynamicSmemBytes = sizeof(SolveSmem<V>);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = j ? 1 : 0;   // the first step waits for all that the stream holds
    e = cudaLaunchKernelEx(&cfg, kern, v, k, src, out);
  }
  return e;
}
template <bool HERM>
static cudaError_t solve_small(const BatchView& v, bool mixed, const double2* src, double2* out, cudaStream_t s) {
  if (!mixed) return solve_steps<double2, double2, HERM>(v, src, out, s);
  return v.mean ? solve_steps<float4, double2, HERM>(v, src, out, s) : solve_steps<float4, float4, HERM>(v, src, out, s);
}
// The products with the inverse block in every CTA pay until the first step has
// a few waves of CTAs.  Solves of one evaluation, in ms (this way / one CTA):
// mixed, 3280 modes (26 blocks) 8 points 3.3 / 4.1, 16 points 7.3 / 6.8; 1000
// modes (8 blocks) 32 points 1.09 / 1.22, 64 points 1.83 / 1.54; 240 modes 128
// points 0.20 / 0.21.  Float64, whose products cost more: 2000 modes (16 blocks)
// 4 points 1.36 / 1.43, 8 points 2.11 / 1.45; 240 modes 32 points 0.12 / 0.13,
// 64 points 0.18 / 0.13.
static bool solve_is_small(const BatchView& v, bool mixed) {
  return (int64_t)SOLVE_SPLIT * v.P * v.max_nt <= (mixed ? 8 : 2) * device_sms();
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
  if (solve_is_small(v, mixed)) return solve_small<true>(v, mixed, v.vec_y, out, s);
  if (!mixed) return bwd_impl<double2, double2>(v, out, s);
  return v.mean ? bwd_impl<float4, double2>(v, out, s) : bwd_impl<float4, float4>(v, out, s);
}

cudaError_t launch_solve_fwd(const BatchView& v, bool mixed, const double2* rhs, cudaStream_t s) {
  if (solve_is_small(v, mixed)) return solve_small<false>(v, mixed, rhs, v.vec_y, s);
  cudaError_t e = cudaSuccess;
  for (int k = -1; k + 1 < v.max_nt && e == cudaSuccess; ++k) e = launch_fwd_step(v, mixed, rhs, k, s, 0);
  return e;
}

cudaError_t launch_solve(const BatchView& v, bool mixed, const double2* rhs, double2* out, cudaStream_t s) {
  cudaError_t e = launch_solve_fwd(v, mixed, rhs, s);
  return e == cudaSuccess ? launch_bwd(v, mixed, out, s) : e;
}

int solve_launch_count(int max_nt) { return 2 * max_nt; }

}  // namespace beor
