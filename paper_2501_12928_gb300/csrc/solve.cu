// Triangular solves with the factor (both precisions).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>
#include <utility>

#include "diag_common.cuh"

namespace beor {

namespace cg = cooperative_groups;

// --------------------------------------------------------------------------
// Triangular solves with the factor: out = L^-H L^-1 rhs, blocked by 128.  Step k
// has two parts: its block of the solution, y_k = Linv_k r_k, and the update of
// the other blocks, r_i -= L_ik y_k (backward: with L_ki^H).
//   - Large batches launch one after the other: the block, then the update with a CTA
//     per tile. Small ones do both in one launch, a CTA per quarter tile, every four
//     forming y_k for themselves (cheaper than a launch that waits for one CTA).
//   - lnL: four CTAs of a cluster form y_k together, eight lanes per row, and exchange
//     it through distributed shared memory.  Its 33,000 float64 products take 8 us on
//     one SM (and 9 as chains of 128 pairs): with all of it in every CTA one point of
//     3280 modes took 7.57 ms and 64 points 46.1, now 6.63 and 45.3.  (In double-float,
//     which loses the last bits of r_k, 6.66 and 45.1.)  With more problems than SMs
//     float64's pipe bounds the blocks: 200 points of 240 modes 1.80 ms (1.69 in
//     double-float).  The float64 path and the posterior mean keep one chain per sum:
//     any other order changes the bits of the mean's amplitudes.
//   - Inverse block and quarter tile are copied to shared memory by cp.async, all
//     in flight at once, before the step waits for the one before (programmatic
//     dependent launch): the factor is final by then.
//   - Real and imaginary part of an update's sum go to two threads.
// Off-diagonal products: float64 for the float64 path, double-float (fp32 pairs,
// error-free sums) for the mixed path's double-float factor; the inverse blocks are
// applied in float64.  The order of each sum is fixed, so the results do not depend
// on the batch.
// Bound by memory in large batches, by the launch and by the chains of dependent
// products in small ones.  A step with one CTA per tile and 16 rounds of loads,
// the inverse block in one CTA at its end, took 35 us with one point of 3280
// modes and 71 with 64; now 7 and 70.  Float64, one point of 2000 modes: 38
// -> 30 us, whose chains of 128 dependent pairs of products alone are 9 us.
// --------------------------------------------------------------------------
constexpr int SOLVE_SPLIT = 4;                       // CTAs per tile
constexpr int SOLVE_ROWS = BEOR_TB / SOLVE_SPLIT;
constexpr int SOLVE_THREADS = 512;
template <typename V>   // V: the factor's real type, double or dfl
struct SolveVecs {
  double2 yk[BEOR_TB];
  double rd[2][BEOR_TB];               // r_k by component
  V yv[2][BEOR_TB];                    // y_k by component
  V part[2][SOLVE_ROWS];
};
// Who forms y_k = Linv_k r_k: a CTA alone, one chain per sum (the order of the
// float64 path and of the posterior mean), or SHARE CTAs, a quarter of the rows or
// all of them each, eight chains per sum (lnL).
constexpr int SOLVE_CHAIN = 0;
// A quarter's rows: four rows in turn give one to each quarter.  Row s of quarter c
// (backward: column, counted from the last); it has solve_row + 1 terms, stored from
// solve_row_off on.
constexpr int SOLVE_QUARTER = 2 * SOLVE_ROWS * (SOLVE_ROWS + 1);   // elements
__device__ __forceinline__ int solve_row(int c, int s) { return 4 * s + (s & 1 ? 3 - c : c); }
__device__ __forceinline__ int solve_row_off(int s) { return 2 * s * (s + 1); }
// shared memory: Linv_k, packed or by quarters; the quarter tile,
// forward [column][own row], backward [own column][row]; the vectors
constexpr size_t solve_li(int share) { return share == SOLVE_CHAIN ? DG_PACK : SOLVE_SPLIT / share * SOLVE_QUARTER; }
template <typename V>
constexpr size_t solve_smem(int share, bool both) {
  return sizeof(double2) * (solve_li(share) + (both ? BEOR_TB * SOLVE_ROWS : 0)) + sizeof(SolveVecs<V>);
}

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

// yk = Linv rk or (HERM) Linv^H rk, by 256 threads, one per row and component; the
// two warps of an SM quarter get rows of 160 terms together.
template <bool HERM>
__device__ __forceinline__ void solve_diag(const double2* li, const double (*rd)[BEOR_TB], double2* yk) {
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

// The same by SHARE CTAs, eight lanes per row, both components.  The warps of an SM
// quarter get rows of about the same number of terms together.  Row results go to
// every CTA of the cluster (SHARE 1: no cluster).
template <bool HERM, int SHARE>
__device__ __forceinline__ void solve_diag_shared(const double2* s_li, int rank, const double (*rd)[BEOR_TB], double2* yk) {
  constexpr int NQ = SOLVE_SPLIT / SHARE, NG = 8 * NQ;   // quarters of this CTA, groups of four rows by length
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lane8 = lane & 7;
  for (int w = warp; w < NG; w += SOLVE_THREADS / 32) {
    const int gl = w < NG / 2 ? NG - 1 - w : w - NG / 2, q = gl % NQ, c = SHARE == 1 ? q : rank;
    const int s = 4 * (gl / NQ) + (lane >> 3), n = solve_row(c, s), t = HERM ? BEOR_TB - 1 - n : n;
    const double2* li = s_li + q * SOLVE_QUARTER + solve_row_off(s);
    double a[2] = {0.0, 0.0};
#pragma unroll 2
    for (int m = lane8; m <= n; m += 8) {
      const int u = HERM ? t + m : m;
#pragma unroll
      for (int comp = 0; comp < 2; ++comp) mac_part(a[comp], li + m, HERM, comp, rd[comp][u], rd[1 - comp][u]);
    }
    __syncwarp();
    // the even lanes add up the real parts, the odd ones the imaginary
    const int comp = lane8 & 1;
    double sum = a[comp ? 1 : 0] + shfl_part(a[comp ? 0 : 1], 1);
    sum += shfl_part(sum, 2);
    sum += shfl_part(sum, 4);
    const int peer = lane8 >> 1;
    if (peer < SHARE) {
      double2* o = SHARE == 1 ? yk : cg::this_cluster().map_shared_rank(yk, peer);
      (comp ? o[t].y : o[t].x) = sum;
    }
  }
}

// Step k's block of y = L^-1 src or, HERM, of out = L^-H src; BOTH: and its update,
// by CTA (SOLVE_SPLIT (i - k - 1) + quarter, p) or, HERM, (SOLVE_SPLIT i + quarter,
// p), where problems join when k < their nt.  src: the right-hand side; the running
// one is vec_t.
template <typename WS, bool HERM, bool BOTH, int SHARE>
__global__ void __launch_bounds__(SOLVE_THREADS, 1)
    solve_step_kernel(BatchView v, int kg, const double2* src, double2* out) {
  using V = typename std::conditional<std::is_same<WS, float4>::value, dfl, double>::type;
  extern __shared__ __align__(16) unsigned char ss_raw[];
  double2* const s_li = reinterpret_cast<double2*>(ss_raw);
  double2* const s_tile = s_li + solve_li(SHARE);
  SolveVecs<V>& sm = *reinterpret_cast<SolveVecs<V>*>(s_tile + (BOTH ? BEOR_TB * SOLVE_ROWS : 0));
  const int tid = threadIdx.x, p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = HERM ? kg : kg - pr.k_off;   // this problem's step
  const int i = (HERM ? 0 : k + 1) + blockIdx.x / SOLVE_SPLIT, c0 = blockIdx.x % SOLVE_SPLIT * SOLVE_ROWS;
  const bool upd = BOTH && (HERM ? i < k : i < pr.nt);   // has a block to update
  const int ti = HERM ? k : i, tj = HERM ? i : k;
  // CTAs that share are on together, whatever becomes of the status meanwhile
  const bool skipped = prob_skipped(v.status[p]);
  bool on = k >= 0 && k < pr.nt && (upd || blockIdx.x < (SHARE > 1 ? SHARE : 1)) && (SHARE > 1 || !skipped);
  on = on && BEOR_INBOUNDS(v.flags, pr.row_off + (int64_t)pr.nt * BEOR_TB <= v.rows, BC_SOLVE_VEC) &&
       BEOR_INBOUNDS(v.flags, !upd || pr.ws_off + (tri_index(ti, tj) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_SOLVE_VEC) &&
       BEOR_INBOUNDS(v.flags, pr.dinv_off + (int64_t)(k + 1) * DG_PACK <= v.dinv_elems, BC_DIAG_DINV);
  if (on) {
    const double2* li = v.dinv + pr.dinv_off + (int64_t)k * DG_PACK;
    if constexpr (SHARE == SOLVE_CHAIN) {
      for (int e = tid; e < DG_PACK; e += SOLVE_THREADS) cp_async16(&s_li[e], li + e);
    } else {
      for (int w = tid >> 5; w < SOLVE_ROWS * SOLVE_SPLIT / SHARE; w += SOLVE_THREADS / 32) {
        const int s = w % SOLVE_ROWS, q = w / SOLVE_ROWS, n = solve_row(SHARE == 1 ? q : blockIdx.x % SHARE, s);
        for (int m = tid & 31; m <= n; m += 32)
          cp_async16(&s_li[q * SOLVE_QUARTER + solve_row_off(s) + m],
                     li + (HERM ? pk(BEOR_TB - 1 - n + m, BEOR_TB - 1 - n) : pk(n, m)));
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (upd) {
      const double2* t = reinterpret_cast<const double2*>(v.ws) + pr.ws_off + tri_index(ti, tj) * BEOR_TILE_ELEMS;
#pragma unroll
      for (int q = 0; q < BEOR_TB * SOLVE_ROWS / SOLVE_THREADS; ++q) {
        const int e = tid + q * SOLVE_THREADS;
        cp_async16(&s_tile[e], HERM ? t + c0 * BEOR_TB + e : t + e / SOLVE_ROWS * BEOR_TB + c0 + e % SOLVE_ROWS);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (SHARE > 1) cg::cluster_group::barrier_arrive();
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
  if (last) cur = reinterpret_cast<const double*>(r + i * BEOR_TB + c0 + own)[comp];
  if (tid < BEOR_TB) {
    const double2 q = r[k * BEOR_TB + tid];
    sm.rd[0][tid] = q.x;
    sm.rd[1][tid] = q.y;
  }
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();
  if constexpr (SHARE == SOLVE_CHAIN) {
    solve_diag<HERM>(s_li, sm.rd, sm.yk);
  } else {
    if (SHARE > 1) cg::cluster_group::barrier_wait();   // every CTA of the cluster has started
    solve_diag_shared<HERM, SHARE>(s_li, blockIdx.x % SHARE, sm.rd, sm.yk);
  }
  if (SHARE > 1)
    cg::this_cluster().sync();   // the last access to another CTA's memory is behind
  else
    __syncthreads();
  if (SHARE > 1 && skipped) return;
  if (tid < BEOR_TB) {
    const double2 q = sm.yk[tid];
    if (blockIdx.x == 0) out[pr.row_off + k * BEOR_TB + tid] = q;
    to_real(sm.yv[0][tid], q.x);
    to_real(sm.yv[1][tid], q.y);
  }
  if (!upd) return;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const WS* t = reinterpret_cast<const WS*>(s_tile);
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

// The update of step k alone, a CTA per tile: the tile streams through registers,
// 16 elements in flight per thread (held in shared memory, a tile's quarters wait
// for their last element and then for the chains: 117 us for 25 tiles of each of
// 64 points; 85 here, 62 at the copy rate).  y: vec_y or, HERM, the solution.
template <typename WS, bool HERM>
__global__ void __launch_bounds__(256, 2)
    solve_update_kernel(BatchView v, int kg, const double2* src, const double2* y) {
  using V = typename std::conditional<std::is_same<WS, float4>::value, dfl, double>::type;
  __shared__ V yv[2][BEOR_TB], part[2][BEOR_TB];
  const int tid = threadIdx.x, p = blockIdx.y;
  const Prob pr = v.prob[p];
  const int k = HERM ? kg : kg - pr.k_off;   // this problem's step
  const int i = (HERM ? 0 : k + 1) + blockIdx.x, ti = HERM ? k : i, tj = HERM ? i : k;
  const bool on = k >= 0 && k < pr.nt && (HERM ? i < k : i < pr.nt) && !prob_skipped(v.status[p]) &&
                  BEOR_INBOUNDS(v.flags, pr.row_off + (int64_t)pr.nt * BEOR_TB <= v.rows, BC_SOLVE_VEC) &&
                  BEOR_INBOUNDS(v.flags, pr.ws_off + (tri_index(ti, tj) + 1) * BEOR_TILE_ELEMS <= v.ws_elems, BC_SOLVE_VEC);
  // forward: row and half of the columns; backward: eight lanes per column,
  // interleaved rows, four columns per warp in turn
  const int row = tid & 127, half = tid >> 7;
  const int col = (tid >> 5) * 16 + ((tid >> 3) & 3), mo = tid & 7;
  const WS* __restrict__ t = reinterpret_cast<const WS*>(v.ws) + pr.ws_off + (on ? tri_index(ti, tj) : 0) * BEOR_TILE_ELEMS +
                             (HERM ? col * BEOR_TB + mo : half * 64 * BEOR_TB + row);
  WS a[8], b[8];
  auto load = [&](WS* o, int c) {   // chunk c of eight elements
#pragma unroll
    for (int q = 0; q < 8; ++q) o[q] = __ldcs(t + (HERM ? (c >> 1) * 4 * BEOR_TB + 8 * ((c & 1) * 8 + q) : (8 * c + q) * BEOR_TB));
  };
  if (on) load(a, 0);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (!on) return;
  const double2* r = (k == (HERM ? pr.nt - 1 : 0) ? src : v.vec_t) + pr.row_off + i * BEOR_TB;
  double2* const out = v.vec_t + pr.row_off + i * BEOR_TB;
  if (tid < BEOR_TB) {
    const double2 q = y[pr.row_off + k * BEOR_TB + tid];
    to_real(yv[0][tid], q.x);
    to_real(yv[1][tid], q.y);
  }
  __syncthreads();
  V acc[2] = {};
  auto mac = [&](const WS* l, int c) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int m = HERM ? mo + 8 * ((c & 1) * 8 + q) : half * 64 + 8 * c + q;
#pragma unroll
      for (int comp = 0; comp < 2; ++comp) mac_part(acc[comp], l + q, HERM, comp, yv[comp][m], yv[1 - comp][m]);
    }
  };
#pragma unroll 1
  for (int c = 0; c < 8; c += 2) {
    load(b, c + 1);
    mac(a, c);
    if (c + 2 < 8) load(a, c + 2);
    mac(b, c + 1);
    if (HERM) {
#pragma unroll
      for (int comp = 0; comp < 2; ++comp)
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) add_part(acc[comp], shfl_part(acc[comp], o));
      if (mo == 0) {
        const int cc = col + 2 * c;
        const double2 cur = r[cc];
        out[cc] = make_double2(cur.x - get_part(acc[0]), cur.y - get_part(acc[1]));
      }
      acc[0] = acc[1] = V{};
    }
  }
  if (!HERM) {
    if (half) {
      part[0][row] = acc[0];
      part[1][row] = acc[1];
    }
    __syncthreads();
    if (!half) {
      const double2 cur = r[row];
      add_part(acc[0], part[0][row]);
      add_part(acc[1], part[1][row]);
      out[row] = make_double2(cur.x - get_part(acc[0]), cur.y - get_part(acc[1]));
    }
  }
}

// after: the launch before on the stream is the step before (its results, not the
// factor, are what is waited for)
template <typename... Exp, typename... Act>
static cudaError_t launch_after(void (*kern)(Exp...), dim3 grid, int threads, size_t smem, cudaStream_t s, bool after,
                                int cluster, Act&&... args) {
  cudaLaunchAttribute at[2];
  int n = 0;
  if (after) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = cluster;
    at[n].val.clusterDim.y = 1;
    at[n++].val.clusterDim.z = 1;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Act>(args)...);
}
template <typename WS, bool HERM, bool BOTH, int SHARE>
static cudaError_t launch_block(const BatchView& v, int k, int blocks, const double2* src, double2* out, cudaStream_t s,
                                bool after) {
  using V = typename std::conditional<std::is_same<WS, float4>::value, dfl, double>::type;
  static_assert(SHARE <= 1 || SHARE == SOLVE_SPLIT, "a cluster is the CTAs of one tile");
  constexpr int ctas = SHARE > 1 ? SHARE : 1;
  constexpr size_t need = solve_smem<V>(SHARE, BOTH), most = 120 * 1024;
  // Float64's pipe bounds the block alone: its CTAs, which start beside the update
  // before them, must not gather on the SMs that are free first.  Where n of them
  // belong on an SM, each takes more than 1 / (n + 1) of its 227 KB: 11.5 -> 5 us a
  // step after the update's end with 16 points of 3280 modes, 15 -> 8 with 64.
  const int64_t n = ((int64_t)ctas * v.P + device_sms() - 1) / device_sms();
  const size_t smem = SHARE <= 1 || BOTH ? need : std::max(need, 2 * most / (size_t)(n + 1));
  const cudaError_t attr = allow_smem<solve_step_kernel<WS, HERM, BOTH, SHARE>>((int)(SHARE <= 1 || BOTH ? need : most));
  if (attr != cudaSuccess) return attr;
  return launch_after(solve_step_kernel<WS, HERM, BOTH, SHARE>, dim3(BOTH ? std::max(ctas, SOLVE_SPLIT * blocks) : ctas, v.P),
                      SOLVE_THREADS, smem, s, after, ctas, v, k, src, out);
}
// The products with the inverse block beside every tile pay while the first step's
// CTAs fit the SMs once.  Solves of one evaluation in ms (one launch per step / two):
// mixed, 3280 modes (26 blocks) one point 0.89 / 0.96, two 1.06 / 1.02; 1000 modes
// (8 blocks) four points 0.28 / 0.30, eight 0.35 / 0.32.  Float64, 2000 modes (16
// blocks) two points 0.95 / 0.96, four 1.33 / 1.04.
static bool solve_is_small(const BatchView& v) { return (int64_t)SOLVE_SPLIT * v.P * v.max_nt <= device_sms(); }
// Step k of one pass.
template <bool HERM, typename WS, int SHARE>
static cudaError_t step_as(const BatchView& v, bool both, int k, const double2* src, double2* out, cudaStream_t s, bool after) {
  const int blocks = HERM ? k : v.max_nt - 1 - k;   // to update
  if (both) return launch_block<WS, HERM, true, SHARE>(v, k, blocks, src, out, s, after);
  const cudaError_t e = launch_block<WS, HERM, false, SHARE>(v, k, blocks, src, out, s, after);
  if (e != cudaSuccess || blocks == 0) return e;
  return launch_after(solve_update_kernel<WS, HERM>, dim3(blocks, v.P), 256, 0, s, true, 1, v, k, src, (const double2*)out);
}
template <bool HERM>
static cudaError_t solve_step(const BatchView& v, bool mixed, bool both, int k, const double2* src, double2* out,
                              cudaStream_t s, bool after) {
  return !mixed   ? step_as<HERM, double2, SOLVE_CHAIN>(v, both, k, src, out, s, after)
         : v.mean ? step_as<HERM, float4, SOLVE_CHAIN>(v, both, k, src, out, s, after)
                  : step_as<HERM, float4, SOLVE_SPLIT>(v, both, k, src, out, s, after);
}

// Step k (0 .. max_nt - 1) of vec_y = L^-1 rhs, beside other work: the parts one
// after the other, which take less of an SM than both in one, and no clusters but in
// the last two steps, which nothing else runs beside (16 -> 9 us each).
cudaError_t launch_fwd_step(const BatchView& v, bool mixed, const double2* rhs, int k, cudaStream_t s) {
  if (mixed && !v.mean && k + 2 < v.max_nt) return step_as<false, float4, 1>(v, false, k, rhs, v.vec_y, s, false);
  return solve_step<false>(v, mixed, false, k, rhs, v.vec_y, s, false);
}
int fwd_step_launches(const BatchView& v, int k) { return k + 1 < v.max_nt ? 2 : 1; }

// vec_y = L^-1 rhs and out = L^-H vec_y, every problem.
cudaError_t launch_solve_fwd(const BatchView& v, bool mixed, const double2* rhs, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < v.max_nt && e == cudaSuccess; ++k)
    e = solve_step<false>(v, mixed, solve_is_small(v), k, rhs, v.vec_y, s, k > 0);
  return e;
}
cudaError_t launch_bwd(const BatchView& v, bool mixed, double2* out, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int k = v.max_nt - 1; k >= 0 && e == cudaSuccess; --k)
    e = solve_step<true>(v, mixed, solve_is_small(v), k, v.vec_y, out, s, k + 1 < v.max_nt);
  return e;
}
cudaError_t launch_solve(const BatchView& v, bool mixed, const double2* rhs, double2* out, cudaStream_t s) {
  cudaError_t e = launch_solve_fwd(v, mixed, rhs, s);
  return e == cudaSuccess ? launch_bwd(v, mixed, out, s) : e;
}
int solve_pass_launches(const BatchView& v) { return solve_is_small(v) ? v.max_nt : 2 * v.max_nt - 1; }

}  // namespace beor
