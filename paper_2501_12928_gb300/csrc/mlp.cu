// Learned emulator of lnL(phi): a multilayer perceptron n_in -> depth x width
// (GELU) -> 1, trained and evaluated by the library's own kernels.
//
// Numbers: bf16 weights and activations feed the tensor cores
// (mma.sync m16n8k16, fp32 accumulation); pre-activations, gradients of the
// loss, master weights and the Adam moments are fp32.  The emulator only
// pre-screens candidate prior points for the nested sampler; every accepted
// point is evaluated exactly.
//
// Two kernels per training step, one per inference:
//  * rows_kernel: a CTA takes 16 to 64 rows through the whole network (and, in
//    training, the loss and the chain of data gradients back to the first
//    hidden layer), activations in shared memory, weights streamed through it;
//  * grad_kernel: the weight and bias gradients of every layer, each tile's
//    Adam update in its epilogue.
// What bounds them: the network is small (1.2 MFLOP per row and training step),
// so a step of 1024 rows is a chain of latencies: 23 launches of 3 to 73 us
// (weight gradients on 16 CTAs with element-wise loads) took 660 us; two
// launches of 64 and 141 CTAs take 33 + 13 us.  Every sum keeps its order (K
// ascending in steps of 16, column sums by 256 strided partial sums), so the
// results are those of the layer-by-layer kernels bit for bit, the loss's sum
// over rows apart.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/beor.h"
#include "beor_internal.h"

namespace {

constexpr int kMaxLayers = 9;
constexpr int kMaxW = 256;
constexpr int kThreads = 256;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

struct Net {
  int L, n, n_in;                        // layers, rows, inputs
  int kin[kMaxLayers], kout[kMaxLayers]; // padded sizes
  int fin[kMaxLayers], fout[kMaxLayers]; // logical sizes
  __nv_bfloat16* Wb[kMaxLayers];         // kout x kin
  float* b[kMaxLayers];
  const float* x;                        // n x n_in
  const float *x_shift, *x_scale;
  float y_shift, y_scale;
  float* y;                              // inference: n predictions
  // training
  const float* t;                        // targets
  __nv_bfloat16* H[kMaxLayers];          // inputs of layer l, n x kin
  float* dZ[kMaxLayers];                 // gradients of layer l's pre-activation, n x kout (last layer: n)
  __nv_bfloat16* dZb[kMaxLayers];        // the same in bf16, n x kout
  float* loss_part;                      // per CTA of rows_kernel
  float* loss;
  int nparts;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes global -> shared, zeros when !ok
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

constexpr int kKC = 64;                    // K rows of weights per stage
constexpr int kActLd = kMaxW + 8;          // activations [row][kActLd]
constexpr int kWLd = kKC + 8;              // forward stage [n][kWLd]
constexpr int kWtLd = kMaxW + 8;           // backward stage [k][kWtLd]
constexpr int kStage = kMaxW * kWLd;       // bf16 elements per stage (36,864 bytes)
template <int MT, int ST, bool TRAIN>
constexpr int rows_smem(int depth) {
  return (MT * 16 * kActLd + ST * kStage) * 2 + (TRAIN ? depth * MT * 16 * kMaxW * 4 : 0);
}

// Rows [16 MT blockIdx.x, ..) through the network.  Eight warps, 32 output
// columns each; the weights come in chunks of 64 K rows through a ring of ST
// stages, ST - 1 chunks ahead.  MT = 1 where the rows are few (the chain of
// layers is latency), MT = 4 with two CTAs per SM, one's GELUs beside the
// other's products, where every SM has rows enough: each CTA reads all the
// weights (0.5 MB) from L2.  64 rows through 256 x 4: 15 us (five layers'
// launches of 14 us before), 20,000 rows: 66 us (219 us), of which the products
// take 35 at the rate of mma.sync and the rest is GELU and the rows beyond a
// whole wave.  (Sixteen warps of 16 columns: the same times.)
template <int MT, int ST, bool TRAIN>
__global__ void __launch_bounds__(kThreads) rows_kernel(const __grid_constant__ Net g) {
  extern __shared__ __align__(16) __nv_bfloat16 sm_rows[];
  __nv_bfloat16* act = sm_rows;
  __nv_bfloat16* ring = act + MT * 16 * kActLd;
  float* Z = reinterpret_cast<float*>(ring + ST * kStage);   // TRAIN: [hidden layer][row][kMaxW]
  __shared__ float s_dz[MT * 16], s_red[kThreads / 32];
  constexpr int R = MT * 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int width = g.kout[0];
  // the next chunk of the sequence: forward layers 0 .. L-1, then (training)
  // backward layers L-1 .. 1, into the next stage of the ring
  int ll = 0, lk = 0, lst = 0;
  bool lback = false;
  auto load = [&]() {
    __nv_bfloat16* st = ring + lst * kStage;
    lst = lst + 1 == ST ? 0 : lst + 1;
    if (ll < 0) return;   // every chunk is on its way
    const int K = lback ? g.kout[ll] : g.kin[ll], N = lback ? g.kin[ll] : g.kout[ll];
    const __nv_bfloat16* W = g.Wb[ll];
    if (!lback) {         // [n][64 k]: eight 16-byte pieces per row
      const int q = (tid & 7) * 8;
      if (lk + q < K)
        for (int n = tid >> 3; n < N; n += kThreads / 8)
          cp16(smem_addr(st + n * kWLd + q), W + (int64_t)n * K + lk + q, true);
    } else {              // [64 k][n]: a warp per row
      if (lane * 8 < N)
        for (int k = warp; k < min(kKC, K - lk); k += kThreads / 32)
          cp16(smem_addr(st + k * kWtLd + lane * 8), W + (int64_t)(lk + k) * N + lane * 8, true);
    }
    lk += kKC;
    if (lk < K) return;
    lk = 0;
    if (lback)
      ll = ll > 1 ? ll - 1 : -1;
    else if (ll + 1 < g.L)
      ++ll;
    else if (TRAIN)
      lback = true;
    else
      ll = -1;
  };
  const int m0 = blockIdx.x * R;
  for (int c = 0; c < ST - 1; ++c) {
    load();
    cp_commit();
  }
  // normalised, zero-padded bf16 inputs
  const int ld0 = g.kin[0];
  for (int e = tid; e < R * ld0; e += kThreads) {
    const int m = e / ld0, i = e % ld0;
    const float v = i < g.n_in && m0 + m < g.n ? (g.x[(int64_t)(m0 + m) * g.n_in + i] - g.x_shift[i]) * g.x_scale[i] : 0.0f;
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    act[m * kActLd + i] = h;
    if (TRAIN && m0 + m < g.n) g.H[0][(int64_t)(m0 + m) * ld0 + i] = h;
  }
  float acc[MT][4][4];
  int cst = 0;   // ring stage of the next chunk to multiply
  // acc = act x the layer's weights; returns with every warp past its last read of act
  auto layer = [&](int K, int ntile, bool back) {
#pragma unroll
    for (int a = 0; a < MT; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[a][b][q] = 0.0f;
    for (int k0 = 0; k0 < K; k0 += kKC) {
      cp_wait<ST - 2>();
      __syncthreads();   // this chunk (and, at k0 = 0, the layer's input) is in shared memory, the last one is read
      load();
      cp_commit();
      const __nv_bfloat16* st = ring + cst * kStage;
      cst = cst + 1 == ST ? 0 : cst + 1;
      if (ntile > 0)
        for (int kk = 0; kk < min(kKC, K - k0); kk += 16) {
          uint32_t a[MT][4], b[2][4];
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)
            ldm4(a[mt], smem_addr(act + (mt * 16 + (lane & 15)) * kActLd + k0 + kk + (lane >> 4) * 8));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int n = warp * 32 + h * 16;
            if (back)
              ldm4t(b[h], smem_addr(st + (kk + (lane & 15)) * kWtLd + min(n, kMaxW - 16) + (lane >> 4) * 8));
            else
              ldm4(b[h], smem_addr(st + (n + (lane & 7) + (lane >> 4) * 8) * kWLd + kk + ((lane >> 3) & 1) * 8));
          }
#pragma unroll
          for (int nt = 0; nt < 4; ++nt)
            if (nt < ntile)
#pragma unroll
              for (int mt = 0; mt < MT; ++mt)
                mma16(acc[mt][nt], a[mt], b[nt >> 1][(nt & 1) * 2], b[nt >> 1][(nt & 1) * 2 + 1]);
        }
    }
    __syncthreads();   // every warp is past its last read of act
  };
  const int gq = lane >> 2, tq = lane & 3;
  const int ntile = max(0, min(4, (width - warp * 32) / 8));
  for (int l = 0; l + 1 < g.L; ++l) {
    float2 bias[4];   // loaded ahead of the products
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
      if (nt < ntile) bias[nt] = *reinterpret_cast<const float2*>(g.b[l] + warp * 32 + nt * 8 + 2 * tq);
    layer(g.kin[l], ntile, false);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
        if (nt < ntile)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int r = mt * 16 + gq + 8 * h, n = warp * 32 + nt * 8 + 2 * tq;
            const float z0 = acc[mt][nt][2 * h] + bias[nt].x, z1 = acc[mt][nt][2 * h + 1] + bias[nt].y;
            const __nv_bfloat162 v = __floats2bfloat162_rn(gelu(z0), gelu(z1));
            *reinterpret_cast<__nv_bfloat162*>(act + r * kActLd + n) = v;
            if (TRAIN) {
              *reinterpret_cast<float2*>(Z + (l * R + r) * kMaxW + n) = make_float2(z0, z1);
              if (m0 + r < g.n) *reinterpret_cast<__nv_bfloat162*>(g.H[l + 1] + (int64_t)(m0 + r) * width + n) = v;
            }
          }
  }
  const int lo = g.L - 1;
  layer(g.kin[lo], warp == 0 ? 1 : 0, false);
  if (warp == 0 && tq == 0)
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = mt * 16 + gq + 8 * h;
        const float y = acc[mt][0][2 * h] + g.b[lo][0];
        if (!TRAIN) {
          if (m0 + r < g.n) g.y[m0 + r] = y * g.y_scale + g.y_shift;   // the network's output units to lnL units
        } else {
          s_dz[r] = y;
        }
      }
  if constexpr (TRAIN) {
    // loss = mean (y - t)^2 in normalised units; seed gradient dZ_out = 2 (y - t) / n
    __syncthreads();
    float part = 0.0f;
    for (int r = tid; r < R; r += kThreads) {
      float gdz = 0.0f;
      if (m0 + r < g.n) {
        const float target = (g.t[m0 + r] - g.y_shift) / g.y_scale;
        const float d = s_dz[r] - target;
        part += d * d;
        gdz = 2.0f * d / (float)g.n;
        g.dZ[lo][m0 + r] = gdz;
      }
      for (int i = 0; i < 16; ++i) {
        const __nv_bfloat16 v = __float2bfloat16_rn(i == 0 ? gdz : 0.0f);
        act[r * kActLd + i] = v;
        if (m0 + r < g.n) g.dZb[lo][(int64_t)(m0 + r) * 16 + i] = v;
      }
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) s_red[warp] = part;
    __syncthreads();
    if (tid == 0) {
      float s = 0.0f;
      for (int w = 0; w < kThreads / 32; ++w) s += s_red[w];
      g.loss_part[blockIdx.x] = s;
    }
    // dZ_{l-1} = (dZ_l W_l) * gelu'(Z_{l-1})
    for (int l = lo; l > 0; --l) {
      layer(g.kout[l], ntile, true);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
          if (nt < ntile)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int r = mt * 16 + gq + 8 * h, n = warp * 32 + nt * 8 + 2 * tq;
              const float2 z = *reinterpret_cast<const float2*>(Z + ((l - 1) * R + r) * kMaxW + n);
              const float d0 = acc[mt][nt][2 * h] * gelu_grad(z.x), d1 = acc[mt][nt][2 * h + 1] * gelu_grad(z.y);
              const __nv_bfloat162 v = __floats2bfloat162_rn(d0, d1);
              *reinterpret_cast<__nv_bfloat162*>(act + r * kActLd + n) = v;
              if (m0 + r < g.n) {
                *reinterpret_cast<float2*>(g.dZ[l - 1] + (int64_t)(m0 + r) * width + n) = make_float2(d0, d1);
                *reinterpret_cast<__nv_bfloat162*>(g.dZb[l - 1] + (int64_t)(m0 + r) * width + n) = v;
              }
            }
    }
  }
}

// Adam on one parameter (beta1, beta2, eps; c1 = 1 - beta1^t, c2 = 1 - beta2^t)
struct Adam {
  float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ float adam(const Adam& a, float gr, float* pp, float* mp, float* vp) {
  const float m = a.b1 * *mp + (1.0f - a.b1) * gr;
  const float v = a.b2 * *vp + (1.0f - a.b2) * gr * gr;
  *mp = m;
  *vp = v;
  const float p = *pp - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
  *pp = p;
  return p;
}

struct Params {
  float *W[kMaxLayers], *mW[kMaxLayers], *vW[kMaxLayers], *gW[kMaxLayers];
  float *b[kMaxLayers], *mb[kMaxLayers], *vb[kMaxLayers], *gb[kMaxLayers];
  int first[kMaxLayers + 1];   // first CTA of layer l's weight tiles; then of its bias columns
  int bfirst[kMaxLayers + 1];
  Adam adam;
  int update;                  // 1: Adam, 0: write the gradients
};

constexpr int kGO = 32, kGI = 64, kGS = 3;              // weight-gradient tile (out x in), stages
constexpr int kGALd = kGO + 8, kGBLd = kGI + 8;
constexpr int kGStage = kKC * (kGALd + kGBLd);          // bf16 elements per stage

// Gradients of every layer: gW[o][i] = sum_m dZ[m][o] H[m][i] (a 32 x 64 tile
// per CTA, the rows in order), gb[o] = sum_m dZ[m][o] (32 columns per CTA).
__global__ void __launch_bounds__(kThreads) grad_kernel(const __grid_constant__ Net g, const __grid_constant__ Params q) {
  __shared__ __align__(16) __nv_bfloat16 st[kGS * kGStage];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if ((int)blockIdx.x < q.first[g.L]) {
    int l = 0;
    while ((int)blockIdx.x >= q.first[l + 1]) ++l;
    const int ni = (g.fin[l] + kGI - 1) / kGI, t = blockIdx.x - q.first[l];
    const int o0 = t / ni * kGO, i0 = t % ni * kGI;
    const int lda = g.kout[l], ldb = g.kin[l];
    const __nv_bfloat16 *A = g.dZb[l], *B = g.H[l];
    const int nk = (g.n + kKC - 1) / kKC;
    auto load = [&](int kc) {
      __nv_bfloat16* s = st + kc % kGS * kGStage;
      static_assert(kThreads == 256 && kKC == 64 && kGO == 32 && kGI == 64, "pieces of 16 bytes per thread");
      {   // 64 rows x 32 columns of dZ: one piece per thread
        const int k = tid >> 2, col = (tid & 3) * 8, m = kc * kKC + k;
        const bool ok = m < g.n && o0 + col < lda;
        cp16(smem_addr(s + k * kGALd + col), ok ? A + (int64_t)m * lda + o0 + col : A, ok);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // 64 rows x 64 columns of H: two
        const int k = (tid >> 3) + 32 * h, col = (tid & 7) * 8, m = kc * kKC + k;
        const bool ok = m < g.n && i0 + col < ldb;
        cp16(smem_addr(s + kKC * kGALd + k * kGBLd + col), ok ? B + (int64_t)m * ldb + i0 + col : B, ok);
      }
    };
    float acc[2][4] = {};
    for (int kc = 0; kc < kGS - 1; ++kc) {
      if (kc < nk) load(kc);
      cp_commit();
    }
    const int wo = (warp & 1) * 16, wi = (warp >> 1) * 16;
    for (int kc = 0; kc < nk; ++kc) {
      cp_wait<kGS - 2>();
      __syncthreads();   // chunk kc has landed; every warp is done with chunk kc - 1
      if (kc + kGS - 1 < nk) load(kc + kGS - 1);
      cp_commit();
      const __nv_bfloat16* s = st + kc % kGS * kGStage;
#pragma unroll
      for (int kk = 0; kk < kKC; kk += 16) {
        uint32_t a[4], b[4];
        ldm4t(a, smem_addr(s + (kk + (lane & 7) + (lane >> 4) * 8) * kGALd + wo + ((lane >> 3) & 1) * 8));
        ldm4t(b, smem_addr(s + kKC * kGALd + (kk + (lane & 15)) * kGBLd + wi + (lane >> 4) * 8));
        mma16(acc[0], a, b[0], b[1]);
        mma16(acc[1], a, b[2], b[3]);
      }
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int o = o0 + wo + (lane >> 2) + (c & 2 ? 8 : 0), i = i0 + wi + nt * 8 + 2 * (lane & 3) + (c & 1);
        if (o >= g.fout[l] || i >= g.fin[l]) continue;
        const int64_t e = (int64_t)o * g.fin[l] + i;
        if (q.update) {
          const float p = adam(q.adam, acc[nt][c], q.W[l] + e, q.mW[l] + e, q.vW[l] + e);
          g.Wb[l][(int64_t)o * ldb + i] = __float2bfloat16_rn(p);
        } else {
          q.gW[l][e] = acc[nt][c];
        }
      }
    return;
  }
  int l = 0;
  while ((int)blockIdx.x >= q.bfirst[l + 1]) ++l;
  // column o: 256 partial sums over rows t, t + 256, ..; the 32 of a warp added
  // up by halving, then the eight warps' in order.  Thread (column, warp).
  float* red = reinterpret_cast<float*>(st);
  const int o = (blockIdx.x - q.bfirst[l]) * 32 + lane, w = warp;
  const int ld = l == g.L - 1 ? 1 : g.kout[l];
  float a[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) a[t] = 0.0f;
  const float* col = g.dZ[l] + min(o, g.fout[l] - 1);
  for (int m0 = 32 * w; m0 < g.n; m0 += kThreads) {   // 32 loads in flight
    float d[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) d[t] = col[(int64_t)min(m0 + t, g.n - 1) * ld];
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if (m0 + t < g.n) a[t] += d[t];
  }
#pragma unroll
  for (int h = 16; h > 0; h >>= 1)
#pragma unroll
    for (int t = 0; t < 32; ++t)
      if (t < h) a[t] += a[t + h];
  red[w * 32 + lane] = a[0];
  __syncthreads();
  if (w == 0 && o < g.fout[l]) {
    float s = 0.0f;
    for (int v = 0; v < kThreads / 32; ++v) s += red[v * 32 + lane];
    if (q.update)
      adam(q.adam, s, q.b[l] + o, q.mb[l] + o, q.vb[l] + o);
    else
      q.gb[l][o] = s;
  }
  if (l == g.L - 1 && w == 1) {   // the loss
    float s = 0.0f;
    for (int i = lane; i < g.nparts; i += 32) s += g.loss_part[i];
    for (int h = 16; h > 0; h >>= 1) s += __shfl_xor_sync(0xffffffffu, s, h);
    if (lane == 0) *g.loss = s / (float)g.n;
  }
}

// He-uniform initial weights from a counter-based generator (SplitMix64 of
// seed, layer and index): W ~ U(-sqrt(6 / fan_in), sqrt(6 / fan_in)).
__global__ void init_kernel(float* W, int64_t n, int fan_in, uint64_t seed, int layer) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(i + 1) + ((uint64_t)layer << 48);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);   // [0, 1)
    const double lim = sqrt(6.0 / (double)fan_in);
    W[i] = (float)((2.0 * u - 1.0) * lim);
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ W, int rows, int cols, int ldb, __nv_bfloat16* __restrict__ Wb) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)rows * cols) return;
  const int r = (int)(e / cols), c = (int)(e % cols);
  Wb[(int64_t)r * ldb + c] = __float2bfloat16_rn(W[e]);
}

// Where a caller's array lies: host memory, device memory, or device memory that
// the kernels of `device` may address as it stands (that device's own, on a float
// boundary; anything else a copy reaches, and only a copy).
enum Where { HOST, DEVICE, HERE };
Where where_is(const void* p, int device) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return HOST;
  }
  if (a.type == cudaMemoryTypeDevice && a.device == device && reinterpret_cast<uintptr_t>(p) % alignof(float) == 0) return HERE;
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged ? DEVICE : HOST;
}
bool on_device(const void* p) { return where_is(p, -1) != HOST; }

int pad16(int x) { return (x + 15) / 16 * 16; }

}  // namespace

struct beor_mlp {
  int device = 0, n_in = 0, width = 0, depth = 0, L = 0;
  int fin[kMaxLayers], fout[kMaxLayers];      // logical sizes
  int kin[kMaxLayers], kout[kMaxLayers];      // padded sizes (bf16 copies, activations)
  float *W[kMaxLayers] = {}, *b[kMaxLayers] = {}, *gW[kMaxLayers] = {}, *gb[kMaxLayers] = {};
  float *mW[kMaxLayers] = {}, *vW[kMaxLayers] = {}, *mb[kMaxLayers] = {}, *vb[kMaxLayers] = {};
  __nv_bfloat16* Wb[kMaxLayers] = {};
  float *x_shift = nullptr, *x_scale = nullptr;
  float y_shift = 0.0f, y_scale = 1.0f;
  int64_t step = 0;
  // batch workspace (training)
  int cap = 0;
  __nv_bfloat16* H[kMaxLayers] = {};          // inputs of layer l (H[0] = normalised input)
  float* dZ[kMaxLayers] = {};                 // gradients of the pre-activations
  __nv_bfloat16* dZb[kMaxLayers] = {};
  float *loss_part = nullptr, *loss = nullptr;
  // host inputs and outputs
  int iocap = 0;
  float *xin = nullptr, *tin = nullptr, *yout = nullptr;
  std::vector<void*> owned;
};

namespace {

cudaError_t dalloc(beor_mlp* m, void** p, size_t bytes) {
  cudaError_t e = beor::device_malloc(p, bytes);
  if (e == cudaSuccess) {
    m->owned.push_back(*p);
    cudaMemset(*p, 0, bytes);
  }
  return e;
}

void release(beor_mlp* m, void* p) {
  if (!p) return;
  for (auto& q : m->owned)
    if (q == p) q = nullptr;
  cudaFree(p);
}

// device copies of host inputs and outputs for n rows
cudaError_t ensure_io(beor_mlp* m, int n) {
  if (n <= m->iocap) return cudaSuccess;
  m->iocap = 0;
  release(m, m->xin);
  release(m, m->tin);
  release(m, m->yout);
  m->xin = m->tin = m->yout = nullptr;
  int cap = 1024;
  while (cap < n) cap *= 2;
  cudaError_t e = dalloc(m, (void**)&m->xin, sizeof(float) * (size_t)cap * m->n_in);
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->tin, sizeof(float) * (size_t)cap);
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->yout, sizeof(float) * (size_t)cap);
  if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);   // the fills, before another stream's work
  if (e == cudaSuccess) m->iocap = cap;
  return e;
}

cudaError_t ensure_cap(beor_mlp* m, int n) {
  cudaError_t e = ensure_io(m, n);
  if (e != cudaSuccess || n <= m->cap) return e;
  // release the old batch workspace
  m->cap = 0;
  for (int l = 0; l < m->L; ++l) {
    release(m, m->H[l]);
    release(m, m->dZ[l]);
    release(m, m->dZb[l]);
    m->H[l] = m->dZb[l] = nullptr;
    m->dZ[l] = nullptr;
  }
  release(m, m->loss_part);
  m->loss_part = nullptr;
  int cap = 1024;
  while (cap < n) cap *= 2;
  for (int l = 0; l < m->L && e == cudaSuccess; ++l) {
    e = dalloc(m, (void**)&m->H[l], sizeof(__nv_bfloat16) * (size_t)cap * m->kin[l]);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->dZ[l], sizeof(float) * (size_t)cap * (l == m->L - 1 ? 1 : m->kout[l]));
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->dZb[l], sizeof(__nv_bfloat16) * (size_t)cap * m->kout[l]);
  }
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->loss_part, sizeof(float) * (size_t)(cap / 16));
  if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
  if (e == cudaSuccess) m->cap = cap;
  return e;
}

cudaError_t copy_in(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  return cudaMemcpyAsync(dst, src, bytes, on_device(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s);
}

Net net_of(const beor_mlp* m, const float* x, int n) {
  Net g{};
  g.L = m->L;
  g.n = n;
  g.n_in = m->n_in;
  for (int l = 0; l < m->L; ++l) {
    g.kin[l] = m->kin[l];
    g.kout[l] = m->kout[l];
    g.fin[l] = m->fin[l];
    g.fout[l] = m->fout[l];
    g.Wb[l] = m->Wb[l];
    g.b[l] = m->b[l];
    g.H[l] = m->H[l];
    g.dZ[l] = m->dZ[l];
    g.dZb[l] = m->dZb[l];
  }
  g.x = x;
  g.x_shift = m->x_shift;
  g.x_scale = m->x_scale;
  g.y_shift = m->y_shift;
  g.y_scale = m->y_scale;
  g.loss_part = m->loss_part;
  g.loss = m->loss;
  return g;
}

template <int MT, int ST, bool TRAIN>
cudaError_t launch_rows(const Net& g, cudaStream_t s) {
  constexpr int deepest = TRAIN && ST > 2 ? 4 : kMaxLayers - 1;
  const cudaError_t attr = beor::allow_smem<rows_kernel<MT, ST, TRAIN>>(rows_smem<MT, ST, TRAIN>(deepest));
  if (attr != cudaSuccess) return attr;
  rows_kernel<MT, ST, TRAIN><<<(g.n + 16 * MT - 1) / (16 * MT), kThreads, rows_smem<MT, ST, TRAIN>(g.L - 1), s>>>(g);
  return cudaGetLastError();
}

// predictions of n rows (device x and y)
cudaError_t predict(beor_mlp* m, const float* x, int n, float* y, cudaStream_t s) {
  Net g = net_of(m, x, n);
  g.y = y;
  if (n <= 16 * 2 * beor::device_sms()) return launch_rows<1, 5, false>(g, s);
  // whole waves of 64 rows and two CTAs per SM (50 us); a short rest goes 16 rows
  // to a CTA, 16 us on idle SMs, where the start of another wave takes 21: 20,000
  // rows 66 us, 71 in one launch
  const int wave = 64 * 2 * beor::device_sms(), rest = n % wave;
  if (rest == 0 || rest > 16 * beor::device_sms() || n < wave) return launch_rows<4, 2, false>(g, s);
  g.n = n - rest;
  const cudaError_t e = launch_rows<4, 2, false>(g, s);
  if (e != cudaSuccess) return e;
  g.x += (int64_t)g.n * g.n_in;
  g.y += g.n;
  g.n = rest;
  return launch_rows<1, 5, false>(g, s);
}

// loss, and gradients of every parameter or one Adam step (device x and t)
cudaError_t train(beor_mlp* m, const float* x, const float* t, int n, const Adam* adam, cudaStream_t s) {
  Net g = net_of(m, x, n);
  g.t = t;
  g.nparts = (n + 15) / 16;
  // pre-activations of at most four hidden layers leave room for a four-stage ring
  cudaError_t e = m->L <= 5 ? launch_rows<1, 4, true>(g, s) : launch_rows<1, 2, true>(g, s);
  if (e != cudaSuccess) return e;
  Params q{};
  q.update = adam != nullptr;
  if (adam) q.adam = *adam;
  int cta = 0;
  for (int l = 0; l < m->L; ++l) {
    q.W[l] = m->W[l];
    q.mW[l] = m->mW[l];
    q.vW[l] = m->vW[l];
    q.gW[l] = m->gW[l];
    q.b[l] = m->b[l];
    q.mb[l] = m->mb[l];
    q.vb[l] = m->vb[l];
    q.gb[l] = m->gb[l];
    q.first[l] = cta;
    cta += ((m->fout[l] + kGO - 1) / kGO) * ((m->fin[l] + kGI - 1) / kGI);
  }
  q.first[m->L] = cta;
  for (int l = 0; l < m->L; ++l) {
    q.bfirst[l] = cta;
    cta += (m->fout[l] + 31) / 32;
  }
  q.bfirst[m->L] = cta;
  grad_kernel<<<cta, kThreads, 0, s>>>(g, q);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

int beor_mlp_create(beor_mlp** out, int device, int n_in, int width, int depth, uint64_t seed) {
  if (!out || n_in < 1 || n_in > 16 || width < 16 || width > 256 || width % 16 || depth < 1 || depth > 8)
    return BEOR_EINVAL;
  *out = nullptr;
  if (cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    return BEOR_EINVAL;
  }
  beor_mlp* m = new beor_mlp();
  m->device = device;
  m->n_in = n_in;
  m->width = width;
  m->depth = depth;
  m->L = depth + 1;
  for (int l = 0; l < m->L; ++l) {
    m->fin[l] = l == 0 ? n_in : width;
    m->fout[l] = l == m->L - 1 ? 1 : width;
    m->kin[l] = pad16(m->fin[l]);
    m->kout[l] = l == m->L - 1 ? 16 : width;
  }
  cudaError_t e = cudaSuccess;
  for (int l = 0; l < m->L && e == cudaSuccess; ++l) {
    const size_t nw = (size_t)m->fout[l] * m->fin[l];
    e = dalloc(m, (void**)&m->W[l], sizeof(float) * nw);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->gW[l], sizeof(float) * nw);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->mW[l], sizeof(float) * nw);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->vW[l], sizeof(float) * nw);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->b[l], sizeof(float) * m->fout[l]);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->gb[l], sizeof(float) * m->fout[l]);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->mb[l], sizeof(float) * m->fout[l]);
    if (e == cudaSuccess) e = dalloc(m, (void**)&m->vb[l], sizeof(float) * m->fout[l]);
    if (e == cudaSuccess)
      e = dalloc(m, (void**)&m->Wb[l], sizeof(__nv_bfloat16) * (size_t)m->kout[l] * m->kin[l]);
    if (e == cudaSuccess) {
      init_kernel<<<256, 256>>>(m->W[l], (int64_t)nw, m->fin[l], seed, l);
      to_bf16_kernel<<<(unsigned)((nw + 255) / 256), 256>>>(m->W[l], m->fout[l], m->fin[l], m->kin[l], m->Wb[l]);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->x_shift, sizeof(float) * n_in);
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->x_scale, sizeof(float) * n_in);
  if (e == cudaSuccess) e = dalloc(m, (void**)&m->loss, sizeof(float));
  if (e == cudaSuccess) {
    std::vector<float> one(n_in, 1.0f);
    e = cudaMemcpy(m->x_scale, one.data(), sizeof(float) * n_in, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = ensure_cap(m, 1024);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    for (void* p : m->owned)
      if (p) cudaFree(p);
    delete m;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? BEOR_ENOMEM : BEOR_ECUDA;
  }
  *out = m;
  return BEOR_OK;
}

int beor_mlp_destroy(beor_mlp* m) {
  if (!m) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  cudaDeviceSynchronize();
  for (void* p : m->owned)
    if (p) cudaFree(p);
  delete m;
  return BEOR_OK;
}

int beor_mlp_set_norm(beor_mlp* m, const float* x_shift, const float* x_scale, float y_shift, float y_scale) {
  if (!m || !x_shift || !x_scale || !(y_scale != 0.0f)) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  if (copy_in(m->x_shift, x_shift, sizeof(float) * m->n_in, 0) != cudaSuccess ||
      copy_in(m->x_scale, x_scale, sizeof(float) * m->n_in, 0) != cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess)
    return BEOR_ECUDA;
  m->y_shift = y_shift;
  m->y_scale = y_scale;
  return BEOR_OK;
}

int beor_mlp_infer(beor_mlp* m, const float* x, int n, float* y_out, void* stream) {
  if (!m || !x || !y_out || n <= 0) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  const int chunk = 65536;
  // In place where the kernel may address the caller's memory; predictions that
  // would go over inputs which other CTAs have yet to read are copied out after
  // the chunk's kernel, as those to other memory are.
  const uintptr_t x0 = reinterpret_cast<uintptr_t>(x), y0 = reinterpret_cast<uintptr_t>(y_out);
  const bool apart = y0 + sizeof(float) * (size_t)n <= x0 || x0 + sizeof(float) * (size_t)n * m->n_in <= y0;
  const Where xw = where_is(x, m->device), yw = where_is(y_out, m->device);
  const bool x_here = xw == HERE, y_here = yw == HERE && (apart || !x_here), dev_out = yw != HOST;
  if ((!x_here || !y_here) && ensure_io(m, std::min(n, chunk)) != cudaSuccess) return BEOR_ENOMEM;
  for (int off = 0; off < n; off += chunk) {
    const int c = std::min(chunk, n - off);
    const float* xc = x + (int64_t)off * m->n_in;
    if (!x_here) {
      if (cudaMemcpyAsync(m->xin, xc, sizeof(float) * (size_t)c * m->n_in,
                          xw == HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return BEOR_ECUDA;
      xc = m->xin;
    }
    if (predict(m, xc, c, y_here ? y_out + off : m->yout, s) != cudaSuccess) return BEOR_ECUDA;
    if (!y_here && cudaMemcpyAsync(y_out + off, m->yout, sizeof(float) * c,
                                   dev_out ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s) != cudaSuccess)
      return BEOR_ECUDA;
  }
  if (!dev_out && cudaStreamSynchronize(s) != cudaSuccess) return BEOR_ECUDA;
  return cudaGetLastError() == cudaSuccess ? BEOR_OK : BEOR_ECUDA;
}

static int mlp_train(beor_mlp* m, const float* x, const float* y, int n, const Adam* adam, float* loss_out,
                     cudaStream_t s) {
  if (ensure_cap(m, n) != cudaSuccess) return BEOR_ENOMEM;
  if (copy_in(m->xin, x, sizeof(float) * (size_t)n * m->n_in, s) != cudaSuccess) return BEOR_ECUDA;
  if (copy_in(m->tin, y, sizeof(float) * (size_t)n, s) != cudaSuccess) return BEOR_ECUDA;
  if (train(m, m->xin, m->tin, n, adam, s) != cudaSuccess) return BEOR_ECUDA;
  if (loss_out) {
    if (cudaMemcpyAsync(loss_out, m->loss, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess) return BEOR_ECUDA;
  }
  return BEOR_OK;
}

int beor_mlp_train_step(beor_mlp* m, const float* x, const float* y, int n, float lr, float beta1, float beta2,
                        float eps, float* loss_out, void* stream) {
  if (!m || !x || !y || n <= 0 || !(lr > 0.0f)) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  const float step = (float)(m->step + 1);
  const Adam a{lr, beta1, beta2, eps, 1.0f - powf(beta1, step), 1.0f - powf(beta2, step)};
  const int r = mlp_train(m, x, y, n, &a, loss_out, s);
  if (r) return r;
  m->step += 1;
  if (loss_out && cudaStreamSynchronize(s) != cudaSuccess) return BEOR_ECUDA;
  return BEOR_OK;
}

int beor_mlp_grad(beor_mlp* m, const float* x, const float* y, int n, int layer, float* dW, float* db,
                  float* loss_out) {
  if (!m || !x || !y || n <= 0 || layer < 0 || layer >= m->L) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  int r = mlp_train(m, x, y, n, nullptr, loss_out, 0);
  if (r) return r;
  if (cudaDeviceSynchronize() != cudaSuccess) return BEOR_ECUDA;
  if (dW && cudaMemcpy(dW, m->gW[layer], sizeof(float) * (size_t)m->fout[layer] * m->fin[layer],
                       cudaMemcpyDeviceToHost) != cudaSuccess)
    return BEOR_ECUDA;
  if (db && cudaMemcpy(db, m->gb[layer], sizeof(float) * m->fout[layer], cudaMemcpyDeviceToHost) != cudaSuccess)
    return BEOR_ECUDA;
  return BEOR_OK;
}

int beor_mlp_get_params(beor_mlp* m, int layer, float* W, float* b) {
  if (!m || layer < 0 || layer >= m->L) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  if (W && cudaMemcpy(W, m->W[layer], sizeof(float) * (size_t)m->fout[layer] * m->fin[layer],
                      cudaMemcpyDeviceToHost) != cudaSuccess)
    return BEOR_ECUDA;
  if (b && cudaMemcpy(b, m->b[layer], sizeof(float) * m->fout[layer], cudaMemcpyDeviceToHost) != cudaSuccess)
    return BEOR_ECUDA;
  return BEOR_OK;
}

int beor_mlp_set_params(beor_mlp* m, int layer, const float* W, const float* b) {
  if (!m || layer < 0 || layer >= m->L) return BEOR_EINVAL;
  cudaSetDevice(m->device);
  const size_t nw = (size_t)m->fout[layer] * m->fin[layer];
  if (W) {
    if (copy_in(m->W[layer], W, sizeof(float) * nw, 0) != cudaSuccess) return BEOR_ECUDA;
    to_bf16_kernel<<<(unsigned)((nw + 255) / 256), 256>>>(m->W[layer], m->fout[layer], m->fin[layer], m->kin[layer],
                                                          m->Wb[layer]);
  }
  if (b && copy_in(m->b[layer], b, sizeof(float) * m->fout[layer], 0) != cudaSuccess) return BEOR_ECUDA;
  return cudaDeviceSynchronize() == cudaSuccess ? BEOR_OK : BEOR_ECUDA;
}

}  // extern "C"
