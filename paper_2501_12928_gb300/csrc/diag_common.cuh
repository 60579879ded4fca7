// Pieces shared by the kernels of the diagonal blocks (diag_cluster.cu,
// diag_tc.cu): packed lower storage and the bf16 slices of the inverse's rows.
#pragma once

#include "beor_common.cuh"
#include "beor_internal.h"

namespace beor {

#define DG_PACK (BEOR_TB * (BEOR_TB + 1) / 2)
__device__ __forceinline__ int pk(int i, int j) { return i * (i + 1) / 2 + j; }

// Slices of Linv (B operand of the panel product L_ik = A_ik Linv^H): columns
// c0 .. c0 + 7 (c0 a multiple of 8) of row r of problem p, exponent e: 16 bytes
// of every plane; value = 2^(e-7) sum_s sigma_s 2^(-8 s), sigma_s integers with
// |sigma_s| <= 128.  Af: packed lower double-float elements.
__device__ __forceinline__ void linv_slice_chunk(const BatchView& v, int p, const float4* Af, int r, int c0, int e) {
  const int64_t lrows = (int64_t)v.P * BEOR_TB, ps = lrows * BEOR_TB;   // plane slice_plane(slice, part) at ps each
  __nv_bfloat16* dst = v.linv_sl + slice_elem_off((int64_t)p * BEOR_TB + r, c0, lrows);
  if (c0 > r) {   // above the diagonal
#pragma unroll
    for (int pl = 0; pl < BEOR_NPLANE; ++pl) *reinterpret_cast<uint4*>(dst + pl * ps) = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  uint32_t packed[BEOR_NPLANE][4];
#pragma unroll
  for (int q = 0; q < 8; q += 2) {
    float val[2][BEOR_NPLANE];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int m = c0 + q + u;
      const float4 a = m <= r ? Af[pk(r, m)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        float dv[BEOR_NSLICE];
        balanced_digits5(part ? a.z : a.x, part ? a.w : a.y, e, dv);
#pragma unroll
        for (int sl = 0; sl < BEOR_NSLICE; ++sl) {
          if (part == 0) {
            val[u][slice_plane(sl, BEOR_PART_RE)] = dv[sl];
          } else {
            val[u][slice_plane(sl, BEOR_PART_IM)] = dv[sl];
            val[u][slice_plane(sl, BEOR_PART_NEGIM)] = -dv[sl];
          }
        }
      }
    }
#pragma unroll
    for (int pl = 0; pl < BEOR_NPLANE; ++pl) {
      const __nv_bfloat162 h2 = __floats2bfloat162_rn(val[0][pl], val[1][pl]);   // .x at the lower address
      packed[pl][q / 2] = *reinterpret_cast<const uint32_t*>(&h2);
    }
  }
#pragma unroll
  for (int pl = 0; pl < BEOR_NPLANE; ++pl)
    *reinterpret_cast<uint4*>(dst + pl * ps) = make_uint4(packed[pl][0], packed[pl][1], packed[pl][2], packed[pl][3]);
}

}  // namespace beor
