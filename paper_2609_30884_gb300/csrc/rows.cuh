// Device helpers of the decode rows: fp32 rows between the layers, split into bf16 terms where a
// weight pass multiplies them, and the partial sums that such a pass leaves for its consumer.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace crf {

// Element (r, col) of a weight pass's output: its K splits summed in order, the loads of up to
// eight of them in flight together (one L2 round trip).
__device__ __forceinline__ float part_sum(const RowPart& t, int r, int col) {
  const float* q = t.p + static_cast<size_t>(r) * t.ncols + col;
  float v = __ldcg(q);
  if (t.splits == 1) return v;
  const size_t stride = static_cast<size_t>(t.rows) * t.ncols;
  for (int s0 = 1; s0 < t.splits; s0 += 8) {
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = s0 + i < t.splits ? __ldcg(q + (s0 + i) * stride) : 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) v += x[i];
  }
  return v;
}

// One row of an up factor B [out, rank] (rank 4, 8 or 16) in registers: weights, so it may be
// read before the kernel that a launch depends on has finished.
struct UpRow {
  uint4 a, b;
};
__device__ __forceinline__ UpRow up_row(const __nv_bfloat16* __restrict__ B, int j, int rank) {
  UpRow u;
  u.a = u.b = make_uint4(0u, 0u, 0u, 0u);
  if (!B) return u;
  const __nv_bfloat16* br = B + static_cast<size_t>(j) * rank;
  if (rank == 16) {
    u.a = __ldg(reinterpret_cast<const uint4*>(br));
    u.b = __ldg(reinterpret_cast<const uint4*>(br) + 1);
  } else if (rank == 8) {
    u.a = __ldg(reinterpret_cast<const uint4*>(br));
  } else {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(br));
    u.a.x = v.x;
    u.a.y = v.y;
  }
  return u;
}
// sum_k B[j, k] xa[k] over 16 entries (those past the rank are zero on both sides)
__device__ __forceinline__ float up_dot(const UpRow& u, const float* xa) {
  const uint32_t w[8] = {u.a.x, u.a.y, u.a.z, u.a.w, u.b.x, u.b.y, u.b.z, u.b.w};
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) s += bf16_lo(w[i]) * xa[2 * i] + bf16_hi(w[i]) * xa[2 * i + 1];
  return s;
}

// v as kTerms bf16 terms (each the rounding of what the ones before leave), stored `dim` apart:
// two keep about 16 mantissa bits, three all 24 of an fp32 value. An infinity or NaN is its first term
// alone, and a value that would round to infinity is cut off instead: its terms still sum to it.
template <int kTerms>
__device__ __forceinline__ void store_terms(__nv_bfloat16* dst, int dim, float v) {
  __nv_bfloat16 h = __float2bfloat16_rn(v);
  float rest = v - __bfloat162float(h);
  if (!isfinite(rest)) {
    if (isfinite(v)) h = __float2bfloat16_rz(v);
    rest = isfinite(v) ? v - __bfloat162float(h) : 0.f;
  }
  dst[0] = h;
#pragma unroll
  for (int t = 1; t < kTerms; ++t) {
    h = __float2bfloat16_rn(rest);
    dst[static_cast<size_t>(t) * dim] = h;
    rest -= __bfloat162float(h);
  }
}

}  // namespace crf
