// Device helpers of the multi-resolution hash-grid encoding (Sections 3.1
// and 3.3 of the paper): the 8 corner rows of a cell and their trilinear
// weights, and vector loads of one table row.
#pragma once

#include "nvc_internal.cuh"

namespace nvc {

template <int F>
struct FeatVec {
  float v[F];
};

template <int F>
__device__ __forceinline__ FeatVec<F> load_feat(const float* p) {
  FeatVec<F> r;
  if constexpr (F == 1) {
    r.v[0] = __ldg(p);
  } else if constexpr (F == 2) {
    const float2 a = __ldg(reinterpret_cast<const float2*>(p));
    r.v[0] = a.x;
    r.v[1] = a.y;
  } else {
#pragma unroll
    for (int k = 0; k < F; k += 4) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(p + k));
      r.v[k] = a.x;
      r.v[k + 1] = a.y;
      r.v[k + 2] = a.z;
      r.v[k + 3] = a.w;
    }
  }
  return r;
}

// Corner rows and trilinear weights of one (position, level).
struct Corners {
  uint32_t row[8];
  float w[8];
};

__device__ __forceinline__ void level_corners(const EncodeParams& ep, int l, float x, float y,
                                              float z, Corners& cr) {
  const int n = ep.res[l];
  int cx, cy, cz;
  float fx, fy, fz;
  grid_cell(x, n, cx, fx);
  grid_cell(y, n, cy, fy);
  grid_cell(z, n, cz, fz);
  const uint32_t mask = (1u << ep.log2_table) - 1u;
  const float gx[2] = {1.0f - fx, fx}, gy[2] = {1.0f - fy, fy}, gz[2] = {1.0f - fz, fz};
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const int dx = d & 1, dy = (d >> 1) & 1, dz = (d >> 2) & 1;
    cr.row[d] = grid_hash((uint32_t)(cx + dx), (uint32_t)(cy + dy), (uint32_t)(cz + dz)) & mask;
    cr.w[d] = gx[dx] * gy[dy] * gz[dz];
  }
}

// The trilinear blend of one (position, level): corners in order, each
// feature one chain of fused multiply-adds.
template <int F>
__device__ __forceinline__ void encode_corners(const EncodeParams& ep, const float* __restrict__ table,
                                               int l, float x, float y, float z, float (&acc)[F]) {
  Corners cr;
  level_corners(ep, l, x, y, z, cr);
  const float* tab = table + ((int64_t)l << ep.log2_table) * F;
#pragma unroll
  for (int f = 0; f < F; ++f) acc[f] = 0.0f;
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const FeatVec<F> v = load_feat<F>(tab + (int64_t)cr.row[d] * F);
#pragma unroll
    for (int f = 0; f < F; ++f) acc[f] = fmaf(cr.w[d], v.v[f], acc[f]);
  }
}

// Adds the adjoint of one (position, level) into the table gradient: the
// feature gradient g times the corner's weight into each corner row.
template <int F>
__device__ __forceinline__ void scatter_corners(const EncodeParams& ep, float* grad, int l, float x,
                                                float y, float z, const float (&g)[F]) {
  Corners cr;
  level_corners(ep, l, x, y, z, cr);
  float* tab = grad + ((int64_t)l << ep.log2_table) * F;
  if constexpr (F == 2) {
    // The x-corners d, d + 1 of each (y, z) pair: when their rows are the two
    // rows of one aligned 16-byte pair -- always for an even cell x, as the
    // x prime is 1 and so hash(x + 1) = hash(x) ^ 1 -- one 16-byte atomic
    // adds both; otherwise two 8-byte atomics.
#pragma unroll
    for (int d = 0; d < 8; d += 2) {
      const uint32_t r0 = cr.row[d], r1 = cr.row[d + 1];
      const float2 g0 = make_float2(cr.w[d] * g[0], cr.w[d] * g[1]);
      const float2 g1 = make_float2(cr.w[d + 1] * g[0], cr.w[d + 1] * g[1]);
      if ((r0 ^ r1) == 1u) {
        const float4 v = (r0 & 1u) ? make_float4(g1.x, g1.y, g0.x, g0.y)
                                   : make_float4(g0.x, g0.y, g1.x, g1.y);
        atomicAdd(reinterpret_cast<float4*>(tab + (int64_t)(r0 & ~1u) * 2), v);
      } else {
        atomicAdd(reinterpret_cast<float2*>(tab + (int64_t)r0 * 2), g0);
        atomicAdd(reinterpret_cast<float2*>(tab + (int64_t)r1 * 2), g1);
      }
    }
    return;
  }
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    float* dst = tab + (int64_t)cr.row[d] * F;
    if constexpr (F % 4 == 0) {
#pragma unroll
      for (int k = 0; k < F; k += 4)
        atomicAdd(reinterpret_cast<float4*>(dst + k),
                  make_float4(cr.w[d] * g[k], cr.w[d] * g[k + 1], cr.w[d] * g[k + 2],
                              cr.w[d] * g[k + 3]));
    } else {
#pragma unroll
      for (int f = 0; f < F; ++f) atomicAdd(dst + f, cr.w[d] * g[f]);
    }
  }
}

}  // namespace nvc
