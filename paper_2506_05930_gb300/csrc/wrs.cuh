// The streaming integer reservoir over float32 weights (Section 3.1's
// weighted reservoir sampling) in its general form.
#pragma once
#include "nvc_internal.cuh"

namespace nvc {

// Reservoir over the weights wfn(0 .. L-1), the largest of which is wmax;
// the selected index or -1.
template <typename WFn>
__device__ __forceinline__ int wrs_stream(WFn wfn, int L, float wmax, uint32_t pixel,
                                          uint32_t frame, uint32_t view, uint32_t k0,
                                          uint32_t k1) {
  if (!(wmax > 0.0f)) return -1;
  const int e = ilogbf(wmax);
  uint64_t Q = 0;
  int sel = -1;
  uint4 r = make_uint4(0, 0, 0, 0);
  for (int i = 0; i < L; ++i) {
    if ((i & 3) == 0)
      r = philox4x32_10(make_uint4(pixel, frame, view, ((uint32_t)(i >> 2) << 4) | kTagWrs), k0, k1);
    const uint32_t ri = (i & 3) == 0 ? r.x : (i & 3) == 1 ? r.y : (i & 3) == 2 ? r.z : r.w;
    const uint32_t q = quantize_weight(wfn(i), e);
    Q += q;
    if (q != 0u && (uint64_t)ri * Q < ((uint64_t)q << 32)) sel = i;
  }
  return sel;
}

}  // namespace nvc
