// Light weights and weighted reservoir sampling (Section 3.1 of the paper) on
// float32 values already in memory.
//
// WRS runs in integers so that its decision does not depend on the order
// of floating-point sums: per pixel, e = ilogb(max w), q_i = max(1,
// floor(w_i 2^(23-e))) for w_i > 0, Q_i = q_1 + ... + q_i, and candidate i
// replaces the reservoir iff r_i Q_i < q_i 2^32 (r_i a 32-bit Philox word),
// which is the streaming reservoir rule "keep i with probability
// q_i / Q_i".  One thread per pixel streams over the lights in order.
#include "nvc_internal.cuh"
#include "wrs.cuh"

namespace nvc {

namespace {

__global__ void light_weights_kernel(const float* __restrict__ lights, int L,
                                     const float* __restrict__ pos, const float* __restrict__ nrm,
                                     const float* __restrict__ vis, int64_t n,
                                     float* __restrict__ c_out, float* __restrict__ w_out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * L) return;
  const int64_t p = t / L;
  const int i = (int)(t - p * L);
  const float4 lt = reinterpret_cast<const float4*>(lights)[i];
  const float i_over_pi = __fmul_rn(lt.w, bits_f(kInvPiBits));
  const float c = contribution(pos[3 * p], pos[3 * p + 1], pos[3 * p + 2], nrm[3 * p],
                               nrm[3 * p + 1], nrm[3 * p + 2], lt.x, lt.y, lt.z, i_over_pi);
  if (c_out) c_out[t] = c;
  if (w_out) w_out[t] = __fmul_rn(fmaxf(vis[t], bits_f(kVisClampBits)), c);
}

__global__ void wrs_from_weights_kernel(const float* __restrict__ w, int64_t n, int L,
                                        uint32_t k0, uint32_t k1, uint32_t frame, uint32_t view,
                                        int64_t pixel_offset, int32_t* __restrict__ idx,
                                        float* __restrict__ pdf, float* __restrict__ wsum) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float* wp = w + p * L;
  float wmax = 0.0f, sum = 0.0f;
  for (int i = 0; i < L; ++i) {
    const float wi = wp[i];
    wmax = fmaxf(wmax, wi);
    sum += wi;
  }
  const int sel = wrs_stream([&](int i) { return wp[i]; }, L, wmax,
                             (uint32_t)(pixel_offset + p), frame, view, k0, k1);
  if (idx) idx[p] = sel;
  if (pdf) pdf[p] = sel >= 0 ? wp[sel] / sum : 0.0f;
  if (wsum) wsum[p] = sum;
}

}  // namespace

cudaError_t launch_light_weights(const nvc_scene* sc, const float* pos, const float* nrm,
                                 const float* vis, int64_t n, float* c, float* w,
                                 cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t total = n * sc->n_lights;
  light_weights_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(sc->lights, sc->n_lights,
                                                                     pos, nrm, vis, n, c, w);
  return cudaGetLastError();
}

cudaError_t launch_wrs_from_weights(const float* w, int64_t n, int L, uint64_t seed,
                                    uint32_t frame, uint32_t view, int64_t pixel_offset,
                                    int32_t* idx, float* pdf, float* wsum, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  wrs_from_weights_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(
      w, n, L, (uint32_t)seed, (uint32_t)(seed >> 32), frame, view, pixel_offset, idx, pdf, wsum);
  return cudaGetLastError();
}

}  // namespace nvc
