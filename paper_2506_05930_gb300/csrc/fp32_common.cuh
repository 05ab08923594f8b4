// Pieces shared by the float32 kernels that run the whole network on chip
// (fp32_shade.cu, fp32_train.cu): the geometry of the staged weights and the
// 32-row matrix product of one layer.
#pragma once
#include "nvc_internal.cuh"

namespace nvc {
namespace f32 {

constexpr int kMaxLayers = NVC_MAX_HIDDEN_LAYERS + 1;
constexpr int kRows = 32;   // samples of a tile
// Activations lie feature-major, [feature][kLd floats], sample r at r: a
// lane's own sample is conflict-free, and four consecutive samples are one
// 16-byte access whose eight lanes of a phase cover all banks, along the
// samples and (36 = 4 mod 32) along the features.
constexpr int kLd = 36;

struct Net {
  int n_layers;
  int in[kMaxLayers], out[kMaxLayers];
  int po[kMaxLayers];         // outputs rounded up to 8
  int64_t w_off[kMaxLayers];  // float offset of W_k in the parameters
  // staged transposed, [in][po + 4] (the 4 spreads the staging's writes over
  // the banks), zero past the real outputs: float offset of layer k
  int t_off[kMaxLayers];
  int t_floats;
  float slope;
};

__host__ __device__ inline int round8(int x) { return (x + 7) & ~7; }

inline Net make_net(const nvc_handle* h) {
  Net n{};
  n.n_layers = h->n_layers;
  n.slope = h->cfg.leaky_slope;
  int off = 0;
  for (int k = 0; k < h->n_layers; ++k) {
    n.in[k] = h->w_in[k];
    n.out[k] = h->w_out[k];
    n.po[k] = round8(h->w_out[k]);
    n.w_off[k] = h->w_off[k];
    n.t_off[k] = off;
    off += n.in[k] * (n.po[k] + 4);
  }
  n.t_floats = off;
  return n;
}

// Stages every layer transposed at sw and, with `rows`, also as stored, [out]
// [in rounded up to 8], at sw + r_off[k] (zero padding); threads t of nt share
// the work, the caller synchronises.  Reads run along the parameters' rows.
template <bool ROWS = false>
__device__ __forceinline__ void stage_weights(const Net& net, const float* __restrict__ params,
                                              float* sw, int t, int nt,
                                              const int* r_off = nullptr) {
  for (int k = 0; k < net.n_layers; ++k) {
    const int in = net.in[k], out = net.out[k], ld = net.po[k] + 4, pi = round8(in);
    const float* src = params + net.w_off[k];
    float* dst = sw + net.t_off[k];
    // j = e / in by a multiplication, exact for e < 2^16 and 2 <= in <= 128
    const uint32_t inv = (uint32_t)(((1ull << 32) + in - 1) / in);
#pragma unroll 8
    for (int e = t; e < in * out; e += nt) {
      const int j = in == 1 ? e : (int)__umulhi((uint32_t)e, inv), i = e - j * in;
      const float w = __ldg(src + e);
      dst[i * ld + j] = w;
      if constexpr (ROWS) sw[r_off[k] + j * pi + i] = w;
    }
    const int pad = net.po[k] - out;
    for (int e = t; e < in * pad; e += nt) dst[(e / pad) * ld + out + e % pad] = 0.0f;
    if constexpr (ROWS) {
      const int rp = pi - in;
      for (int e = t; e < out * rp; e += nt) sw[r_off[k] + (e / rp) * pi + in + e % rp] = 0.0f;
    }
  }
}

__device__ __forceinline__ float act_fn(float z, float slope) { return z > 0.0f ? z : slope * z; }
__device__ __forceinline__ float sigmoid_f(float z) { return 1.0f / (1.0f + expf(-z)); }

// acc[r][p] = sum over k < n of x[k][4 rg + r] (w[k][2 p], w[k][2 p + 1]), the
// terms added in order of k by fused multiply-adds, two outputs per packed
// one: 4 samples x 2 P outputs a thread, one 16-byte read of x and P/2 of w
// per k, so the FMA pipe and not shared memory sets the rate.
template <int P>
__device__ __forceinline__ void dot_rows(const float* x, const float* w, int ldw, int n,
                                         float2 (&acc)[4][P]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int p = 0; p < P; ++p) acc[r][p] = make_float2(0.0f, 0.0f);
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const float4 xv = *reinterpret_cast<const float4*>(x + k * kLd);
    float2 wv[P];
    if constexpr (P % 2 == 0) {
#pragma unroll
      for (int p = 0; p < P; p += 2) {
        const float4 q = *reinterpret_cast<const float4*>(w + k * ldw + 2 * p);
        wv[p] = make_float2(q.x, q.y);
        wv[p + 1] = make_float2(q.z, q.w);
      }
    } else {
#pragma unroll
      for (int p = 0; p < P; ++p) wv[p] = *reinterpret_cast<const float2*>(w + k * ldw + 2 * p);
    }
    const float xr[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int p = 0; p < P; ++p)
        acc[r][p] = __ffma2_rn(make_float2(xr[r], xr[r]), wv[p], acc[r][p]);
  }
}

// Output column 2 p + e of the four samples as one 16-byte value.
template <int P>
__device__ __forceinline__ float4 column(const float2 (&acc)[4][P], int p, int e) {
  return e ? make_float4(acc[0][p].y, acc[1][p].y, acc[2][p].y, acc[3][p].y)
           : make_float4(acc[0][p].x, acc[1][p].x, acc[2][p].x, acc[3][p].x);
}

}  // namespace f32
}  // namespace nvc
