// One float32 training pass in one kernel (Sections 3.3 and 3.4 of the
// paper): encode, forward, loss and its gradient, the hand-written backward,
// the weight gradients and the hash-grid scatter of a batch whose positions
// and targets are in memory.
//
// A CTA of four warps takes 32 samples at a time and keeps their activations
// and deltas in shared memory; the layers' products are dot_rows with 4
// samples x 2 columns a lane (the warps split the columns), the weight
// gradients 2 x 4 entries a lane over the tile's samples, added to the
// gradient by coalesced atomics, and the encode's and scatter's levels are
// split between the warps (lane = sample).  Small tiles put a batch of a few
// thousand positions on every SM; what bounds the pass there is the latency
// of its chain of layers, which as separate kernels paid a launch and a round
// trip through memory per link.
//
// Activations, deltas and loss terms are formed as the separate kernels form
// them (same operations, same order); the gradient sums' order is that of the
// atomics either way.
//
// Measured: the paper's preset (8192 positions x 32 lights, shadow rays and
// Adam included) 161 -> 69 us a step, and 1024 positions x 4 lights within a
// 64x64 float32 frame 100 -> 49 us a frame together with fp32_shade.cu,
// against eight kernels a pass.
#include "fp32_common.cuh"
#include "hashgrid.cuh"

namespace nvc {

namespace {

using namespace f32;

constexpr int kWarps = 4;
constexpr int kThreads = kWarps * 32;
constexpr size_t kSmemOptin = 227 * 1024;

struct TrainArgs {
  const float* pos;
  const float* target;
  int64_t n;
  const float* params;
  EncodeParams ep;
  Net net;
  int r_off[kMaxLayers];   // float offsets: W_k as stored, [out][pi], for the backward;
  int pi[kMaxLayers];      // inputs rounded up to 8
  int act_off[kMaxLayers]; // activations k, [in_k][kLd];
  int d_off[2];            // the two delta tiles
  int loss;
  float grad_scale;        // loss scale / (n L)
  float* grad;
  double* partials;
  int32_t* status;
};

// Entries (2 tj + q, ti + p ni4) of dW_k over the tile's samples: q < 2, p < 4.
// Consecutive lanes take consecutive columns, so the reads of a (kLd = 4 mod
// 32) are conflict-free, those of d broadcast, and the atomics coalesce.
__device__ __forceinline__ bool weight_gradient(const float* d, const float* act, int out, int in,
                                                float* dw, int t) {
  const int ni4 = (in + 3) >> 2, nj2 = (out + 1) >> 1;
  bool bad = false;
  for (int e = t; e < ni4 * nj2; e += kThreads) {
    const int tj = e / ni4, ti = e - tj * ni4;
    const int j1 = 2 * tj + 1 < out ? 2 * tj + 1 : 2 * tj;
    float2 acc[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[q][p] = make_float2(0.0f, 0.0f);
#pragma unroll 4
    for (int b = 0; b < kRows; b += 4) {
      const float4 d0 = *reinterpret_cast<const float4*>(d + 2 * tj * kLd + b);
      const float4 d1 = *reinterpret_cast<const float4*>(d + j1 * kLd + b);
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int i = ti + p * ni4 < in ? ti + p * ni4 : ti;
        const float4 av = *reinterpret_cast<const float4*>(act + i * kLd + b);
        acc[0][p] = __ffma2_rn(make_float2(d0.x, d0.y), make_float2(av.x, av.y), acc[0][p]);
        acc[0][p] = __ffma2_rn(make_float2(d0.z, d0.w), make_float2(av.z, av.w), acc[0][p]);
        acc[1][p] = __ffma2_rn(make_float2(d1.x, d1.y), make_float2(av.x, av.y), acc[1][p]);
        acc[1][p] = __ffma2_rn(make_float2(d1.z, d1.w), make_float2(av.z, av.w), acc[1][p]);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int j = 2 * tj + q, i = ti + p * ni4;
        if (j < out && i < in) {
          const float v = acc[q][p].x + acc[q][p].y;
          bad = bad || !isfinite(v);
          atomicAdd(dw + (int64_t)j * in + i, v);
        }
      }
  }
  return bad;
}

template <int F>
__global__ void __launch_bounds__(kThreads) train_f32_kernel(const __grid_constant__ TrainArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ double s_red[kWarps];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rg = lane & 7, og = lane >> 3;
  const int last = a.net.n_layers - 1, L = a.net.out[last];
  stage_weights<true>(a.net, a.params, sm, t, kThreads, a.r_off);
  double loss_acc = 0.0;
  bool bad = false;
  const int64_t n_tiles = (a.n + kRows - 1) / kRows;
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t row0 = tile * kRows;
    const bool live = row0 + lane < a.n;
    float x = 0.f, y = 0.f, z = 0.f;
    if (live) {
      const float* p = a.pos + 3 * (row0 + lane);
      x = normalise(__ldg(p), a.ep.lo[0], a.ep.ext[0]);
      y = normalise(__ldg(p + 1), a.ep.lo[1], a.ep.ext[1]);
      z = normalise(__ldg(p + 2), a.ep.lo[2], a.ep.ext[2]);
    }
    for (int l = warp; l < a.ep.n_levels; l += kWarps) {
      float acc[F];
      encode_corners<F>(a.ep, a.params, l, x, y, z, acc);
#pragma unroll
      for (int f = 0; f < F; ++f)
        sm[a.act_off[0] + (l * F + f) * kLd + lane] = live ? acc[f] : 0.0f;
    }
    __syncthreads();
    // ---- forward and loss ------------------------------------------------------
    int cur = 0;
    for (int k = 0; k <= last; ++k) {
      const int po = a.net.po[k], ldw = po + 4;
      for (int j0 = 0; j0 < po; j0 += 32) {
        const int jb = j0 + warp * 8 + og * 2;
        if (jb >= po) continue;
        float2 acc[4][1];
        dot_rows<1>(sm + a.act_off[k] + rg * 4, sm + a.net.t_off[k] + jb, ldw, a.net.in[k], acc);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = jb + e;
          const float4 zv = column<1>(acc, 0, e);
          float v[4] = {zv.x, zv.y, zv.z, zv.w};
          if (k < last) {
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = act_fn(v[r], a.net.slope);
          } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int64_t row = row0 + rg * 4 + r;
              float g = 0.0f;
              if (row < a.n && j < L) {
                const float zz = v[r], yy = __ldg(a.target + row * L + j);
                const float s = sigmoid_f(zz);
                if (a.loss == NVC_LOSS_BCE) {
                  loss_acc += (double)(fmaxf(zz, 0.0f) + log1pf(expf(-fabsf(zz))) - yy * zz);
                  g = s - yy;
                } else {
                  const float d = s - yy;
                  loss_acc += (double)d * (double)d;
                  g = 2.0f * d * s * (1.0f - s);
                }
                g *= a.grad_scale;
                bad = bad || !isfinite(zz) || !isfinite(g);
              }
              v[r] = g;
            }
          }
          const int dst = k < last ? a.act_off[k + 1] : a.d_off[0];
          *reinterpret_cast<float4*>(sm + dst + j * kLd + rg * 4) = make_float4(v[0], v[1], v[2], v[3]);
        }
      }
      __syncthreads();
    }
    // ---- backward ----------------------------------------------------------------
    for (int k = last; k >= 0; --k) {
      const int in = a.net.in[k], out = a.net.out[k], pi = a.pi[k];
      const float* d = sm + a.d_off[cur];
      float* dn = sm + a.d_off[cur ^ 1];
      const float* act = sm + a.act_off[k];
      // g = delta W_k, times act' below the top (act_k holds leaky_relu(z_{k-1}))
      for (int i0 = 0; i0 < pi; i0 += 32) {
        const int ib = i0 + warp * 8 + og * 2;
        if (ib >= pi) continue;
        float2 acc[4][1];
        dot_rows<1>(d + rg * 4, sm + a.r_off[k] + ib, pi, out, acc);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          if (ib + e >= in) continue;
          float4 g = column<1>(acc, 0, e);
          if (k > 0) {
            const float4 h = *reinterpret_cast<const float4*>(act + (ib + e) * kLd + rg * 4);
            g.x = h.x > 0.0f ? g.x : a.net.slope * g.x;
            g.y = h.y > 0.0f ? g.y : a.net.slope * g.y;
            g.z = h.z > 0.0f ? g.z : a.net.slope * g.z;
            g.w = h.w > 0.0f ? g.w : a.net.slope * g.w;
          }
          *reinterpret_cast<float4*>(dn + (ib + e) * kLd + rg * 4) = g;
        }
      }
      bad = weight_gradient(d, act, out, in, a.grad + a.net.w_off[k], t) || bad;
      __syncthreads();
      cur ^= 1;
    }
    // ---- the encoding's adjoint ------------------------------------------------
    if (live) {
      const float* df = sm + a.d_off[cur];
      for (int l = warp; l < a.ep.n_levels; l += kWarps) {
        float g[F];
        bool finite = true;
#pragma unroll
        for (int f = 0; f < F; ++f) {
          g[f] = df[(l * F + f) * kLd + lane];
          finite = finite && isfinite(g[f]);
        }
        if (finite)
          scatter_corners<F>(a.ep, a.grad, l, x, y, z, g);
        else
          bad = true;
      }
    }
    __syncthreads();   // the next tile rewrites what this one still reads
  }
  for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_down_sync(0xffffffffu, loss_acc, o);
  if (lane == 0) s_red[warp] = loss_acc;
  const bool any_bad = __syncthreads_or(bad) != 0;
  if (t == 0) {
    double s = 0.0;
    for (int w = 0; w < kWarps; ++w) s += s_red[w];
    a.partials[blockIdx.x] = s;
    if (any_bad) atomicOr(a.status + kStNonFinite, 1);
  }
}

// Shared memory of the pass; fills the offsets of `a`.
size_t plan(const nvc_handle* h, TrainArgs& a) {
  a.net = make_net(h);
  int off = (a.net.t_floats + 3) & ~3, widest = 0;
  for (int k = 0; k < h->n_layers; ++k) {
    a.pi[k] = round8(a.net.in[k]);
    a.r_off[k] = off;
    off += a.net.out[k] * a.pi[k];
  }
  for (int k = 0; k < h->n_layers; ++k) {
    a.act_off[k] = off;
    off += a.net.in[k] * kLd;
    widest = a.net.in[k] > widest ? a.net.in[k] : widest;
    widest = a.net.po[k] > widest ? a.net.po[k] : widest;
  }
  for (int b = 0; b < 2; ++b) {
    a.d_off[b] = off;
    off += widest * kLd;
  }
  return sizeof(float) * (size_t)off;
}

template <int F>
cudaError_t launch_typed(const TrainArgs& a, int grid, size_t smem, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(train_f32_kernel<F>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  train_f32_kernel<F><<<grid, kThreads, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

bool train_f32_fits(const nvc_handle* h) {
  TrainArgs a{};
  return plan(h, a) <= kSmemOptin - 64;   // 64: the kernel's static shared memory
}

cudaError_t launch_train_f32(nvc_handle* h, int64_t n, int* blocks_used, cudaStream_t s) {
  TrainArgs a{};
  const size_t smem = plan(h, a);
  a.pos = h->t_pos;
  a.target = h->t_target;
  a.n = n;
  a.params = h->params;
  a.ep = encode_params(h);
  a.loss = h->cfg.loss;
  a.grad_scale = h->cfg.loss_scale / (float)(n * h->L);
  a.grad = h->grad;
  a.partials = h->loss_partials;
  a.status = h->status;
  const int64_t tiles = (n + kRows - 1) / kRows;
  const int grid = (int)(tiles < h->n_loss_partials ? tiles : h->n_loss_partials);
  *blocks_used = grid;
  switch (h->F) {
    case 1: return launch_typed<1>(a, grid, smem, s);
    case 2: return launch_typed<2>(a, grid, smem, s);
    case 4: return launch_typed<4>(a, grid, smem, s);
    case 8: return launch_typed<8>(a, grid, smem, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace nvc
