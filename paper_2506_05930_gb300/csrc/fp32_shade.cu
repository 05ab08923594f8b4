// Float32 inference, weighted reservoir sampling and Neural DI in one kernel
// (Sections 3.1 to 3.3 of the paper): the shading path of nvc_shade with
// fused = 0 and of float32 handles.
//
// A warp takes 32 consecutive pixels at a time and keeps them to the end:
// lane = pixel for the encode and the sampler, 4 pixels x 8 outputs per lane
// in the layers (dot_rows), activations in the warp's own shared memory, so
// only warp barriers stand between the phases and the warps of an SM overlap
// one another's gathers, products and sampler arithmetic.  The weights are
// staged once per CTA; warps stride over the tiles.
//
// Neighbouring pixels share the coarse levels' cells, so with a pixel per
// lane a warp's row gathers coalesce.  A pixel's visibilities, then its
// light weights, stay in shared memory between the sampler's passes.
//
// Every pixel's arithmetic is that of the separate encode and MLP kernels
// (same operations in the same order), so the results are theirs bit for bit.
//
// Measured, 1920x1080 pixels of the paper's preset (10 levels x 4 features,
// MLP 40-32-32-32, 32 lights): 0.611 ms; as three kernels that staged
// features and visibilities in memory, 65,536 pixels at a time, 2.78 ms (MLP
// 1.57, encode 0.48, sampler 0.77).  Bound by instruction issue; 24 warps an
// SM (80 registers) took 0.611 ms, 16 warps 0.625, and contributions one
// light at a time 0.666.
#include <cfloat>

#include "exact_pair.cuh"
#include "fp32_common.cuh"
#include "fused_common.cuh"
#include "hashgrid.cuh"
#include "wrs.cuh"

namespace nvc {

namespace {

using namespace f32;

struct ShadeArgs {
  const float* pos;
  const float* nrm;
  int64_t n;
  const float* params;
  EncodeParams ep;
  Net net;
  int light_off;        // float offsets in shared memory: the lights,
  int warp_off;         // the first warp's activations and
  int warp_floats;      // their size per warp;
  int odd_off;          // activations of odd layers within the warp's area
  const float* lights;
  int L;
  uint32_t k0, k1, frame, view;
  int64_t pixel_offset;
  float neg0;           // -0.0f (exact_pair.cuh)
  int32_t* idx;
  float* pdf;
  float* wsum;
  float* radiance;
  float* vis;           // !SHADE: [n][L]
};

constexpr int kWarps = 8;

template <int F, bool SHADE>
__global__ void __launch_bounds__(kWarps * 32, 3) shade_f32_kernel(const __grid_constant__ ShadeArgs a) {
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  stage_weights(a.net, a.params, sm, threadIdx.x, blockDim.x);
  float4* s_l = reinterpret_cast<float4*>(sm + a.light_off);
  bool lights_ok = true;
  if constexpr (SHADE) {
    // in groups of four, zero lights past the last
    for (int e = threadIdx.x; e < ((a.L + 3) & ~3); e += blockDim.x) {
      float4 l = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < a.L) l = reinterpret_cast<const float4*>(a.lights)[e];
      l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
      xp::put_light(s_l, e, l);
      lights_ok = lights_ok && xp::light_ok(l);
    }
  }
  lights_ok = __syncthreads_and(lights_ok) != 0;
  float* buf = sm + a.warp_off + warp * a.warp_floats;
  const int rg = lane & 7, og = lane >> 3;   // the lane's 4 pixels and 8 outputs of 32
  const int L = a.L, last = a.net.n_layers - 1;
  const int64_t n_tiles = (a.n + kRows - 1) / kRows;
  for (int64_t tile = (int64_t)blockIdx.x * n_warps + warp; tile < n_tiles;
       tile += (int64_t)gridDim.x * n_warps) {
    const int64_t row = tile * kRows + lane;
    const bool live = row < a.n;
    float px = 0.f, py = 0.f, pz = 0.f;
    if (live) {
      px = __ldg(a.pos + 3 * row);
      py = __ldg(a.pos + 3 * row + 1);
      pz = __ldg(a.pos + 3 * row + 2);
    }
    // ---- encode --------------------------------------------------------------
    {
      const float x = normalise(px, a.ep.lo[0], a.ep.ext[0]);
      const float y = normalise(py, a.ep.lo[1], a.ep.ext[1]);
      const float z = normalise(pz, a.ep.lo[2], a.ep.ext[2]);
      for (int l = 0; l < a.ep.n_levels; ++l) {
        float acc[F];
        encode_corners<F>(a.ep, a.params, l, x, y, z, acc);
#pragma unroll
        for (int f = 0; f < F; ++f) buf[(l * F + f) * kLd + lane] = acc[f];
      }
    }
    __syncwarp();
    // ---- the network ---------------------------------------------------------
    for (int k = 0; k <= last; ++k) {
      const int po = a.net.po[k], ldw = po + 4;
      const float* src = buf + ((k & 1) ? a.odd_off : 0);
      float* dst = buf + ((k & 1) ? 0 : a.odd_off);
      const float* wk = sm + a.net.t_off[k];
      for (int j0 = 0; j0 < po; j0 += 32) {
        const int jb = j0 + og * 8;
        float2 acc[4][4];
        if (jb < po) dot_rows<4>(src + rg * 4, wk + jb, ldw, a.net.in[k], acc);
        __syncwarp();   // dst may be src (every layer within one 32-output pass)
        if (jb < po) {
          if (k < last || SHADE) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                float4 v = column<4>(acc, p, e);
                if (k < last)
                  v = make_float4(act_fn(v.x, a.net.slope), act_fn(v.y, a.net.slope),
                                  act_fn(v.z, a.net.slope), act_fn(v.w, a.net.slope));
                else
                  v = make_float4(sigmoid_f(v.x), sigmoid_f(v.y), sigmoid_f(v.z), sigmoid_f(v.w));
                *reinterpret_cast<float4*>(dst + (jb + 2 * p + e) * kLd + rg * 4) = v;
              }
          } else {
            const bool wide = (L & 3) == 0 && (reinterpret_cast<uintptr_t>(a.vis) & 15) == 0;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const int64_t q = tile * kRows + rg * 4 + r;
              if (q >= a.n) break;
              float* out = a.vis + q * L + jb;
#pragma unroll
              for (int p = 0; p < 4; p += 2) {
                const float4 v = make_float4(sigmoid_f(acc[r][p].x), sigmoid_f(acc[r][p].y),
                                             sigmoid_f(acc[r][p + 1].x), sigmoid_f(acc[r][p + 1].y));
                if (wide) {   // L is a multiple of 4: a group of 4 is real or padding
                  if (jb + 2 * p < L) *reinterpret_cast<float4*>(out + 2 * p) = v;
                } else {
                  const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                  for (int c = 0; c < 4; ++c)
                    if (jb + 2 * p + c < L) out[2 * p + c] = vv[c];
                }
              }
            }
          }
        }
      }
      __syncwarp();
    }
    // ---- light weights, reservoir, Neural DI ---------------------------------
    if constexpr (SHADE) {
      if (live) {
        float* v = buf + ((a.net.n_layers & 1) ? a.odd_off : 0) + lane;
        const float nx = __ldg(a.nrm + 3 * row), ny = __ldg(a.nrm + 3 * row + 1),
                    nz = __ldg(a.nrm + 3 * row + 2);
        float wmax = 0.0f, sum = 0.0f, di = 0.0f;
        const xp::Pixel pixel_pairs = xp::make_pixel(px, py, pz, nx, ny, nz, a.neg0, lights_ok);
        for (int i0 = 0; i0 < L; i0 += 4) {
          float c[4];
          xp::staged_contributions<2>(pixel_pairs, s_l + i0, c);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (i0 + q < L) {
              const float vi = v[(i0 + q) * kLd];
              const float wi = __fmul_rn(fmaxf(vi, bits_f(kVisClampBits)), c[q]);
              wmax = fmaxf(wmax, wi);
              sum += wi;
              di = fmaf(vi, c[q], di);
              v[(i0 + q) * kLd] = wi;
            }
          }
        }
        int sel = -1;
        const uint32_t pixel = (uint32_t)(a.pixel_offset + row);
        if (!(wmax <= FLT_MAX)) {   // an infinite weight: the general form
          sel = wrs_stream([&](int i) { return v[i * kLd]; }, L, wmax, pixel, a.frame, a.view, a.k0,
                           a.k1);
        } else if (wmax > 0.0f) {
          const fz::QuantScale qs = fz::quant_scale(wmax);
          uint32_t Q = 0;
          for (int i0 = 0; i0 < L; i0 += 4) {
            const uint4 r = philox4x32_10(
                make_uint4(pixel, a.frame, a.view, ((uint32_t)(i0 >> 2) << 4) | kTagWrs), a.k0, a.k1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              if (i0 + c < L) {
                const uint32_t q =
                    fz::quantize_scaled(__fmul_rn(v[(i0 + c) * kLd], qs.pre), qs.scale);
                Q += q;
                if (__umulhi(fz::pick_word(r, c), Q) < q) sel = i0 + c;
              }
            }
          }
        }
        if (a.idx) a.idx[row] = sel;
        if (a.pdf) a.pdf[row] = sel >= 0 ? v[sel * kLd] / sum : 0.0f;
        if (a.wsum) a.wsum[row] = sum;
        if (a.radiance) a.radiance[row] = di;
      }
      __syncwarp();
    }
  }
}

// Sampling and Neural DI on visibilities in memory (vis [n][L]), a pixel per
// thread: the second half of the staged form below.
__global__ void __launch_bounds__(128) shade_from_vis_kernel(
    const float* __restrict__ lights, int L, const float* __restrict__ pos,
    const float* __restrict__ nrm, const float* __restrict__ vis, int64_t n, uint32_t k0,
    uint32_t k1, uint32_t frame, uint32_t view, int64_t pixel_offset, int32_t* __restrict__ idx,
    float* __restrict__ pdf, float* __restrict__ wsum, float* __restrict__ radiance, float neg0) {
  extern __shared__ float4 s_lights[];
  bool lights_ok = true;
  for (int e = threadIdx.x; e < ((L + 3) & ~3); e += blockDim.x) {
    float4 l = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < L) l = reinterpret_cast<const float4*>(lights)[e];
    l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
    xp::put_light(s_lights, e, l);
    lights_ok = lights_ok && xp::light_ok(l);
  }
  lights_ok = __syncthreads_and(lights_ok) != 0;
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float px = pos[3 * p], py = pos[3 * p + 1], pz = pos[3 * p + 2];
  const xp::Pixel pp = xp::make_pixel(px, py, pz, nrm[3 * p], nrm[3 * p + 1], nrm[3 * p + 2], neg0,
                                      lights_ok);
  const float* vp = vis + p * L;
  auto weights4 = [&](int i0, float (&c)[4], float (&v)[4], float (&w)[4]) {
    xp::staged_contributions<2>(pp, s_lights + i0, c);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = i0 + q < L ? __ldg(vp + i0 + q) : 0.0f;
      w[q] = __fmul_rn(fmaxf(v[q], bits_f(kVisClampBits)), c[q]);
    }
  };
  float wmax = 0.0f, sum = 0.0f, di = 0.0f;
  for (int i0 = 0; i0 < L; i0 += 4) {
    float c[4], v[4], w[4];
    weights4(i0, c, v, w);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i0 + q < L) {
        wmax = fmaxf(wmax, w[q]);
        sum += w[q];
        di = fmaf(v[q], c[q], di);
      }
  }
  int sel = -1;
  float wsel = 0.0f;
  if (wmax > 0.0f) {
    const bool finite = wmax <= FLT_MAX;   // else quantize_weight itself
    const fz::QuantScale qs = fz::quant_scale(wmax);
    const int e = ilogbf(wmax);
    const uint32_t pixel = (uint32_t)(pixel_offset + p);
    uint64_t Q = 0;
    for (int i0 = 0; i0 < L; i0 += 4) {
      float c[4], v[4], w[4];
      weights4(i0, c, v, w);
      const uint4 r = philox4x32_10(
          make_uint4(pixel, frame, view, ((uint32_t)(i0 >> 2) << 4) | kTagWrs), k0, k1);
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        if (i0 + q4 < L) {
          const uint32_t q = finite ? fz::quantize_scaled(__fmul_rn(w[q4], qs.pre), qs.scale)
                                    : quantize_weight(w[q4], e);
          Q += q;
          if (q != 0u && (uint64_t)fz::pick_word(r, q4) * Q < ((uint64_t)q << 32)) {
            sel = i0 + q4;
            wsel = w[q4];
          }
        }
      }
    }
  }
  if (idx) idx[p] = sel;
  if (pdf) pdf[p] = sel >= 0 ? wsel / sum : 0.0f;
  if (wsum) wsum[p] = sum;
  if (radiance) radiance[p] = di;
}

// Shared memory with `warps` warps per CTA; fills the plan when `a` is given.
// shade: the outputs stay in shared memory too.
size_t plan_smem(const nvc_handle* h, const Net& net, int warps, bool shade, ShadeArgs* a) {
  // activation k (0: the encoded input, n_layers: the outputs) lies in area
  // k & 1; one area serves both while every layer is one 32-output pass,
  // whose products are all read before the first is written back
  int dims[2] = {h->din, 0}, widest = 0;
  for (int k = 0; k < net.n_layers - (shade ? 0 : 1); ++k) {
    int& d = dims[(k + 1) & 1];
    d = net.po[k] > d ? net.po[k] : d;
    widest = net.po[k] > widest ? net.po[k] : widest;
  }
  const bool one = widest <= 32;
  const int area = (one ? (dims[0] > dims[1] ? dims[0] : dims[1]) : dims[0] + dims[1]) * kLd;
  const int light_off = (net.t_floats + 3) & ~3;
  const int warp_off = light_off + 4 * ((h->L + 3) & ~3);
  if (a) {
    a->light_off = light_off;
    a->warp_off = warp_off;
    a->warp_floats = area;
    a->odd_off = one ? 0 : dims[0] * kLd;
  }
  return sizeof(float) * ((size_t)warp_off + (size_t)warps * area);
}

template <int F, bool SHADE>
cudaError_t launch_typed(ShadeArgs& a, const nvc_handle* h, cudaStream_t s) {
  auto kern = shade_f32_kernel<F, SHADE>;
  // four warps share a CTA's weights while there are fewer tiles than eight
  // warps on every SM would take, else eight
  const int64_t tiles = (a.n + kRows - 1) / kRows;
  int warps = tiles >= (int64_t)kWarps * h->num_sms ? kWarps : 4;
  size_t smem = plan_smem(h, a.net, warps, SHADE, &a);
  while (smem > 227 * 1024 && warps > 1) smem = plan_smem(h, a.net, warps /= 2, SHADE, &a);
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t want = (tiles + warps - 1) / warps;
  const int64_t cap = (int64_t)h->num_sms * blocks_per_sm((const void*)kern, warps * 32, smem);
  kern<<<(unsigned)(want < cap ? want : cap), warps * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <bool SHADE>
cudaError_t launch(ShadeArgs& a, const nvc_handle* h, cudaStream_t s) {
  switch (h->F) {
    case 1: return launch_typed<1, SHADE>(a, h, s);
    case 2: return launch_typed<2, SHADE>(a, h, s);
    case 4: return launch_typed<4, SHADE>(a, h, s);
    case 8: return launch_typed<8, SHADE>(a, h, s);
  }
  return cudaErrorInvalidValue;
}

ShadeArgs common_args(const nvc_handle* h, const float* pos, int64_t n) {
  ShadeArgs a{};
  a.pos = pos;
  a.n = n;
  a.params = h->params;
  a.ep = encode_params(h);
  a.net = make_net(h);
  a.L = h->L;
  a.neg0 = -0.0f;
  return a;
}

}  // namespace

cudaError_t launch_infer_f32(const nvc_handle* h, const float* pos, int64_t n, float* vis,
                             cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ShadeArgs a = common_args(h, pos, n);
  a.vis = vis;
  return launch<false>(a, h, s);
}

cudaError_t launch_shade_f32(const nvc_handle* h, const nvc_scene* sc, const float* pos,
                             const float* nrm, int64_t n, uint64_t seed, uint32_t frame,
                             uint32_t view, int64_t pixel_offset, int32_t* idx, float* pdf,
                             float* wsum, float* radiance, cudaStream_t s, int* launches) {
  *launches = 0;
  if (n == 0) return cudaSuccess;
  ShadeArgs a = common_args(h, pos, n);
  a.nrm = nrm;
  a.lights = sc->lights;
  a.k0 = (uint32_t)seed;
  a.k1 = (uint32_t)(seed >> 32);
  a.frame = frame;
  a.view = view;
  a.pixel_offset = pixel_offset;
  a.idx = idx;
  a.pdf = pdf;
  a.wsum = wsum;
  a.radiance = radiance;
  // While four warps' activations, outputs among them, fit beside the weights,
  // all on chip; a wider output layer leaves room for fewer warps than the SM
  // has schedulers, and its visibilities go through the handle's staging.
  // MLP 32-64-64-64-L, 578,731 pixels, on chip / staged (and the three-kernel
  // form before) in us: 32 lights 476 / 769 (1,395), 128 1,434 / 1,533
  // (2,999), 192 3,783 / 2,598 (4,094), 256 4,733 / 3,210 (4,771).
  if (plan_smem(h, a.net, 4, true, nullptr) <= 227 * 1024) {
    *launches = 1;
    return launch<true>(a, h, s);
  }
  const size_t smem = sizeof(float4) * ((h->L + 3) & ~3);
  for (int64_t o = 0; o < n; o += h->stage_pixels) {
    const int64_t m = n - o < h->stage_pixels ? n - o : h->stage_pixels;
    cudaError_t e = launch_infer_f32(h, pos + 3 * o, m, h->s_vis, s);
    if (e != cudaSuccess) return e;
    shade_from_vis_kernel<<<(unsigned)((m + 127) / 128), 128, smem, s>>>(
        sc->lights, h->L, pos + 3 * o, nrm + 3 * o, h->s_vis, m, a.k0, a.k1, frame, view,
        pixel_offset + o, idx ? idx + o : nullptr, pdf ? pdf + o : nullptr,
        wsum ? wsum + o : nullptr, radiance ? radiance + o : nullptr, a.neg0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    *launches += 2;
  }
  return cudaSuccess;
}

}  // namespace nvc
