// The shading pass and the all-lights reference.
//
// Shading (Section 3.1): every pixel casts one shadow ray towards the light
// its reservoir picked and forms the one-sample estimate of Eq. 1,
// V_s c_s / p_s, which is unbiased because the sampler gives every light
// with c_i > 0 a nonzero probability.  A running mean over frames
// (a <- a + (e - a) / k for frame k) accumulates it.
//
// Exact direct illumination (the comparison in Section 4.4): a shadow ray
// from every pixel to every light, sum_i V_i c_i.
//
// Both use the shading path's correctly rounded float32 contribution and
// the shadow-ray tests of the training targets, so each binary decision and
// each float32 result is reproducible operation by operation: the estimate
// is c / p (one division), the running mean three correctly rounded steps,
// and the exact DI a sum over lights in order.
#include "exact_pair.cuh"
#include "nvc_internal.cuh"
#include "shadow.cuh"

namespace nvc {

namespace {

template <bool FEW>
__global__ void __launch_bounds__(256) shade_estimate_kernel(
    const float* __restrict__ lights, const float* __restrict__ spheres, int n_sph,
    const float* __restrict__ boxes, int n_box, const float* __restrict__ pos,
    const float* __restrict__ nrm, int64_t n, const int32_t* __restrict__ idx,
    const float* __restrict__ pdf, float* __restrict__ estimate, float* __restrict__ accum,
    uint32_t count) {
  extern __shared__ float4 s_scene4[];
  const Occluders occ =
      stage_occluders<FEW>(spheres, n_sph, boxes, n_box, s_scene4, threadIdx.x, blockDim.x);
  __syncthreads();
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    float e = 0.0f;
    const int32_t s = idx[p];
    const float pr = pdf[p];
    if (s >= 0 && pr > 0.0f) {
      const float4 l = reinterpret_cast<const float4*>(lights)[s];
      const float px = pos[3 * p], py = pos[3 * p + 1], pz = pos[3 * p + 2];
      const float c = contribution(px, py, pz, nrm[3 * p], nrm[3 * p + 1], nrm[3 * p + 2], l.x,
                                   l.y, l.z, __fmul_rn(l.w, bits_f(kInvPiBits)));
      if (c > 0.0f && !segment_blocked<FEW>(px, py, pz, l.x, l.y, l.z, occ))
        e = __fdiv_rn(c, pr);
    }
    if (estimate) estimate[p] = e;
    if (accum) {
      const float a = accum[p];
      accum[p] = count <= 1u ? e : __fadd_rn(a, __fdiv_rn(__fsub_rn(e, a), (float)count));
    }
  }
}

// One light at a time for the whole warp (warp_segments_blocked), its
// contribution two lights per packed operation (exact_pair.cuh).  A warp whose
// pixels are not neighbours -- a light's vote keeps more than a quarter of the
// occluders -- takes segment_blocked from there on, so the votes cost it that
// many tests.
// 1920x1080 x 32 lights, 32 spheres + 32 boxes: 2.80 -> 0.756 ms; bound by
// instruction issue (9,900 a warp and 32 lights; 75% of the slots).  With the
// limit at an eighth 0.773, at a half, left only after every kept occluder's
// test, 0.760, and 4,096 pixels x 32 lights, 500 + 500, 1,009 us where a
// quarter takes 515 (every occluder tested: 654).
// kSmemLights: the lights (with I / pi) are staged after the occluders as
// pairs, in groups of four with zero lights past the last; otherwise they are
// read through the read-only cache and scaled here (the same rounding), for
// scenes whose lights do not fit on chip.
template <bool kSmemLights>
__global__ void __launch_bounds__(256, 3) exact_di_kernel(
    const float* __restrict__ lights, int L, const float* __restrict__ spheres, int n_sph,
    const float* __restrict__ boxes, int n_box, const float* __restrict__ pos,
    const float* __restrict__ nrm, int64_t n, float* __restrict__ di, float neg0) {
  extern __shared__ float4 s_scene4[];
  const int L4 = (L + 3) & ~3;
  const Occluders occ = stage_occluders(spheres, n_sph, boxes, n_box,
                                        s_scene4 + (kSmemLights ? L4 : 0), threadIdx.x, blockDim.x);
  bool lights_ok = true;
  if (kSmemLights) {
    for (int e = threadIdx.x; e < L4; e += blockDim.x) {
      float4 l = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < L) l = reinterpret_cast<const float4*>(lights)[e];
      l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
      xp::put_light(s_scene4, e, l);
      lights_ok = lights_ok && xp::light_ok(l);
    }
  }
  lights_ok = __syncthreads_and(lights_ok) != 0;
  const int limit = (2 * occ.n_pairs + occ.n_box) / 4 + 2;
  // whole warps walk the pixels: a lane past the end repeats the warp's first
  // pixel and writes nothing
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); p0 < n;
       p0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = p0 + (threadIdx.x & 31);
    const bool live = p < n;
    const int64_t pl = live ? p : p0;
    const float px = pos[3 * pl], py = pos[3 * pl + 1], pz = pos[3 * pl + 2];
    const float nx = nrm[3 * pl], ny = nrm[3 * pl + 1], nz = nrm[3 * pl + 2];
    xp::Pixel pp = xp::make_pixel(px, py, pz, nx, ny, nz, neg0, lights_ok);
    const bool pixel_ok = pp.ok;
    const WarpHull hull = warp_hull(px, py, pz);
    bool together = hull.scale <= 1e18f;   // not an infinite position among them
    float sum = 0.0f;
    for (int i0 = 0; i0 < L; i0 += 4) {
      float4 lt[4];
      float c[4];
      if (kSmemLights) {
        xp::staged_contributions<2>(pp, s_scene4 + i0, c);
#pragma unroll
        for (int q = 0; q < 4; ++q) lt[q] = xp::pair_light(s_scene4 + i0, q);
      } else {
        pp.ok = pixel_ok;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          lt[q] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (i0 + q < L) lt[q] = __ldg(reinterpret_cast<const float4*>(lights) + i0 + q);
          lt[q].w = __fmul_rn(lt[q].w, bits_f(kInvPiBits));
          pp.ok = pp.ok && xp::light_ok(lt[q]);
        }
        const float4 ab[4] = {make_float4(lt[0].x, lt[1].x, lt[0].y, lt[1].y),
                              make_float4(lt[0].z, lt[1].z, lt[0].w, lt[1].w),
                              make_float4(lt[2].x, lt[3].x, lt[2].y, lt[3].y),
                              make_float4(lt[2].z, lt[3].z, lt[2].w, lt[3].w)};
        xp::contributions<2>(pp, ab, c);
      }
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const float cq = q == 0 ? c[0] : q == 1 ? c[1] : q == 2 ? c[2] : c[3];
        const float4 l = q == 0 ? lt[0] : q == 1 ? lt[1] : q == 2 ? lt[2] : lt[3];
        const bool want = live && i0 + q < L && cq > 0.0f;
        if (!__any_sync(0xffffffffu, want)) continue;
        bool blocked = false;
        if (together)
          together = warp_segments_blocked(hull, want, px, py, pz, l.x, l.y, l.z, occ, limit, &blocked);
        if (!together && want) blocked = segment_blocked(px, py, pz, l.x, l.y, l.z, occ);
        if (want && !blocked) sum = __fadd_rn(sum, cq);
      }
    }
    if (live) di[p] = sum;
  }
}

// Few occluders: a light at a time for each pixel by itself.  The warp's vote,
// the packed contributions and 80 registers a thread cost more there than they
// save.  130,000 pixels x 32 lights, this kernel / the one above in us:
// no occluder 12 / 23, 4 spheres 35 / 55, 8 boxes 53 / 57, 6 + 6 78 / 74
// (random positions 78 / 99), 8 + 8 94 / 84 (96 / 111).
template <bool kSmemLights>
__global__ void __launch_bounds__(256) exact_di_few_kernel(
    const float* __restrict__ lights, int L, const float* __restrict__ spheres, int n_sph,
    const float* __restrict__ boxes, int n_box, const float* __restrict__ pos,
    const float* __restrict__ nrm, int64_t n, float* __restrict__ di, float) {
  extern __shared__ float4 s_scene4[];
  const Occluders occ = stage_occluders<true>(spheres, n_sph, boxes, n_box,
                                              s_scene4 + (kSmemLights ? (L + 3) & ~3 : 0),
                                              threadIdx.x, blockDim.x);
  if (kSmemLights) {
    for (int e = threadIdx.x; e < L; e += blockDim.x) {
      float4 l = reinterpret_cast<const float4*>(lights)[e];
      l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
      s_scene4[e] = l;
    }
  }
  __syncthreads();
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const float px = pos[3 * p], py = pos[3 * p + 1], pz = pos[3 * p + 2];
    const float nx = nrm[3 * p], ny = nrm[3 * p + 1], nz = nrm[3 * p + 2];
    float sum = 0.0f;
    for (int i = 0; i < L; ++i) {
      float4 l;
      if (kSmemLights) {
        l = s_scene4[i];
      } else {
        l = __ldg(reinterpret_cast<const float4*>(lights) + i);
        l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
      }
      const float c = contribution(px, py, pz, nx, ny, nz, l.x, l.y, l.z, l.w);
      if (c > 0.0f && !segment_blocked<true>(px, py, pz, l.x, l.y, l.z, occ)) sum = __fadd_rn(sum, c);
    }
    di[p] = sum;
  }
}

int grid_for(int64_t n, int num_sms) {
  const int64_t want = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms * 8;
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

}  // namespace

cudaError_t launch_shade_estimate(const nvc_scene* sc, const float* pos, const float* nrm,
                                  int64_t n, const int32_t* idx, const float* pdf,
                                  float* estimate, float* accum, uint32_t count, int num_sms,
                                  cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const size_t smem = occluder_bytes(sc->n_spheres, sc->n_boxes);
  auto kern = few_occluders(sc->n_spheres, sc->n_boxes) ? shade_estimate_kernel<true>
                                                        : shade_estimate_kernel<false>;
  const cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid_for(n, num_sms), 256, smem, s>>>(
      sc->lights, sc->spheres, sc->n_spheres, sc->boxes, sc->n_boxes, pos, nrm, n, idx, pdf,
      estimate, accum, count);
  return cudaGetLastError();
}

cudaError_t launch_exact_di(const nvc_scene* sc, const float* pos, const float* nrm, int64_t n,
                            float* di, int num_sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const size_t occ = occluder_bytes(sc->n_spheres, sc->n_boxes);
  const size_t lt = sizeof(float) * 4 * (((size_t)sc->n_lights + 3) & ~(size_t)3);
  const bool on_chip = occ + lt <= 227 * 1024;
  const size_t smem = on_chip ? occ + lt : occ;
  const bool few = sc->n_spheres + sc->n_boxes <= 12;
  auto kern = few ? (on_chip ? exact_di_few_kernel<true> : exact_di_few_kernel<false>)
                  : (on_chip ? exact_di_kernel<true> : exact_di_kernel<false>);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<grid_for(n, num_sms), 256, smem, s>>>(sc->lights, sc->n_lights, sc->spheres,
                                               sc->n_spheres, sc->boxes, sc->n_boxes, pos, nrm,
                                               n, di, -0.0f);
  return cudaGetLastError();
}

}  // namespace nvc
