// Clustered neural visibility cache (Section 3.6 of the paper): the lights
// are grouped by k-means, the network's outputs are the clusters' average
// visibilities, and a light is sampled in two steps -- a weighted reservoir
// over the clusters, then streaming resampled importance sampling (RIS)
// among a few members of the chosen cluster.
//
// k-means runs on the host in float64 (Lloyd's iterations from given seed
// lights).  On the device:
//   cluster_targets_kernel   training targets: for each (position, cluster)
//                            the binary visibility of one member drawn
//                            uniformly, so the network learns the average;
//   sample_sum_kernel        per pixel: c_hat_y = sum of the members'
//                            contributions, w_y = max(v_y, 0.001) c_hat_y,
//                            the integer reservoir over the clusters, then
//                            kRis uniform members of cluster y, one kept by
//                            the integer reservoir on their contributions,
//                            and its unbiased contribution weight
//                            W = (sum_j c_j / M) / (p(x) c(x)),
//                            p(x) = (w(y) / w_sum) / m_y;
//   sample_visibility_kernel the same with w_y = max(v_y, 0.001) alone.
// Every float32 result is rounded in a fixed order and every random choice
// is a fixed Philox word, so the kernels are reproducible bit for bit.
#include <vector>

#include "exact_pair.cuh"
#include "fused_common.cuh"
#include "nvc_internal.cuh"
#include "shadow.cuh"

namespace nvc {

namespace {

constexpr uint32_t kTagRis = 4;       // candidates in the chosen cluster and their pick
constexpr uint32_t kTagCluster = 5;   // a member light per cluster for the training targets
constexpr int kRis = 4;               // RIS candidates
constexpr int kMaxClusters = 32;

// Word i of the stream (id, frame, view, tag).
__device__ __forceinline__ uint32_t stream_word(uint32_t id, uint32_t frame, uint32_t view,
                                                uint32_t tag, int i, uint32_t k0, uint32_t k1) {
  const uint4 r = philox4x32_10(make_uint4(id, frame, view, ((uint32_t)(i >> 2) << 4) | tag), k0, k1);
  const int l = i & 3;
  return l == 0 ? r.x : l == 1 ? r.y : l == 2 ? r.z : r.w;
}

// Member of cluster y chosen by the word r: floor(r m_y / 2^32).
__device__ __forceinline__ int member_of(const int32_t* off, const int32_t* mem, int y, uint32_t r) {
  const uint32_t m = (uint32_t)(off[y + 1] - off[y]);
  return mem[off[y] + (int)(((uint64_t)r * m) >> 32)];
}

template <bool FEW>
__global__ void __launch_bounds__(256) cluster_targets_kernel(
    const float* __restrict__ lights, const float* __restrict__ spheres, int n_sph,
    const float* __restrict__ boxes, int n_box, const int32_t* __restrict__ off,
    const int32_t* __restrict__ mem, int k, const float* __restrict__ pos, int64_t n,
    uint32_t k0, uint32_t k1, uint32_t frame, float* __restrict__ target) {
  extern __shared__ float4 s_occ[];
  const Occluders occ =
      stage_occluders<FEW>(spheres, n_sph, boxes, n_box, s_occ, threadIdx.x, blockDim.x);
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int64_t b = t / k;
  const int y = (int)(t - b * k);
  float v = 0.0f;
  if (off[y + 1] > off[y]) {
    const int x = member_of(off, mem, y, stream_word((uint32_t)b, frame, 0u, kTagCluster, y, k0, k1));
    const float4 l = reinterpret_cast<const float4*>(lights)[x];
    const float px = pos[3 * b], py = pos[3 * b + 1], pz = pos[3 * b + 2];
    v = segment_blocked<FEW>(px, py, pz, l.x, l.y, l.z, occ) ? 0.0f : 1.0f;
  }
  target[t] = v;
}

// Integer reservoir over the first n of N float32 weights w (>= 0) with the
// words r_i: candidate i replaces the pick when r_i Q_i < q_i 2^32, Q_i the
// running sum of the quantised weights (< 2^32).  Loops run over N so the
// arrays stay in registers.
template <int N>
__device__ __forceinline__ int integer_reservoir(const float (&w)[N], int n, const uint32_t (&r)[N]) {
  float wmax = 0.0f;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < n) wmax = fmaxf(wmax, w[i]);
  if (!(wmax > 0.0f)) return -1;
  const int e = ilogbf(wmax);
  uint32_t Q = 0;
  int sel = -1;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (i < n) {
      const uint32_t q = quantize_weight(w[i], e);
      Q += q;
      if (q > 0u && __umulhi(r[i], Q) < q) sel = i;
    }
  }
  return sel;
}

// Integer reservoir over the k cluster weights wfn(y) with the words of
// stream (pixel, frame, view, kTagWrs), drawn four at a time as the scan
// reaches them: the same picks as integer_reservoir with r[y] = word y.  wfn
// is called with constants below kMaxClusters (weights may be registers).
template <typename WFn>
__device__ __forceinline__ int cluster_reservoir(WFn wfn, int k, uint32_t pixel, uint32_t frame,
                                                 uint32_t view, uint32_t k0, uint32_t k1) {
  float wmax = 0.0f;
#pragma unroll
  for (int y = 0; y < kMaxClusters; ++y)
    if (y < k) wmax = fmaxf(wmax, wfn(y));
  if (!(wmax > 0.0f)) return -1;
  const int e = ilogbf(wmax);
  uint32_t Q = 0;
  int sel = -1;
#pragma unroll
  for (int g = 0; g < kMaxClusters / 4; ++g) {
    if (4 * g < k) {
      const uint4 r4 = philox4x32_10(make_uint4(pixel, frame, view, ((uint32_t)g << 4) | kTagWrs), k0, k1);
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int y = 4 * g + l;
        if (y < k) {
          const float w = wfn(y);
          const uint32_t q = quantize_weight(w, e);
          Q += q;
          if (q > 0u && __umulhi(fz::pick_word(r4, l), Q) < q) sel = y;
        }
      }
    }
  }
  return sel;
}

// What both first steps share: the scene, the cluster table and the outputs.
struct ClusterArgs {
  const float* lights;
  int n_lights;
  const float* spheres;
  int n_sph;
  const float* boxes;
  int n_box;
  const int32_t* off;
  const int32_t* mem;
  int k;
  const float* vis;
  const float* pos;
  const float* nrm;
  int64_t n;
  int64_t pixel_offset;
  uint32_t k0, k1, frame, view;
  int32_t* light_out;
  float* weight_out;
  float* estimate;
  float neg0;               // -0.0f (exact_pair.cuh)
  int tile;                 // staged light slots (sum weights)
};

// Step 2 and the outputs of pixel p: streaming RIS among kRis uniform members
// of cluster y (y < 0: nothing contributes) with weight w_y of wsum, the
// unbiased contribution weight, and the one-ray estimate.  light(slot): the
// light at a place of the cluster table, I / pi in w.
template <bool FEW, typename LightFn>
__device__ __forceinline__ void finish_pixel(const ClusterArgs& a, int64_t p, int y, float w_y,
                                             float wsum, int base, uint32_t m_y, float px, float py,
                                             float pz, xp::Pixel pp, LightFn light,
                                             const Occluders& occ) {
  const uint32_t pixel = (uint32_t)(a.pixel_offset + p);
  int sel_light = -1;
  float W = 0.0f, cx = 0.0f;
  if (y >= 0) {
    const uint4 u = philox4x32_10(make_uint4(pixel, a.frame, a.view, (0u << 4) | kTagRis), a.k0, a.k1);
    const uint4 v = philox4x32_10(make_uint4(pixel, a.frame, a.view, (1u << 4) | kTagRis), a.k0, a.k1);
    const uint32_t ru[kRis] = {u.x, u.y, u.z, u.w};
    const uint32_t rr[kRis] = {v.x, v.y, v.z, v.w};
    int slot[kRis];
    float4 lt[kRis];
#pragma unroll
    for (int t = 0; t < kRis; ++t) {
      slot[t] = base + (int)(((uint64_t)ru[t] * m_y) >> 32);
      lt[t] = light(slot[t]);
      pp.ok = pp.ok && xp::light_ok(lt[t]);
    }
    const float4 ab[kRis] = {make_float4(lt[0].x, lt[1].x, lt[0].y, lt[1].y),
                             make_float4(lt[0].z, lt[1].z, lt[0].w, lt[1].w),
                             make_float4(lt[2].x, lt[3].x, lt[2].y, lt[3].y),
                             make_float4(lt[2].z, lt[3].z, lt[2].w, lt[3].w)};
    float cc[kRis];
    xp::contributions<kRis / 2>(pp, ab, cc);
    const int j = integer_reservoir(cc, kRis, rr);
    if (j >= 0) {
      float sum = 0.0f;
#pragma unroll
      for (int t = 0; t < kRis; ++t) sum = __fadd_rn(sum, cc[t]);
      float c_j = 0.0f;
      int s_j = 0;
#pragma unroll
      for (int t = 0; t < kRis; ++t)
        if (t == j) {
          c_j = cc[t];
          s_j = slot[t];
        }
      const float mean = __fdiv_rn(sum, (float)kRis);
      const float pr = __fdiv_rn(__fdiv_rn(w_y, wsum), (float)m_y);
      W = __fdiv_rn(mean, __fmul_rn(pr, c_j));
      sel_light = a.mem[s_j];
      cx = c_j;
    }
  }
  if (a.light_out) a.light_out[p] = sel_light;
  if (a.weight_out) a.weight_out[p] = W;
  if (a.estimate) {
    float e = 0.0f;
    if (sel_light >= 0) {
      const float4 l = reinterpret_cast<const float4*>(a.lights)[sel_light];
      if (!segment_blocked<FEW>(px, py, pz, l.x, l.y, l.z, occ)) e = __fmul_rn(cx, W);
    }
    a.estimate[p] = e;
  }
}

// A light of the cluster table from global memory, I / pi in w.
__device__ __forceinline__ float4 table_light(const ClusterArgs& a, int slot) {
  float4 l = __ldg(reinterpret_cast<const float4*>(a.lights) + a.mem[slot]);
  l.w = __fmul_rn(l.w, bits_f(kInvPiBits));
  return l;
}

// ---- first-step weights max(v, 0.001) alone ---------------------------------
// No light loop: a pixel's visibilities are loaded together (16-byte loads
// when the row allows) into the weights' registers.  Bound by the latency of
// its loads and its chain of random picks: 24 warps an SM at 80 registers, with
// quantize_weight as it is, a million pixels, k = 32, no occluders 104 -> 90 us,
// 32 + 32 152 -> 142; 28 and 32 warps 94 and 96 us, and exact multiplications
// with a branch for infinite weights, which pay where one thread walks more
// weights, 7% more.
template <bool FEW>
__global__ void __launch_bounds__(128, 6) sample_visibility_kernel(const __grid_constant__ ClusterArgs a,
                                                                 bool vis_vec4) {
  extern __shared__ float4 s_scene4[];
  int32_t* s_off = reinterpret_cast<int32_t*>(s_scene4);
  const Occluders occ = stage_occluders<FEW>(a.spheres, a.n_sph, a.boxes, a.n_box,
                                             s_scene4 + (kMaxClusters + 4) / 4, threadIdx.x,
                                             blockDim.x);
  const int k = a.k;
  for (int e = threadIdx.x; e <= k; e += blockDim.x) s_off[e] = a.off[e];
  __syncthreads();
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const float px = a.pos[3 * p], py = a.pos[3 * p + 1], pz = a.pos[3 * p + 2];
    const float nx = a.nrm[3 * p], ny = a.nrm[3 * p + 1], nz = a.nrm[3 * p + 2];
    float w[kMaxClusters];
    float wsum = 0.0f;
    const float* vrow = a.vis + p * k;
    if (vis_vec4) {
#pragma unroll
      for (int g = 0; g < kMaxClusters / 4; ++g) {
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (4 * g < k) v = __ldg(reinterpret_cast<const float4*>(vrow) + g);
        w[4 * g] = v.x;
        w[4 * g + 1] = v.y;
        w[4 * g + 2] = v.z;
        w[4 * g + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int t = 0; t < kMaxClusters; ++t) w[t] = t < k ? __ldg(vrow + t) : 0.0f;
    }
#pragma unroll
    for (int t = 0; t < kMaxClusters; ++t) {
      if (t < k) {
        w[t] = s_off[t + 1] > s_off[t] ? fmaxf(w[t], bits_f(kVisClampBits)) : 0.0f;
        wsum = __fadd_rn(wsum, w[t]);
      } else {
        w[t] = 0.0f;
      }
    }
    const int y = cluster_reservoir([&](int t) { return w[t]; }, k, (uint32_t)(a.pixel_offset + p),
                                    a.frame, a.view, a.k0, a.k1);
    float w_y = 0.0f;
#pragma unroll
    for (int t = 0; t < kMaxClusters; ++t)
      if (t == y) w_y = w[t];
    const int base = y < 0 ? 0 : s_off[y];
    finish_pixel<FEW>(a, p, y, w_y, wsum, base, y < 0 ? 0u : (uint32_t)(s_off[y + 1] - base), px, py, pz,
                 xp::make_pixel(px, py, pz, nx, ny, nz, a.neg0, true),
                 [&](int slot) { return table_light(a, slot); }, occ);
  }
}

// ---- first-step weights max(v, 0.001) x sum of the members' contributions ---
// The cost is one correctly rounded contribution per light and pixel, two
// lights per packed operation (exact_pair.cuh).  The lights are staged in
// cluster-table order as pairs, every cluster's run padded to an even count
// with a zero light (its contribution +0 leaves the sum as it is), so no pair
// straddles two clusters; more slots than a tile are walked tile by tile,
// staged together by the CTA, each thread carrying its pixel's running sum
// across tiles.  All threads of a CTA are at the same cluster and slot.  A
// pixel's weights lie in shared memory, [cluster][thread].
//
// Bound by the FMA pipe and its operand reads: a packed operation takes both
// halves' cycles (three distinct operands half as many again), 59 a pair by
// count, some 84 measured.  1920x1080 x 1024 lights, k = 32, with the shadow
// ray: 3.56 -> 2.54 ms a launch.  Two pairs in flight at 24 warps an SM was
// the fastest of 1, 2 and 4 pairs at 16, 24 and 32 warps (within 5%).
constexpr int kLightTile = 1024;
constexpr int kSumThreads = 256;

// Light slots [t0, t0 + tn) of the padded table into s_lt; s_out[y] is set
// where a light of cluster y is outside the packed contribution's bounds.
__device__ __forceinline__ void stage_slots(const ClusterArgs& a, const int32_t* s_off,
                                            const int32_t* s_pad, float4* s_lt, int32_t* s_out, int t0,
                                            int tn) {
  for (int e = threadIdx.x; e < tn; e += blockDim.x) {
    int lo = 0, hi = a.k - 1;   // the cluster whose padded run holds slot t0 + e
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_pad[mid] <= t0 + e) lo = mid; else hi = mid - 1;
    }
    const int at = s_off[lo] + (t0 + e - s_pad[lo]);
    const bool pad = at >= s_off[lo + 1];
    float4 l = table_light(a, pad ? s_off[lo] : at);
    if (pad) l.w = 0.0f;
    xp::put_light(s_lt, e, l);
    if (!xp::light_ok(l)) s_out[lo] = 1;
  }
}

template <bool FEW>
__global__ void __launch_bounds__(kSumThreads, 3)
    sample_sum_kernel(const __grid_constant__ ClusterArgs a) {
  extern __shared__ float4 s_scene4[];
  float4* s_lt = s_scene4;
  float* s_w = reinterpret_cast<float*>(s_lt + a.tile) + threadIdx.x;
  int32_t* s_off = reinterpret_cast<int32_t*>(s_lt + a.tile) + kMaxClusters * kSumThreads;
  int32_t* s_pad = s_off + kMaxClusters + 4;
  int32_t* s_out = s_pad + kMaxClusters + 4;
  const Occluders occ = stage_occluders<FEW>(a.spheres, a.n_sph, a.boxes, a.n_box,
                                             s_out + kMaxClusters + 4, threadIdx.x, blockDim.x);
  const int k = a.k;
  if (threadIdx.x < kMaxClusters) s_out[threadIdx.x] = 0;
  for (int e = threadIdx.x; e <= k; e += blockDim.x) s_off[e] = a.off[e];
  __syncthreads();
  if (threadIdx.x == 0) {
    int at = 0;
    for (int y = 0; y < k; ++y) {
      s_pad[y] = at;
      at += (s_off[y + 1] - s_off[y] + 1) & ~1;
    }
    s_pad[k] = at;
  }
  __syncthreads();
  const int n_slots = s_pad[k];
  const bool whole = n_slots <= a.tile;
  if (whole) {
    stage_slots(a, s_off, s_pad, s_lt, s_out, 0, n_slots);
    __syncthreads();
  }
  for (int64_t b = (int64_t)blockIdx.x * kSumThreads; b < a.n; b += (int64_t)gridDim.x * kSumThreads) {
    const int64_t p = b + threadIdx.x;
    const bool live = p < a.n;
    const int64_t pl = live ? p : 0;
    const float px = a.pos[3 * pl], py = a.pos[3 * pl + 1], pz = a.pos[3 * pl + 2];
    const float nx = a.nrm[3 * pl], ny = a.nrm[3 * pl + 1], nz = a.nrm[3 * pl + 2];
    xp::Pixel pp = xp::make_pixel(px, py, pz, nx, ny, nz, a.neg0, true);
    const bool pixel_ok = pp.ok;
    const float* vrow = a.vis + pl * k;
    float ch = 0.0f;
    int y = 0;
    for (int t0 = 0; t0 < n_slots; t0 += a.tile) {
      const int t1 = min(t0 + a.tile, n_slots);
      if (!whole) {
        __syncthreads();   // the previous tile is read by every thread
        stage_slots(a, s_off, s_pad, s_lt, s_out, t0, t1 - t0);
        __syncthreads();
      }
      int cur = t0;
      while (y < k) {
        const int pad_end = s_pad[y + 1], end = min(pad_end, t1);
        // the run's bounds are checked once; a run that breaks them is summed
        // again, light by light, from where it began, and one that holds a
        // light out of bounds only so (one light of 1024 out of bounds, k = 32,
        // a million pixels: 3,030 -> 1,300 us; none 1,210)
        pp.ok = pixel_ok && s_out[y] == 0;
        const float ch0 = ch;
        float dmin = 1.0f;
        uint32_t tmin = 0xFFFFFFFFu;
        if (pp.ok) {
#pragma unroll 2
          for (int i = cur - t0; i < end - t0; i += 2) {
            const float2 c = xp::contribution2(pp, s_lt[i], s_lt[i + 1], dmin, tmin);
            ch = __fadd_rn(__fadd_rn(ch, c.x), c.y);
          }
        }
        if (!xp::in_bounds(pp, dmin, tmin)) {
          ch = ch0;
#pragma unroll 1
          for (int i = cur - t0; i < end - t0; ++i) {
            const float4 l = xp::pair_light(s_lt, i);
            ch = __fadd_rn(ch, contribution(px, py, pz, nx, ny, nz, l.x, l.y, l.z, l.w));
          }
        }
        cur = end;
        if (pad_end > t1) break;
        s_w[y * kSumThreads] = __fmul_rn(fmaxf(__ldg(vrow + y), bits_f(kVisClampBits)), ch);
        ch = 0.0f;
        ++y;
      }
    }
    if (!live) continue;   // the last batch: no barrier follows
    float wsum = 0.0f;
    for (int t = 0; t < k; ++t) wsum = __fadd_rn(wsum, s_w[t * kSumThreads]);
    y = cluster_reservoir([&](int t) { return s_w[t * kSumThreads]; }, k,
                          (uint32_t)(a.pixel_offset + p), a.frame, a.view, a.k0, a.k1);
    const int base = y < 0 ? 0 : s_off[y];
    pp.ok = pixel_ok;
    finish_pixel<FEW>(a, p, y, y < 0 ? 0.0f : s_w[y * kSumThreads], wsum, base,
                 y < 0 ? 0u : (uint32_t)(s_off[y + 1] - base), px, py, pz, pp,
                 [&](int slot) {
                   return whole ? xp::pair_light(s_lt, s_pad[y] + slot - base) : table_light(a, slot);
                 },
                 occ);
  }
}

// ---- temporal resampling of the cache's reservoirs (ReSTIR, Section 4.2) -----
constexpr uint32_t kTagTemporal = 6;   // the pick between current and previous reservoir
constexpr int kTemporalMCap = 20;      // the previous reservoir counts at most 20x the new one

// p_hat(y) = c_y at the pixel, the correctly rounded float32 contribution
// (0 for y outside [0, n_lights)).
__device__ __forceinline__ float target_of(const float* lights, int n_lights, int y, float px,
                                           float py, float pz, float nx, float ny, float nz) {
  if (y < 0 || y >= n_lights) return 0.0f;
  const float4 l = __ldg(reinterpret_cast<const float4*>(lights) + y);
  return contribution(px, py, pz, nx, ny, nz, l.x, l.y, l.z, __fmul_rn(l.w, bits_f(kInvPiBits)));
}

template <bool FEW>
__global__ void __launch_bounds__(256) temporal_merge_kernel(
    const float* __restrict__ lights, int n_lights, const float* __restrict__ spheres, int n_sph,
    const float* __restrict__ boxes, int n_box, const float* __restrict__ pos,
    const float* __restrict__ nrm, int64_t n, int64_t pixel_offset, uint32_t k0, uint32_t k1,
    uint32_t frame, uint32_t view, const int32_t* __restrict__ cur_light,
    const float* __restrict__ cur_W, const int32_t* __restrict__ prev_light,
    const float* __restrict__ prev_W, const int32_t* __restrict__ prev_M,
    int32_t* __restrict__ light_out, float* __restrict__ W_out, int32_t* __restrict__ M_out,
    float* __restrict__ estimate) {
  extern __shared__ float4 s_occ[];
  Occluders occ = no_occluders(s_occ);
  if (estimate) {
    occ = stage_occluders<FEW>(spheres, n_sph, boxes, n_box, s_occ, threadIdx.x, blockDim.x);
    __syncthreads();
  }
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const float px = pos[3 * p], py = pos[3 * p + 1], pz = pos[3 * p + 2];
    const float nx = nrm[3 * p], ny = nrm[3 * p + 1], nz = nrm[3 * p + 2];
    int yc = cur_light[p];
    int yp = prev_light ? prev_light[p] : -1;
    int Mp = prev_M ? prev_M[p] : 0;
    Mp = Mp < 0 ? 0 : (Mp > kTemporalMCap ? kTemporalMCap : Mp);   // min(M_p, 20 M_c), M_c = 1
    if (yc >= n_lights) yc = -1;
    if (yp >= n_lights || Mp == 0) yp = -1;
    const float pc = target_of(lights, n_lights, yc, px, py, pz, nx, ny, nz);
    const float pp = target_of(lights, n_lights, yp, px, py, pz, nx, ny, nz);
    float w[2];
    w[0] = yc >= 0 ? __fmul_rn(__fmul_rn(1.0f, pc), cur_W[p]) : 0.0f;
    w[1] = yp >= 0 ? __fmul_rn(__fmul_rn((float)Mp, pp), prev_W[p]) : 0.0f;
    const uint4 r4 = philox4x32_10(make_uint4((uint32_t)(pixel_offset + p), frame, view, kTagTemporal),
                                   k0, k1);
    const uint32_t r[2] = {r4.x, r4.y};
    const int j = integer_reservoir(w, 2, r);
    const int y = j == 0 ? yc : j == 1 ? yp : -1;
    const int M = 1 + Mp;
    float W = 0.0f;
    if (y >= 0) W = __fdiv_rn(__fadd_rn(w[0], w[1]), __fmul_rn((float)M, j == 0 ? pc : pp));
    if (light_out) light_out[p] = y;
    if (W_out) W_out[p] = W;
    if (M_out) M_out[p] = M;
    if (estimate) {
      float e = 0.0f;
      if (y >= 0) {
        const float4 l = __ldg(reinterpret_cast<const float4*>(lights) + y);
        if (!segment_blocked<FEW>(px, py, pz, l.x, l.y, l.z, occ))
          e = __fmul_rn(j == 0 ? pc : pp, W);
      }
      estimate[p] = e;
    }
  }
}

}  // namespace

cudaError_t launch_temporal_merge(const nvc_scene* sc, const float* pos, const float* nrm,
                                  int64_t n, int64_t pixel_offset, uint64_t seed, uint32_t frame,
                                  uint32_t view, const int32_t* cur_light, const float* cur_W,
                                  const int32_t* prev_light, const float* prev_W,
                                  const int32_t* prev_M, int32_t* light, float* W, int32_t* M,
                                  float* estimate, int num_sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const size_t smem = estimate ? occluder_bytes(sc->n_spheres, sc->n_boxes) : 0;
  auto kern = few_occluders(sc->n_spheres, sc->n_boxes) ? temporal_merge_kernel<true>
                                                        : temporal_merge_kernel<false>;
  const cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  const int64_t want = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms * 8;
  kern<<<(unsigned)(want < cap ? want : cap), 256, smem, s>>>(
      sc->lights, sc->n_lights, sc->spheres, sc->n_spheres, sc->boxes, sc->n_boxes, pos, nrm, n,
      pixel_offset, (uint32_t)seed, (uint32_t)(seed >> 32), frame, view, cur_light, cur_W,
      prev_light, prev_W, prev_M, light, W, M, estimate);
  return cudaGetLastError();
}

cudaError_t launch_cluster_targets(const nvc_scene* sc, const nvc_clusters* cl, const float* pos,
                                   int64_t n, uint64_t seed, uint32_t frame, float* target,
                                   cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t total = n * cl->k;
  const size_t smem = occluder_bytes(sc->n_spheres, sc->n_boxes);
  auto kern = few_occluders(sc->n_spheres, sc->n_boxes) ? cluster_targets_kernel<true>
                                                        : cluster_targets_kernel<false>;
  const cudaError_t e = allow_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)((total + 255) / 256), 256, smem, s>>>(
      sc->lights, sc->spheres, sc->n_spheres, sc->boxes, sc->n_boxes, cl->offsets, cl->members,
      cl->k, pos, n, (uint32_t)seed, (uint32_t)(seed >> 32), frame, target);
  return cudaGetLastError();
}

// Light slots the sum kernel stages at once: all of them (each cluster may
// add one to be even) up to a tile.
static int light_slots(const nvc_scene* sc, const nvc_clusters* cl) {
  const int64_t all = ((int64_t)sc->n_lights + cl->k + 3) & ~(int64_t)3;
  return (int)(all < kLightTile ? all : kLightTile);
}

size_t sample_clustered_smem(const nvc_scene* sc, const nvc_clusters* cl) {
  const size_t occ =
      occluder_bytes(sc->n_spheres, sc->n_boxes) + sizeof(float4) * ((kMaxClusters + 4) / 4);
  if (cl->weights == NVC_CLUSTER_WEIGHT_VISIBILITY) return occ;   // no light loop
  return occ + sizeof(float4) * (2 * ((kMaxClusters + 4) / 4) + light_slots(sc, cl)) +
         sizeof(float) * kMaxClusters * kSumThreads;
}

cudaError_t launch_sample_clustered(const nvc_scene* sc, const nvc_clusters* cl, const float* vis,
                                    const float* pos, const float* nrm, int64_t n,
                                    int64_t pixel_offset, uint64_t seed, uint32_t frame,
                                    uint32_t view, int32_t* light, float* weight, float* estimate,
                                    int num_sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const size_t smem = sample_clustered_smem(sc, cl);
  const ClusterArgs a{sc->lights, sc->n_lights, sc->spheres, sc->n_spheres, sc->boxes, sc->n_boxes,
                      cl->offsets, cl->members, cl->k, vis, pos, nrm, n, pixel_offset,
                      (uint32_t)seed, (uint32_t)(seed >> 32), frame, view, light, weight, estimate,
                      -0.0f, light_slots(sc, cl)};
  const bool sum = cl->weights != NVC_CLUSTER_WEIGHT_VISIBILITY;
  const bool few = few_occluders(sc->n_spheres, sc->n_boxes);
  auto sum_kern = few ? sample_sum_kernel<true> : sample_sum_kernel<false>;
  auto vis_kern = few ? sample_visibility_kernel<true> : sample_visibility_kernel<false>;
  const void* kern = sum ? (const void*)sum_kern : (const void*)vis_kern;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // one wave of resident CTAs strides over the pixels
  const int threads = sum ? kSumThreads : 128;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm == 0) return cudaErrorInvalidConfiguration;
  const int64_t want = (n + threads - 1) / threads, cap = (int64_t)num_sms * per_sm;
  const int grid = (int)(want < cap ? want : cap);
  if (sum) {
    sum_kern<<<grid, threads, smem, s>>>(a);
  } else {
    // 16-byte loads of a pixel's visibilities need rows of a multiple of 4
    // floats on a 16-byte aligned base
    vis_kern<<<grid, threads, smem, s>>>(
        a, (cl->k & 3) == 0 && (reinterpret_cast<uintptr_t>(vis) & 15) == 0);
  }
  return cudaGetLastError();
}

// Lloyd's k-means in float64, the same steps as the oracle: squared
// distances (dx^2 + dy^2) + dz^2, the first nearest centroid, centroids the
// mean of their members summed in light order, empty clusters unchanged.
void kmeans_host(const float* lights, int n, const int32_t* init, int k, int iters,
                 int32_t* assign, double* centroids_out) {
  std::vector<double> C(3 * (size_t)k);
  for (int y = 0; y < k; ++y)
    for (int d = 0; d < 3; ++d) C[3 * y + d] = (double)lights[4 * (size_t)init[y] + d];
  auto assign_all = [&]() {
    for (int i = 0; i < n; ++i) {
      double best = 0.0;
      int arg = 0;
      for (int y = 0; y < k; ++y) {
        const double dx = (double)lights[4 * (size_t)i] - C[3 * y];
        const double dy = (double)lights[4 * (size_t)i + 1] - C[3 * y + 1];
        const double dz = (double)lights[4 * (size_t)i + 2] - C[3 * y + 2];
        const double d2 = (dx * dx + dy * dy) + dz * dz;
        if (y == 0 || d2 < best) {
          best = d2;
          arg = y;
        }
      }
      assign[i] = arg;
    }
  };
  std::vector<double> S(3 * (size_t)k);
  std::vector<int> cnt((size_t)k);
  for (int it = 0; it < iters; ++it) {
    assign_all();
    std::fill(S.begin(), S.end(), 0.0);
    std::fill(cnt.begin(), cnt.end(), 0);
    for (int i = 0; i < n; ++i) {
      const int y = assign[i];
      for (int d = 0; d < 3; ++d) S[3 * y + d] = S[3 * y + d] + (double)lights[4 * (size_t)i + d];
      ++cnt[y];
    }
    for (int y = 0; y < k; ++y)
      if (cnt[y] > 0)
        for (int d = 0; d < 3; ++d) C[3 * y + d] = S[3 * y + d] / (double)cnt[y];
  }
  assign_all();
  if (centroids_out)
    for (size_t i = 0; i < C.size(); ++i) centroids_out[i] = C[i];
}

}  // namespace nvc
