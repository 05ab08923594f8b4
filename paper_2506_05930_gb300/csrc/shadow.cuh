// Binary shadow rays against the analytic occluders (Section 3.4 targets,
// the shading pass of Section 3.1 and the all-lights reference of Section
// 4.4 share them).  The segment x + t d, t in [1e-4, 1 - 1e-4], d = l - x,
// is blocked by a sphere whose centre is strictly closer than its radius to
// the segment, or by a box the segment meets (closed slab test).  The
// arithmetic is correctly rounded float32 in a fixed order, so the binary
// decision is reproducible operation by operation.
#pragma once
#include "nvc_internal.cuh"

namespace nvc {

// ---- the occluders as the tests read them -----------------------------------
// Kernels stage the scene's occluders in shared memory in this layout:
//   sphere pairs, 32 bytes each: float4 {cx_a, cx_b, cy_a, cy_b}, float4
//   {cz_a, cz_b, r_a^2, r_b^2} (r^2 = fl(r r)); an odd count's last slot is
//   a sphere with r^2 = -1, which blocks nothing;
//   box pairs, 48 bytes each: per axis float4 {c_a, c_b, h_a, h_b}, centre and
//   half extent, the latter rounded up by 2^-16 of the box's coordinates: for
//   the tests that only drop boxes (near_boxes, hull_meets_box).  The exact
//   slab test reads the box itself from the scene's array.
// The pairs are held against a segment two occluders at a time (near_spheres,
// near_boxes), and what stands is tested exactly one by one.
// FEW (few_occluders): every test is exact, and the boxes are staged as they
// are, 24 bytes each: (lo_x, hi_x), (lo_y, hi_y), (lo_z, hi_z).
struct Occluders {
  const float4* sph;   // 2 float4 per sphere pair
  int n_pairs;
  const float4* box;   // 3 float4 per box pair; FEW: 3 float2 per box
  int n_box;
  const float* boxes;  // the scene's boxes, lo and hi (global memory)
};

// Whether a scene's rays take the FEW kernels.  Dropping occluders by pairs
// first costs a ray some 40 operations and its kernel 16 registers a thread
// (48 against 32: 40 warps an SM against 64), which few exact tests do not pay
// back; a sphere's test is about three times a box's.  130,000 points x 32
// lights, FEW / other in us: 4 spheres 32.8 / 45.2, 4 boxes 32.8 / 49.2, 8 + 8
// 77.3 / 84.0, 12 + 12 102.6 / 100.4, 16 + 16 129 / 117.
inline bool few_occluders(int n_sph, int n_box) { return 3 * n_sph + n_box <= 36; }

__host__ __device__ __forceinline__ size_t occluder_bytes(int n_sph, int n_box) {
  return 32 * (size_t)((n_sph + 1) / 2) + 48 * (size_t)((n_box + 1) / 2);
}

// Stages the occluders at dst (16-byte aligned; occluder_bytes(...) long),
// threads tid of nthreads sharing the work; the caller synchronises.
template <bool FEW = false>
__device__ __forceinline__ Occluders stage_occluders(const float* __restrict__ spheres, int n_sph,
                                                     const float* __restrict__ boxes, int n_box,
                                                     void* dst, int tid, int nthreads) {
  Occluders o;
  float* f = static_cast<float*>(dst);
  o.sph = reinterpret_cast<const float4*>(dst);
  o.n_pairs = (n_sph + 1) / 2;
  for (int e = tid; e < 2 * o.n_pairs; e += nthreads) {
    const int pair = e >> 1, lane = e & 1;
    float4 sp = make_float4(0.0f, 0.0f, 0.0f, -1.0f);   // r^2 = -1: blocks nothing
    if (e < n_sph) {
      sp = reinterpret_cast<const float4*>(spheres)[e];
      sp.w = __fmul_rn(sp.w, sp.w);
    }
    float* q = f + 8 * pair + lane;
    q[0] = sp.x;
    q[2] = sp.y;
    q[4] = sp.z;
    q[6] = sp.w;
  }
  float* b = f + 8 * o.n_pairs;
  if constexpr (FEW) {
    for (int e = tid; e < n_box; e += nthreads) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        b[6 * e + 2 * a] = boxes[6 * e + a];
        b[6 * e + 2 * a + 1] = boxes[6 * e + 3 + a];
      }
    }
  } else {
    for (int e = tid; e < ((n_box + 1) & ~1); e += nthreads) {
      float* q = b + 12 * (e >> 1) + (e & 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        float lo = 0.0f, hi = 0.0f;   // an odd count's last slot: never read as a box
        if (e < n_box) {
          lo = boxes[6 * e + a];
          hi = boxes[6 * e + 3 + a];
        }
        q[4 * a] = 0.5f * lo + 0.5f * hi;
        q[4 * a + 2] = fabsf(0.5f * hi - 0.5f * lo) + 0x1p-16f * (fabsf(lo) + fabsf(hi));
      }
    }
  }
  o.box = reinterpret_cast<const float4*>(b);
  o.n_box = n_box;
  o.boxes = boxes;
  return o;
}

// No occluders yet (kernels that stage them only when they need them).
__device__ __forceinline__ Occluders no_occluders(const void* at) {
  Occluders o;
  o.sph = o.box = reinterpret_cast<const float4*>(at);
  o.n_pairs = o.n_box = 0;
  o.boxes = nullptr;
  return o;
}

// ---- the tests ----------------------------------------------------------------
// The divisions are taken once per (position, light): 1/|d|^2 for the
// spheres' closest-point parameter and 1/d per axis for the boxes' slabs;
// each occluder then costs multiplications only.  Sphere (c, r): the
// segment's closest point q = x + t_c d, t_c = clamp(((c - x).d) / |d|^2,
// t0, t1), blocks when |c - q|^2 < r^2.

// One sphere of a staged pair (lane 0 or 1), in scalar correctly rounded
// operations: the compiler fuses a packed multiply into a following packed
// add (one rounding instead of two) even when both carry .rn, so products
// that feed sums stay scalar here.
__device__ __forceinline__ bool sphere_lane_blocks(float px, float py, float pz, float dx,
                                                   float dy, float dz, float inv_dd, float cx,
                                                   float cy, float cz, float r2) {
  const float t0 = bits_f(kSegT0Bits), t1 = bits_f(kSegT1Bits);
  const float ox = __fsub_rn(cx, px), oy = __fsub_rn(cy, py), oz = __fsub_rn(cz, pz);
  float tc = __fmul_rn(dot3_rn(ox, oy, oz, dx, dy, dz), inv_dd);
  tc = fminf(fmaxf(tc, t0), t1);
  const float ex = __fsub_rn(cx, __fadd_rn(px, __fmul_rn(tc, dx)));
  const float ey = __fsub_rn(cy, __fadd_rn(py, __fmul_rn(tc, dy)));
  const float ez = __fsub_rn(cz, __fadd_rn(pz, __fmul_rn(tc, dz)));
  return dot3_rn(ex, ey, ez, ex, ey, ez) < r2;
}

// Closed slab test of one box when no component of d is zero: the entry and
// exit parameters (lo - x) / d and (hi - x) / d of every axis, two per
// packed operation; blocked when max(t0, nearer planes) <= min(t1, farther).
__device__ __forceinline__ bool box_blocks_oblique(float2 px, float2 py, float2 pz, float2 ix,
                                                   float2 iy, float2 iz, const float2* b) {
  const float2 tx = fmul2_rn(fsub2(b[0], px), ix);
  const float2 ty = fmul2_rn(fsub2(b[1], py), iy);
  const float2 tz = fmul2_rn(fsub2(b[2], pz), iz);
  const float tmin = fmaxf(fmaxf(fmaxf(bits_f(kSegT0Bits), fminf(tx.x, tx.y)), fminf(ty.x, ty.y)),
                           fminf(tz.x, tz.y));
  const float tmax = fminf(fminf(fminf(bits_f(kSegT1Bits), fmaxf(tx.x, tx.y)), fmaxf(ty.x, ty.y)),
                           fmaxf(tz.x, tz.y));
  return tmin <= tmax;
}

// The same test with any component of d zero: that axis only checks that x
// lies between its planes.
__device__ __forceinline__ void slab(float xa, float da, float inv_da, float lo, float hi,
                                     float& tmin, float& tmax, bool& miss) {
  if (da == 0.0f) {
    miss = miss || xa < lo || xa > hi;
    return;
  }
  const float ta = __fmul_rn(__fsub_rn(lo, xa), inv_da);
  const float tb = __fmul_rn(__fsub_rn(hi, xa), inv_da);
  tmin = fmaxf(tmin, fminf(ta, tb));
  tmax = fminf(tmax, fmaxf(ta, tb));
}

__device__ __forceinline__ bool box_blocks_general(float px, float py, float pz, float dx, float dy,
                                                   float dz, float ix, float iy, float iz,
                                                   const float2* b) {
  float tmin = bits_f(kSegT0Bits), tmax = bits_f(kSegT1Bits);
  bool miss = false;
  slab(px, dx, ix, b[0].x, b[0].y, tmin, tmax, miss);
  slab(py, dy, iy, b[1].x, b[1].y, tmin, tmax, miss);
  slab(pz, dz, iz, b[2].x, b[2].y, tmin, tmax, miss);
  return !miss && tmin <= tmax;
}

// fl(1 / x): Markstein's correction of the hardware's approximate reciprocal
// (two, the first of the reciprocal itself; exact_pair.cuh names the method,
// and its check of every mantissa pair covers 1 / x), the library's division
// outside [2^-60, 2^60].
__device__ __forceinline__ float rcp_rn(float x) {
  const float ax = fabsf(x);
  if (!(ax >= 0x1p-60f && ax <= 0x1p60f)) return __fdiv_rn(1.0f, x);
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  y = __fmaf_rn(__fmaf_rn(-x, y, 1.0f), y, y);
  return __fmaf_rn(__fmaf_rn(-x, y, 1.0f), y, y);
}

// A segment from x to a light, with the reciprocals the tests share.
struct Segment {
  float px, py, pz, dx, dy, dz;
  float inv_dd, ix, iy, iz;
  bool oblique;   // no component of d is zero
};

__device__ __forceinline__ Segment make_segment(float px, float py, float pz, float lx, float ly,
                                                float lz) {
  Segment g;
  g.px = px;
  g.py = py;
  g.pz = pz;
  g.dx = __fsub_rn(lx, px);
  g.dy = __fsub_rn(ly, py);
  g.dz = __fsub_rn(lz, pz);
  const float dd = dot3_rn(g.dx, g.dy, g.dz, g.dx, g.dy, g.dz);
  // a zero-length segment (light on the point): t stays at t0
  g.inv_dd = dd > 0.0f ? rcp_rn(dd) : 0.0f;
  g.ix = g.dx != 0.0f ? rcp_rn(g.dx) : 0.0f;
  g.iy = g.dy != 0.0f ? rcp_rn(g.dy) : 0.0f;
  g.iz = g.dz != 0.0f ? rcp_rn(g.dz) : 0.0f;
  g.oblique = g.dx != 0.0f && g.dy != 0.0f && g.dz != 0.0f;
  return g;
}

// Staged sphere i (of 2 n_pairs slots) and box i against the segment.
__device__ __forceinline__ bool sphere_blocks(const Segment& g, const Occluders& occ, int i) {
  const float* q = reinterpret_cast<const float*>(occ.sph) + (i >> 1) * 8 + (i & 1);
  return sphere_lane_blocks(g.px, g.py, g.pz, g.dx, g.dy, g.dz, g.inv_dd, q[0], q[2], q[4], q[6]);
}

__device__ __forceinline__ bool box_blocks(const Segment& g, const Occluders& occ, int i) {
  const float* q = occ.boxes + 6 * i;
  const float2 b[3] = {make_float2(__ldg(q), __ldg(q + 3)), make_float2(__ldg(q + 1), __ldg(q + 4)),
                       make_float2(__ldg(q + 2), __ldg(q + 5))};
  if (!g.oblique)
    return box_blocks_general(g.px, g.py, g.pz, g.dx, g.dy, g.dz, g.ix, g.iy, g.iz, b);
  return box_blocks_oblique(make_float2(g.px, g.px), make_float2(g.py, g.py),
                            make_float2(g.pz, g.pz), make_float2(g.ix, g.ix),
                            make_float2(g.iy, g.iy), make_float2(g.iz, g.iz), b);
}

// The spheres of pairs [k0, k1), at most 16 pairs, that may block the segment:
// bit 2 (k - k0) + lane.  The exact test of a sphere is some 26 operations
// that must stay scalar and unfused; this one, 13 packed ones a pair, asks
// only whether the centre's distance from the segment's line clears the
// radius by more than any rounding:
//   oo - (o.d)^2 / dd > r^2,  o = c - x,
// with oo scaled down by 2^-15, r^2 up by 2^-16 and 2^-15 (|x|^2 + |l|^2) added
// to it (`slack`).  The exact test's error is a few 2^-24 of the coordinates
// x, l, c, so of the squares at most 2^-18 (|x|^2 + |l|^2 + |c|^2 + r^2), and
// |c|^2 <= 2 |x|^2 + 2 oo; this one's own is some 20 x 2^-24 of oo.  What is
// not a number is kept.  (1080p temporal merge with its ray, 32 spheres + 32
// boxes: 145 -> 127 us.)
__device__ __forceinline__ uint32_t near_spheres(const Segment& g, const Occluders& occ, int k0, int k1,
                                                 float slack) {
  const float2 npx = make_float2(-g.px, -g.px), npy = make_float2(-g.py, -g.py),
               npz = make_float2(-g.pz, -g.pz);
  const float2 dx = make_float2(g.dx, g.dx), dy = make_float2(g.dy, g.dy), dz = make_float2(g.dz, g.dz);
  const float2 ninv = make_float2(-g.inv_dd, -g.inv_dd);
  uint32_t m = 0, bit = 1;
#pragma unroll 4
  for (int k = k0; k < k1; ++k, bit <<= 2) {
    const float4 A = occ.sph[2 * k], B = occ.sph[2 * k + 1];
    const float2 ox = __fadd2_rn(make_float2(A.x, A.y), npx);
    const float2 oy = __fadd2_rn(make_float2(A.z, A.w), npy);
    const float2 oz = __fadd2_rn(make_float2(B.x, B.y), npz);
    const float2 od = __ffma2_rn(ox, dx, __ffma2_rn(oy, dy, __fmul2_rn(oz, dz)));
    const float2 oo = __ffma2_rn(ox, ox, __ffma2_rn(oy, oy, __fmul2_rn(oz, oz)));
    const float2 c = __ffma2_rn(
        __fmul2_rn(od, ninv), od,
        __ffma2_rn(oo, make_float2(1.0f - 0x1p-15f, 1.0f - 0x1p-15f),
                   __fmul2_rn(make_float2(B.z, B.w), make_float2(-1.0f - 0x1p-16f, -1.0f - 0x1p-16f))));
    if (!(c.x > slack)) m |= bit;
    if (!(c.y > slack)) m |= bit << 1;
  }
  return m;
}

// The boxes of pairs [k0, k1), at most 16 pairs, that may block an oblique
// segment: bit 2 (k - k0) + lane.  The slab test's two planes per axis are
// (c -+ h - x) / d, so from centre and half extent near and far come without
// a minimum and a maximum -- three packed operations an axis for two boxes --
// and only the largest near and smallest far are left to the ALU, which the
// exact test keeps busy with 13 operations a box.  A box is dropped when near
// exceeds far by more than `slack`, 2^-16 of the coordinates of x and the
// light times the largest |1 / d|: the exact test's planes and these ones are
// off by some 4 x 2^-24 of (|x| + |c| + h) / |d|, the box's share of which is
// in h.  What is not a number is kept.  (1080p frame 494 -> 489 us, temporal
// merge with its ray 127 -> 114 us, each with 32 boxes.)
__device__ __forceinline__ uint32_t near_boxes(const Segment& g, const Occluders& occ, int k0, int k1,
                                               float slack) {
  const float2 ix = make_float2(g.ix, g.ix), iy = make_float2(g.iy, g.iy), iz = make_float2(g.iz, g.iz);
  const float2 ax = make_float2(fabsf(g.ix), fabsf(g.ix)), ay = make_float2(fabsf(g.iy), fabsf(g.iy)),
               az = make_float2(fabsf(g.iz), fabsf(g.iz));
  const float2 bx = make_float2(-ax.x, -ax.x), by = make_float2(-ay.x, -ay.x),
               bz = make_float2(-az.x, -az.x);
  const float sx = -g.px * g.ix, sy = -g.py * g.iy, sz = -g.pz * g.iz;
  const float t0 = bits_f(kSegT0Bits), t1 = bits_f(kSegT1Bits);
  uint32_t m = 0, bit = 1;
#pragma unroll 4
  for (int k = k0; k < k1; ++k, bit <<= 2) {
    const float4 X = occ.box[3 * k], Y = occ.box[3 * k + 1], Z = occ.box[3 * k + 2];
    const float2 hx = make_float2(X.z, X.w), hy = make_float2(Y.z, Y.w), hz = make_float2(Z.z, Z.w);
    const float2 mx = __ffma2_rn(make_float2(X.x, X.y), ix, make_float2(sx, sx));
    const float2 my = __ffma2_rn(make_float2(Y.x, Y.y), iy, make_float2(sy, sy));
    const float2 mz = __ffma2_rn(make_float2(Z.x, Z.y), iz, make_float2(sz, sz));
    const float2 nx = __ffma2_rn(hx, bx, mx), ny = __ffma2_rn(hy, by, my), nz = __ffma2_rn(hz, bz, mz);
    const float2 fx = __ffma2_rn(hx, ax, mx), fy = __ffma2_rn(hy, ay, my), fz = __ffma2_rn(hz, az, mz);
    const float na = fmaxf(fmaxf(fmaxf(nx.x, ny.x), nz.x), t0);
    const float fa = fminf(fminf(fminf(fx.x, fy.x), fz.x), t1);
    const float nb = fmaxf(fmaxf(fmaxf(nx.y, ny.y), nz.y), t0);
    const float fb = fminf(fminf(fminf(fx.y, fy.y), fz.y), t1);
    if (!(na - fa > slack)) m |= bit;
    if (!(nb - fb > slack)) m |= bit << 1;
  }
  return 2 * k1 > occ.n_box ? m & ~(1u << (occ.n_box - 2 * k0)) : m;   // not the padding slot
}

// segment_blocked of the FEW kernels: every occluder tested exactly, with the
// reciprocals that the scene's kinds of occluders need.
__device__ __forceinline__ bool segment_blocked_few(float px, float py, float pz, float lx, float ly,
                                                    float lz, const Occluders& occ) {
  const float dx = __fsub_rn(lx, px), dy = __fsub_rn(ly, py), dz = __fsub_rn(lz, pz);
  bool blocked = false;
  if (occ.n_pairs > 0) {
    const float dd = dot3_rn(dx, dy, dz, dx, dy, dz);
    // a zero-length segment (light on the point): t stays at t0
    const float inv_dd = dd > 0.0f ? rcp_rn(dd) : 0.0f;
    for (int k = 0; k < occ.n_pairs && !blocked; ++k) {
      const float4 A = occ.sph[2 * k], B = occ.sph[2 * k + 1];
      blocked = sphere_lane_blocks(px, py, pz, dx, dy, dz, inv_dd, A.x, A.z, B.x, B.z) ||
                sphere_lane_blocks(px, py, pz, dx, dy, dz, inv_dd, A.y, A.w, B.y, B.w);
    }
  }
  if (occ.n_box > 0 && !blocked) {
    const float2* b = reinterpret_cast<const float2*>(occ.box);
    const float ix = dx != 0.0f ? rcp_rn(dx) : 0.0f;
    const float iy = dy != 0.0f ? rcp_rn(dy) : 0.0f;
    const float iz = dz != 0.0f ? rcp_rn(dz) : 0.0f;
    if (dx != 0.0f && dy != 0.0f && dz != 0.0f) {
      const float2 px2 = make_float2(px, px), py2 = make_float2(py, py), pz2 = make_float2(pz, pz);
      const float2 ix2 = make_float2(ix, ix), iy2 = make_float2(iy, iy), iz2 = make_float2(iz, iz);
      for (int k = 0; k < occ.n_box && !blocked; ++k)
        blocked = box_blocks_oblique(px2, py2, pz2, ix2, iy2, iz2, b + 3 * k);
    } else {
      for (int k = 0; k < occ.n_box && !blocked; ++k)
        blocked = box_blocks_general(px, py, pz, dx, dy, dz, ix, iy, iz, b + 3 * k);
    }
  }
  return blocked;
}

// Whether the segment from (px, py, pz) to the light at (lx, ly, lz) is
// blocked by one of the staged occluders (staged with the same FEW): those
// that near_spheres and near_boxes keep are tested exactly.
template <bool FEW = false>
__device__ __forceinline__ bool segment_blocked(float px, float py, float pz, float lx, float ly,
                                                float lz, const Occluders& occ) {
  if constexpr (FEW) return segment_blocked_few(px, py, pz, lx, ly, lz, occ);
  const Segment g = make_segment(px, py, pz, lx, ly, lz);
  const float slack = 0x1p-15f * (px * px + py * py + pz * pz + lx * lx + ly * ly + lz * lz);
  bool blocked = false;
  for (int k0 = 0; k0 < occ.n_pairs; k0 += 16) {
    uint32_t m = near_spheres(g, occ, k0, min(k0 + 16, occ.n_pairs), slack);
    for (; m && !blocked; m &= m - 1) blocked = sphere_blocks(g, occ, 2 * k0 + __ffs(m) - 1);
    if (blocked) return true;
  }
  if (g.oblique) {
    const float far = 0x1p-16f *
                      (fmaxf(fmaxf(fabsf(px), fabsf(py)), fabsf(pz)) +
                       fmaxf(fmaxf(fabsf(lx), fabsf(ly)), fabsf(lz))) *
                      fmaxf(fmaxf(fabsf(g.ix), fabsf(g.iy)), fabsf(g.iz));
    const int n = (occ.n_box + 1) >> 1;
    for (int k0 = 0; k0 < n; k0 += 16) {
      uint32_t m = near_boxes(g, occ, k0, min(k0 + 16, n), far);
      for (; m && !blocked; m &= m - 1) blocked = box_blocks(g, occ, 2 * k0 + __ffs(m) - 1);
      if (blocked) return true;
    }
  } else {
    for (int k = 0; k < occ.n_box && !blocked; ++k) blocked = box_blocks(g, occ, k);
  }
  return blocked;
}

// ---- a warp's segments together ------------------------------------------------
// 32 neighbouring pixels looking at one light sweep a thin volume that most
// occluders are nowhere near.  Each lane holds a different occluder against
// that volume -- the pixels' bounding box moved along the segment from its
// centre to the light -- and only the occluders whose vote stands are tested
// exactly, by all lanes, each against its own segment.
//
// The vote never drops an occluder that an exact test would call blocking:
// every segment lies in the swept box, so the occluder is held against it
// grown by 2^-16 of the largest coordinate involved, 16 times and more what
// the exact tests' roundings (some 2^-20 of it) and the vote's own can add
// up to; and it is written so that anything not a number stands.
struct WarpHull {
  float cx, cy, cz;   // centre and half extents of the 32 positions
  float hx, hy, hz;
  float rad;          // |half extents|, rounded up
  float scale;        // largest coordinate magnitude
};

__device__ __forceinline__ WarpHull warp_hull(float px, float py, float pz) {
  float lo[3] = {px, py, pz}, hi[3] = {px, py, pz};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
      hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
    }
  WarpHull w;
  w.cx = 0.5f * (lo[0] + hi[0]);
  w.cy = 0.5f * (lo[1] + hi[1]);
  w.cz = 0.5f * (lo[2] + hi[2]);
  w.hx = 0.5f * (hi[0] - lo[0]);
  w.hy = 0.5f * (hi[1] - lo[1]);
  w.hz = 0.5f * (hi[2] - lo[2]);
  w.rad = 1.0001f * sqrtf(w.hx * w.hx + w.hy * w.hy + w.hz * w.hz);
  w.scale = fmaxf(fmaxf(fabsf(w.cx) + w.hx, fabsf(w.cy) + w.hy), fabsf(w.cz) + w.hz);
  return w;
}

// Whether the lane's segments' volume may meet staged sphere i / box i.
struct HullRay {
  float dx, dy, dz;      // light - centre
  float inv_dd, ix, iy, iz;
  float scale;
};

__device__ __forceinline__ HullRay hull_ray(const WarpHull& w, float lx, float ly, float lz) {
  HullRay r;
  r.dx = lx - w.cx;
  r.dy = ly - w.cy;
  r.dz = lz - w.cz;
  const float dd = r.dx * r.dx + r.dy * r.dy + r.dz * r.dz;
  r.inv_dd = dd > 0.0f ? __fdividef(1.0f, dd) : 0.0f;
  // a component of zero: as good as zero, but with a finite reciprocal
  r.ix = __fdividef(1.0f, copysignf(fmaxf(fabsf(r.dx), 1e-20f), r.dx));
  r.iy = __fdividef(1.0f, copysignf(fmaxf(fabsf(r.dy), 1e-20f), r.dy));
  r.iz = __fdividef(1.0f, copysignf(fmaxf(fabsf(r.dz), 1e-20f), r.dz));
  r.scale = w.scale + fmaxf(fmaxf(fabsf(lx), fabsf(ly)), fabsf(lz));
  return r;
}

__device__ __forceinline__ bool hull_meets_sphere(const WarpHull& w, const HullRay& r,
                                                  const Occluders& occ, int i) {
  const float* q = reinterpret_cast<const float*>(occ.sph) + (i >> 1) * 8 + (i & 1);
  const float sx = q[0], sy = q[2], sz = q[4], r2 = q[6];
  const float ox = sx - w.cx, oy = sy - w.cy, oz = sz - w.cz;
  const float t = fminf(fmaxf((ox * r.dx + oy * r.dy + oz * r.dz) * r.inv_dd, 0.0f), 1.0f);
  const float ex = ox - t * r.dx, ey = oy - t * r.dy, ez = oz - t * r.dz;
  const float m = 0x1p-16f * (r.scale + fmaxf(fmaxf(fabsf(sx), fabsf(sy)), fabsf(sz)));
  const float reach = 1.0001f * sqrtf(r2) + w.rad + m;
  return r2 >= 0.0f && !(ex * ex + ey * ey + ez * ez > reach * reach);
}

__device__ __forceinline__ bool hull_meets_box(const WarpHull& w, const HullRay& r,
                                               const Occluders& occ, int i) {
  const float* q = reinterpret_cast<const float*>(occ.box + 3 * (i >> 1)) + (i & 1);
  const float m = 0x1p-16f * r.scale;   // the box's own share is in its half extents
  const float ax = fabsf(r.ix), ay = fabsf(r.iy), az = fabsf(r.iz);
  const float mx = (q[0] - w.cx) * r.ix, kx = (q[2] + w.hx + m) * ax;
  const float my = (q[4] - w.cy) * r.iy, ky = (q[6] + w.hy + m) * ay;
  const float mz = (q[8] - w.cz) * r.iz, kz = (q[10] + w.hz + m) * az;
  const float tmin = fmaxf(fmaxf(mx - kx, my - ky), fmaxf(mz - kz, 0.0f));
  const float tmax = fminf(fminf(mx + kx, my + ky), fminf(mz + kz, 1.0f));
  return !(tmin > tmax);
}

// segment_blocked for a whole warp looking at one light: *blocked is the
// answer of the lanes with `want`.  Gives up, with false in every lane, after
// `limit` exact tests.
__device__ __forceinline__ bool warp_segments_blocked(const WarpHull& w, bool want, float px, float py,
                                                      float pz, float lx, float ly, float lz,
                                                      const Occluders& occ, int limit, bool* blocked) {
  const int lane = threadIdx.x & 31;
  const HullRay r = hull_ray(w, lx, ly, lz);
  const Segment g = make_segment(px, py, pz, lx, ly, lz);
  bool open = want;
  *blocked = want;   // until the last occluder is past with lanes still open
  for (int b = 0; b < 2 * occ.n_pairs; b += 32) {
    const bool near = b + lane < 2 * occ.n_pairs && hull_meets_sphere(w, r, occ, b + lane);
    for (unsigned m = __ballot_sync(0xffffffffu, near); m; m &= m - 1) {
      if (--limit < 0) return false;
      open = open && !sphere_blocks(g, occ, b + __ffs(m) - 1);
      if (!__any_sync(0xffffffffu, open)) return true;
    }
  }
  for (int b = 0; b < occ.n_box; b += 32) {
    const bool near = b + lane < occ.n_box && hull_meets_box(w, r, occ, b + lane);
    for (unsigned m = __ballot_sync(0xffffffffu, near); m; m &= m - 1) {
      if (--limit < 0) return false;
      open = open && !box_blocks(g, occ, b + __ffs(m) - 1);
      if (!__any_sync(0xffffffffu, open)) return true;
    }
  }
  *blocked = want && !open;
  return true;
}

// ---- training positions (Section 3.4) ------------------------------------------
// Samples [0, n_world) are uniform in the world box (stream tag 1); the rest
// copy G-buffer pixel floor(r * n_screen / 2^32) (stream tag 2).
struct PosGen {
  float3 lo, ext;
  const float* screen;
  int64_t n_screen, n_world;
  uint32_t k0, k1, frame;
};

__device__ __forceinline__ float3 training_position(int64_t j, const PosGen& g) {
  if (j < g.n_world) {
    const uint4 r = philox4x32_10(make_uint4((uint32_t)j, g.frame, 0u, kTagWorld), g.k0, g.k1);
    return make_float3(__fadd_rn(g.lo.x, __fmul_rn(uniform24(r.x), g.ext.x)),
                       __fadd_rn(g.lo.y, __fmul_rn(uniform24(r.y), g.ext.y)),
                       __fadd_rn(g.lo.z, __fmul_rn(uniform24(r.z), g.ext.z)));
  }
  const uint32_t s = (uint32_t)(j - g.n_world);
  const uint4 r = philox4x32_10(make_uint4(s, g.frame, 0u, kTagScreen), g.k0, g.k1);
  const int64_t pix = (int64_t)(((uint64_t)r.x * (uint64_t)g.n_screen) >> 32);
  return make_float3(g.screen[3 * pix], g.screen[3 * pix + 1], g.screen[3 * pix + 2]);
}

// The generator of a training batch (train.cu): n_world = -1 for the
// default split ceil(batch / 2); every position is world space without
// screen positions.
PosGen pos_gen(const nvc_scene* sc, const float* screen_pos, int64_t n_screen, int64_t batch,
               uint64_t seed, uint32_t frame, int64_t n_world);

}  // namespace nvc
