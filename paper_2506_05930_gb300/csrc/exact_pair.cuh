// The correctly rounded light contribution (nvc_internal.cuh's
// contribution()) for two lights per packed float32x2 operation.
//
// contribution() spends some 50 instructions a light, most of them in the
// library's correctly rounded square root and division.  Both are formed here
// by Markstein's corrections (P. Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34(1),
// 1990) from the hardware's approximate reciprocal square root and
// reciprocal, with fused multiply-adds that packed operations do for two
// lights at once:
//   s = g + (x - g g) r / 2,          g = x r, r ~ 1 / sqrt(x);
//   y = y0 + (1 - b y0) y0, y0 ~ 1/b; q = a y;  q + (a - b q) y.
// Checked on the device against the library's (test_gpu_exact_arithmetic.py
// repeats it, the quotients in part): s for every float of
// [2^-20, 2^64), the quotient for all 2^46 pairs of mantissas; both scale
// with powers of two while nothing leaves the normal range, which the bounds
// below guarantee.  A group of lights outside them takes contribution().
// About 25 packed operations, 4 approximations and 6 others a pair.
#pragma once
#include "nvc_internal.cuh"

namespace nvc {
namespace xp {

// Lights in pairs, coordinate-major: float4 {x, x', y, y'}, {z, z', I/pi,
// I'/pi} at s[2 pair], s[2 pair + 1].
__device__ __forceinline__ float4 pair_light(const float4* s, int i) {
  const float* q = reinterpret_cast<const float*>(s) + (i >> 1) * 8 + (i & 1);
  return make_float4(q[0], q[2], q[4], q[6]);
}

__device__ __forceinline__ void put_light(float4* s, int i, float4 l) {
  float* q = reinterpret_cast<float*>(s) + (i >> 1) * 8 + (i & 1);
  q[0] = l.x;
  q[2] = l.y;
  q[4] = l.z;
  q[6] = l.w;
}

constexpr float kCoordMax = 262144.0f;       // 2^18: positions, normals, light positions
constexpr float kIntensityMax = 1048576.0f;  // 2^20: I/pi
constexpr uint32_t kNumMinBits = 0x21800000u;  // 2^-60

// Whether a light (I/pi in w) is inside the bounds (no NaN passes).
__device__ __forceinline__ bool light_ok(float4 l) {
  return fabsf(l.x) <= kCoordMax && fabsf(l.y) <= kCoordMax && fabsf(l.z) <= kCoordMax &&
         l.w >= 0.0f && l.w <= kIntensityMax;
}

// A pixel as the packed operations read it.  neg0: the host's -0.0f; a
// product taken as fma(a, b, -0) is the rounded product, and with an addend
// the compiler does not know it cannot be fused into the sum that follows.
struct Pixel {
  float2 npx, npy, npz, nx, ny, nz, neg0;
  bool ok;
};

__device__ __forceinline__ Pixel make_pixel(float px, float py, float pz, float nx, float ny,
                                            float nz, float neg0, bool lights_ok) {
  Pixel p;
  p.npx = make_float2(-px, -px);
  p.npy = make_float2(-py, -py);
  p.npz = make_float2(-pz, -pz);
  p.nx = make_float2(nx, nx);
  p.ny = make_float2(ny, ny);
  p.nz = make_float2(nz, nz);
  p.neg0 = make_float2(neg0, neg0);
  p.ok = lights_ok && fabsf(px) <= kCoordMax && fabsf(py) <= kCoordMax && fabsf(pz) <= kCoordMax &&
         fabsf(nx) <= kCoordMax && fabsf(ny) <= kCoordMax && fabsf(nz) <= kCoordMax;
  return p;
}

// sqrt(x) of both halves, correctly rounded for x of [2^-20, 2^64); nx = -x.
__device__ __forceinline__ float2 sqrt2_rn(float2 x, float2 nx) {
  float2 r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(x.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(x.y));
  const float2 g = __fmul2_rn(x, r), h = __fmul2_rn(r, make_float2(-0.5f, -0.5f));
  return __ffma2_rn(__ffma2_rn(g, g, nx), h, g);
}

// -(a / nb) of both halves, correctly rounded while nothing leaves the normal
// range.
__device__ __forceinline__ float2 div2_rn(float2 a, float2 nb) {
  float2 y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(-nb.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(-nb.y));
  y = __ffma2_rn(__ffma2_rn(nb, y, make_float2(1.0f, 1.0f)), y, y);
  const float2 q = __fmul2_rn(a, y);
  return __ffma2_rn(__ffma2_rn(nb, q, a), y, q);
}

// Two contributions; dmin and tmin collect what the bounds check: the least
// |d|^2, and the least positive numerator (bits - 1, so that zero and
// negative ones, whose contribution is 0, come out largest).
__device__ __forceinline__ float2 contribution2(const Pixel& p, float4 A, float4 B, float& dmin,
                                                uint32_t& tmin) {
  const float2 dx = __fadd2_rn(make_float2(A.x, A.y), p.npx);
  const float2 dy = __fadd2_rn(make_float2(A.z, A.w), p.npy);
  const float2 dz = __fadd2_rn(make_float2(B.x, B.y), p.npz);
  const float2 d2 = __fadd2_rn(__fadd2_rn(__ffma2_rn(dx, dx, p.neg0), __ffma2_rn(dy, dy, p.neg0)),
                               __ffma2_rn(dz, dz, p.neg0));
  const float2 ndl = __fadd2_rn(__fadd2_rn(__ffma2_rn(p.nx, dx, p.neg0), __ffma2_rn(p.ny, dy, p.neg0)),
                                __ffma2_rn(p.nz, dz, p.neg0));
  const float2 nd2 = __fmul2_rn(d2, make_float2(-1.0f, -1.0f));
  const float2 nden = __fmul2_rn(sqrt2_rn(d2, nd2), nd2);         // -sqrt(d2) d2, d2 >= 1e-6
  const float2 num = __fmul2_rn(make_float2(B.z, B.w), ndl);
  const float2 c = div2_rn(num, nden);                            // num / den
  dmin = fminf(fminf(dmin, d2.x), d2.y);
  tmin = min(min(tmin, __float_as_uint(num.x) - 1u), __float_as_uint(num.y) - 1u);
  return make_float2(fmaxf(c.x, 0.0f), fmaxf(c.y, 0.0f));   // n.d <= 0 (or NaN) gives 0
}

__device__ __forceinline__ bool in_bounds(const Pixel& p, float dmin, uint32_t tmin) {
  return p.ok && dmin >= bits_f(kD2MinBits) && tmin >= kNumMinBits - 1u;
}

// The contributions of 2 P lights given as P pairs (A, B of each in turn).
template <int P>
__device__ __forceinline__ void contributions(const Pixel& p, const float4 (&ab)[2 * P],
                                              float (&c)[2 * P]) {
  float dmin = 1.0f;
  uint32_t tmin = 0xFFFFFFFFu;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    const float2 v = contribution2(p, ab[2 * k], ab[2 * k + 1], dmin, tmin);
    c[2 * k] = v.x;
    c[2 * k + 1] = v.y;
  }
  if (!in_bounds(p, dmin, tmin)) {
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const float4 A = ab[2 * k], B = ab[2 * k + 1];
      c[2 * k] = contribution(-p.npx.x, -p.npy.x, -p.npz.x, p.nx.x, p.ny.x, p.nz.x, A.x, A.z, B.x, B.z);
      c[2 * k + 1] =
          contribution(-p.npx.x, -p.npy.x, -p.npz.x, p.nx.x, p.ny.x, p.nz.x, A.y, A.w, B.y, B.w);
    }
  }
}

// The same from staged pairs s[0 .. 2 P - 1].
template <int P>
__device__ __forceinline__ void staged_contributions(const Pixel& p, const float4* s, float (&c)[2 * P]) {
  float4 ab[2 * P];
#pragma unroll
  for (int k = 0; k < 2 * P; ++k) ab[k] = s[k];
  contributions<P>(p, ab, c);
}

}  // namespace xp
}  // namespace nvc
