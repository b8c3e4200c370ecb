// ep_lanes.cuh -- the columns of one thread of a marching sweep kernel: two
// adjacent FP32 columns as a float2 (packed arithmetic, one instruction per
// pair), or one FP64 column; the return scale.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace ep {

template <typename V>
struct Splat;
template <>
struct Splat<float2> {
  static __device__ __forceinline__ float2 of(float s) { return make_float2(s, s); }
};
template <>
struct Splat<double> {
  static __device__ __forceinline__ double of(double s) { return s; }
};

__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }

// value of the column left / right of each column, W threads per row (a row's
// first column has no left neighbour and gets an arbitrary value, the last no
// right one)
template <int W>
__device__ __forceinline__ float2 xm(float2 v) { return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1, W), v.x); }
template <int W>
__device__ __forceinline__ float2 xp(float2 v) { return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1, W)); }
template <int W>
__device__ __forceinline__ double xm(double v) { return __shfl_up_sync(0xffffffffu, v, 1, W); }
template <int W>
__device__ __forceinline__ double xp(double v) { return __shfl_down_sync(0xffffffffu, v, 1, W); }

// column E of a value
template <int E>
__device__ __forceinline__ float el(float2 v) { return E == 0 ? v.x : v.y; }
template <int E>
__device__ __forceinline__ double el(double v) { return v; }

// centre scale min(1, Y / sqrt(J2)).  FP32: compare squares, and only where the return
// acts (most cells stay elastic) form the quotient from the reciprocal square root r: J2 r
// and its residual give the root as a sum t + d, and one Newton step on the quotient s = Y r
// takes its residual Y - s (t + d) with fused multiply-adds.  The result is the rounded
// quotient but for near-ties (0.5 ulp; a rounded root and a division make 1.5): an error of the
// scale acts on the same cells in every iteration (95^3 with a per-cell modulus, error against
// 64 bits after 200 of them, median of 16 inputs over that of sqrt and division: 0.99, without
// the residuals 1.01; 55.8 -> 56.5 us an iteration, 67 with sqrt and division).  FP64: below
// Y^2 by more than the rounding of both, sqrt(J2) > Y cannot hold and the scale is 1 without
// the root.
__device__ __forceinline__ float scale_of(float J2, float Y) {
  Y = Y > 0.f ? Y : 0.f;
  if (!(J2 > Y * Y)) return 1.f;
  const float r = rsqrtf(J2), t = J2 * r, d = fmaf(-t, t, J2) * (0.5f * r), s = Y * r;
  const float q = fmaf(fmaf(-s, d, fmaf(-s, t, Y)), r, s);
  return !(J2 < INFINITY) ? s : q > 1.f ? 1.f : q;   // s = 0 where the invariant overflows
}
__device__ __forceinline__ double scale_of(double J2, double Y) {
  Y = Y > 0.0 ? Y : 0.0;
  if (J2 < Y * Y * (1.0 - 1e-15)) return 1.0;
  const double sj = sqrt(J2);
  return sj > Y ? Y / sj : 1.0;
}
// both columns in packed arithmetic where either yields (a warp's neighbours mostly yield
// together), each with the result of its own scale_of
__device__ __forceinline__ float2 vscale(float2 J2, float2 Y) {
  Y = make_float2(Y.x > 0.f ? Y.x : 0.f, Y.y > 0.f ? Y.y : 0.f);
  const float2 Y2 = vmul(Y, Y);
  const bool ax = J2.x > Y2.x, ay = J2.y > Y2.y;
  float2 out = make_float2(1.f, 1.f);
  if (ax || ay) {
    const float2 r = make_float2(rsqrtf(J2.x), rsqrtf(J2.y)), m1 = make_float2(-1.f, -1.f);
    const float2 t = vmul(J2, r), d = vmul(vfma(vmul(t, m1), t, J2), vmul(r, make_float2(0.5f, 0.5f)));
    const float2 s = vmul(Y, r), n = vmul(s, m1), q = vfma(vfma(n, d, vfma(n, t, Y)), r, s);
    if (ax) out.x = !(J2.x < INFINITY) ? s.x : q.x > 1.f ? 1.f : q.x;
    if (ay) out.y = !(J2.y < INFINITY) ? s.y : q.y > 1.f ? 1.f : q.y;
  }
  return out;
}
__device__ __forceinline__ double vscale(double J2, double Y) { return scale_of(J2, Y); }

// a return scale (0 .. 1, or NaN) below one; the FP64 one without the FP64 pipe
__device__ __forceinline__ bool below_one(float s) { return s < 1.f; }
__device__ __forceinline__ bool below_one(double s) { return (unsigned)__double2hiint(s) < 0x3ff00000u; }

}  // namespace ep
