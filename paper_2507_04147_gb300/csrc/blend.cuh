// blend.cuh -- device helpers shared by the compositing kernels and their backward: the test whether
// a Gaussian reaches a patch of pixels, and packed pairs of fp32 values.
#pragma once

#include <cuda_runtime.h>

namespace a3fr {

// Conservative box of the pixels where a Gaussian can reach alpha >= 1/255: the ellipse
// d^T conic d <= 2 ln(255 opacity) has half-extents k sqrt(cov_xx), k sqrt(cov_yy) with cov
// the inverse of the conic; one pixel of margin absorbs rounding.  Empty (never hit) when
// opacity < 1/255.  (x0, x1, y0, y1).
__device__ __forceinline__ float4 support_box(float u, float v, float ca, float cb, float cc, float op) {
  const float k2 = 2.0f * __logf(255.0f * op);
  if (!(k2 > 0.0f)) return make_float4(1e30f, -1e30f, 1e30f, -1e30f);
  const float det = ca * cc - cb * cb;
  const float ex = sqrtf(k2 * cc / det) + 1.0f, ey = sqrtf(k2 * ca / det) + 1.0f;
  if (!(ex < 1e6f) || !(ey < 1e6f)) return make_float4(-1e30f, 1e30f, -1e30f, 1e30f);
  return make_float4(u - ex, u + ex, v - ey, v + ey);
}

// A support box rounded outward to whole pixels in 16 bits (clamped to +-kBoxFar, which no
// pixel reaches): a superset of the float box, so the integer test rejects no more.
constexpr short kBoxFar = 30000;
__device__ __forceinline__ short4 int_box(float4 b) {
  auto lo = [](float v) { return (short)fminf(fmaxf(floorf(v), -(float)kBoxFar), (float)kBoxFar); };
  auto hi = [](float v) { return (short)fminf(fmaxf(ceilf(v), -(float)kBoxFar), (float)kBoxFar); };
  return make_short4(lo(b.x), hi(b.y), lo(b.z), hi(b.w));
}

// Whether a Gaussian can reach alpha >= 1/255 at some point of the rectangle [x0, x1] x
// [y0, y1] (pixel coordinates relative to its centre): the log2 falloff f = A x^2 + B x y +
// C y^2 (A, C < 0: concave) is largest at the centre if the rectangle holds it, else on an
// edge, where the best point along the edge is the clamped stationary point.  thr is the
// falloff alpha = 1/255 needs, lowered by a margin (0.01 in log2) far above the rounding
// of f, of the stationary points and of the kernel's own alpha, so a Gaussian it rejects
// has alpha < 1/255 at every pixel of the rectangle: rejecting it changes no output bit.
__device__ __forceinline__ bool falloff_reaches(float A, float B, float C, float thr, float x0, float x1,
                                                float y0, float y1) {
  if (!(A < 0.0f) || !(C < 0.0f) || !(4.0f * A * C > 1.0001f * B * B)) return true;   // not concave
  if (x0 <= 0.0f && x1 >= 0.0f && y0 <= 0.0f && y1 >= 0.0f) return thr <= 0.0f;
  const float ky = __fdividef(-B, 2.0f * C), kx = __fdividef(-B, 2.0f * A);
  auto f = [&](float x, float y) { return (A * x + B * y) * x + C * y * y; };
  const float ya = fminf(fmaxf(ky * x0, y0), y1), yb = fminf(fmaxf(ky * x1, y0), y1);
  const float xa = fminf(fmaxf(kx * y0, x0), x1), xb = fminf(fmaxf(kx * y1, x0), x1);
  const float best = fmaxf(fmaxf(f(x0, ya), f(x1, yb)), fmaxf(f(xa, y0), f(xb, y1)));
  return best >= thr;
}

// Two fp32 values in one 64-bit register pair, and the packed fp32 arithmetic of sm_100 and
// later (add / mul / fma .rn.f32x2: each half rounded exactly as the scalar instruction), so
// two pixels of a lane take one instruction where the arithmetic is the same for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// 1.0f where a >= b, else 0.0f (one instruction instead of a compare and a select)
__device__ __forceinline__ float ge_factor(float a, float b) {
  float r;
  asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// The sum of the halves.
__device__ __forceinline__ float f2_sum(f32x2 v) {
  float lo, hi;
  f2_unpack(v, lo, hi);
  return lo + hi;
}

}  // namespace a3fr
