// tail_solve.cuh -- the line solve by two geometric tails and the H1 factors of
// complex float, shared by the on-chip 2D stepper (resident.cu) and the tiled
// sweeps (tails.cu).  resident.cu describes the method.
#pragma once

#include "sweep_common.cuh"

namespace rotgp {

// ---------------------------------------------------------------- line solve
// The weights of one line.
struct line_w {
  float2 al, be, g2, gc;
};
// k (v + r): the next value of a tail
__device__ __forceinline__ float2 tail(float2 k, float2 v, float2 r) {
  const float x = v.x + r.x, y = v.y + r.y;
  return make_float2(fmaf(k.x, x, -(k.y * y)), fmaf(k.x, y, k.y * x));
}
// gc psi + g2 (f + b)
__device__ __forceinline__ float2 change(const line_w& k, float2 psi, float2 f, float2 b) {
  const float x = f.x + b.x, y = f.y + b.y;
  return make_float2(
      fmaf(k.g2.x, x, fmaf(-k.g2.y, y, fmaf(k.gc.x, psi.x, -(k.gc.y * psi.y)))),
      fmaf(k.g2.x, y, fmaf(k.g2.y, x, fmaf(k.gc.x, psi.y, k.gc.y * psi.x))));
}
// e^u - 1 to float accuracy relative to u: the Taylor series below 1/4, where
// the steps of practice lie, and exp beyond.
__device__ __forceinline__ float exp_m1(float u) {
  float p = fmaf(u, 1.f / 5040.f, 1.f / 720.f);
  p = fmaf(u, p, 1.f / 120.f);
  p = fmaf(u, p, 1.f / 24.f);
  p = fmaf(u, p, 1.f / 6.f);
  p = fmaf(u, p, 0.5f);
  p = fmaf(u * u, p, u);
  return fabsf(u) < 0.25f ? p : __expf(u) - 1.f;
}

// cos(t) - 1 and sin(t) as rot_t (sweep_common.cuh) gives them: the Taylor
// series below 1/2, rot_t beyond (not inlined: the argument reduction is
// hundreds of instructions).
static __device__ __noinline__ float2 rot_far(float t) {
  float c1, s1;
  rot_t(t, &c1, &s1);
  return make_float2(c1, s1);
}
__device__ __forceinline__ float2 rot_near(float t) {
  const float q = t * t;
  float c = fmaf(q, 1.f / 40320.f, -1.f / 720.f);
  c = fmaf(q, c, 1.f / 24.f);
  c = fmaf(q, c, -0.5f);
  float s = fmaf(q, 1.f / 362880.f, -1.f / 5040.f);
  s = fmaf(q, s, 1.f / 120.f);
  s = fmaf(q, s, -1.f / 6.f);
  return make_float2(q * c, fmaf(t * q, s, t));
}

// H1 of a point v = s psi (rounded) in real time: the advanced value rounded,
// and what the rounding left out.
__device__ __forceinline__ void rotate_split(float2 v, float t, float2* w, float2* rest) {
  const float2 k = fabsf(t) < 0.5f ? rot_near(t) : rot_far(t);
  const float2 dl = make_float2(fmaf(k.x, v.x, k.y * v.y), fmaf(k.x, v.y, -(k.y * v.x)));
  const float2 a = make_float2(__fadd_rn(v.x, dl.x), __fadd_rn(v.y, dl.y));
  *w = a;
  *rest = make_float2(__fsub_rn(dl.x, __fsub_rn(a.x, v.x)), __fsub_rn(dl.y, __fsub_rn(a.y, v.y)));
}

}  // namespace rotgp
