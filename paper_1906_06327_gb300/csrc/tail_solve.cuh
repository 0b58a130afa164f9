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
// H1 of a point psi in imaginary time, (1 + m1) e^u psi.  Where u is small, as in
// the steps of practice, psi + (m1 + (1 + m1) (e^u - 1)) psi with a Taylor series:
// one rounding of psi.  From 1/4 on the product itself: formed as a change of
// psi, a factor below 1e-7 came out as 0 and one of 1e-5 right to 1% (64 x 48 with u
// down to -10: points off by up to 11%, now 2e-6).  Both factors are formed and
// one taken: a branch made a 4096^2 step 3% slower.
__device__ __forceinline__ float2 damp(float2 psi, float u, float m1) {
  float q = fmaf(u, 1.f / 5040.f, 1.f / 720.f);
  q = fmaf(u, q, 1.f / 120.f);
  q = fmaf(u, q, 1.f / 24.f);
  q = fmaf(u, q, 1.f / 6.f);
  q = fmaf(u, q, 0.5f);
  q = fmaf(u * u, q, u);
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(u * 1.4426950408889634f));
  const bool small = fabsf(u) < 0.25f;
  const float f = small ? fmaf(m1, q, q) + m1 : fmaf(m1, e, e), b = small ? 1.f : 0.f;
  return make_float2(fmaf(f, psi.x, b * psi.x), fmaf(f, psi.y, b * psi.y));
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
