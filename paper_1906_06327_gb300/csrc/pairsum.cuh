// pairsum.cuh -- sums for the read-only reductions: running sums of a thread
// (Kahan) and their combination over a block (Knuth's two-sum), in float pairs for
// complex float (hi + lo, 48 bits) and in double for complex double.  Over 8 grids
// from 128^2 to 2048 x 1500 and 128 x 128 x 40, the errors of the norm, the rms sizes, mu
// and E against 64 bits are 0.55, 0.65 to 0.82 and 1.00 times those of sums that
// went over to double per block: what is left is the rounding of each point.
//
// Double precision is scarce here (one operation of a warp takes 76 cycles of
// its scheduler, a division 1,500): a warp's sum of one double through
// shuffles takes as long as 100 float operations.
#pragma once

#include "common.cuh"

namespace rotgp {

struct fpair {
  float hi, lo;
};
__device__ __forceinline__ fpair sum_add(fpair a, fpair b) {
  const float s = __fadd_rn(a.hi, b.hi), t = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ fpair sum_xor(fpair v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double sum_xor(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}
// f times a sum (f exact enough in the working precision: a coordinate square)
__device__ __forceinline__ fpair sum_scale(float f, fpair a) {
  const float p = f * a.hi;
  return {p, fmaf(f, a.hi, -p) + f * a.lo};
}
__device__ __forceinline__ double sum_scale(double f, double a) { return f * a; }
__device__ __forceinline__ double sum_value(fpair a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double sum_value(double a) { return a; }

// Running sum of a thread: compensated in float, plain in double.
template <class T>
struct run_sum;
template <>
struct run_sum<float> {
  using sum = fpair;
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float y = __fsub_rn(x, c), t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
  }
  __device__ __forceinline__ fpair value() const { return {s, -c}; }
};
template <>
struct run_sum<double> {
  using sum = double;
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double value() const { return s; }
};
__device__ __forceinline__ fpair sum_zero(fpair*) { return {0.f, 0.f}; }
__device__ __forceinline__ double sum_zero(double*) { return 0.0; }

// The sums over a block of 256 threads of 16 values a thread: out[v] for v <
// 16 in shared memory (after a barrier).  Each level of the warp's reduction
// halves the values a lane carries, 16 additions in all instead of 80.
template <class S>
__device__ __forceinline__ void block_sums16(S (&v)[16], S (&red)[8][16]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const S send = upper ? v[i] : v[i + h], keep = upper ? v[i + h] : v[i];
      v[i] = sum_add(keep, sum_xor(send, o));
    }
  }
  v[0] = sum_add(v[0], sum_xor(v[0], 1));
  if (!(lane & 1)) red[warp][lane >> 1] = v[0];
  __syncthreads();
}

// Block partials of 16 values into partials[block][16]; true in the block that
// finishes last, which then has the grid's sums in fin[0..15] (combined in a
// fixed order).  MAX15: value 15 is the largest `top` (not negative) instead,
// kept as a double.  256 threads; every thread of the block calls it.
template <bool MAX15, class S>
__device__ __forceinline__ bool grid_sums16(S (&v)[16], double top, double* partials,
                                            unsigned* counter, double (&fin)[16]) {
  __shared__ S red[8][16];
  __shared__ double cmb[16][16];
  __shared__ unsigned long long wtop[8];
  __shared__ bool last;
  const int t = threadIdx.x;
  auto larger = [](unsigned long long a, unsigned long long b) { return a > b ? a : b; };
  if (MAX15) {
    // values that are not negative order as their bits
    unsigned long long m = __double_as_longlong(top);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = larger(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((t & 31) == 0) wtop[t >> 5] = m;
  }
  block_sums16(v, red);
  union word {
    S s;
    double d;
    unsigned long long u;
  };
  static_assert(sizeof(S) == 8, "partials");
  if (t < 16) {
    word w;
    w.s = red[0][t];
#pragma unroll
    for (int i = 1; i < 8; ++i) w.s = sum_add(w.s, red[i][t]);
    if (MAX15 && t == 15) {
      w.u = wtop[0];
#pragma unroll
      for (int i = 1; i < 8; ++i) w.u = larger(w.u, wtop[i]);
    }
    partials[(size_t)blockIdx.x * 16 + t] = w.d;
  }
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  {
    const bool mx = MAX15 && (t & 15) == 15;
    word r;
    r.u = 0;
    for (unsigned b = t >> 4; b < gridDim.x; b += 16) {
      word w;
      w.d = __ldcg(partials + (size_t)b * 16 + (t & 15));
      if (mx)
        r.u = larger(r.u, w.u);
      else
        r.s = sum_add(r.s, w.s);
    }
    cmb[t >> 4][t & 15] = r.d;
  }
  __syncthreads();
  if (t < 16) {
    word r;
    r.d = cmb[0][t];
#pragma unroll
    for (int i = 1; i < 16; ++i) {
      word w;
      w.d = cmb[i][t];
      if (MAX15 && t == 15)
        r.u = larger(r.u, w.u);
      else
        r.s = sum_add(r.s, w.s);
    }
    fin[t] = MAX15 && t == 15 ? r.d : sum_value(r.s);
  }
  if (t == 0) *counter = 0u;
  __syncthreads();
  return true;
}

}  // namespace rotgp
