// warmstart.cu -- the learned warm start: a convolutional encoder-decoder
// that proposes an initial wave function for a rotating run from its
// parameters (Omega, g, nu), standing in for the paper's practice (Sec. 1,
// Sec. 3) of starting a fast-rotating imaginary-time run from a converged
// lattice computed beforehand at a lower Omega.  Its proposal only seeds
// imaginary-time propagation, which decides the converged state.
//
// Network (every convolution 3 x 3, stride 1, zero padding 1, channels last):
//   input  6 planes on the G x G grid of the run: the Thomas-Fermi amplitude
//          of the rotating anisotropic trap, x / L, y / L, Omega, g / 1000,
//          (nu - 1) / 0.1 (features_kernel)
//   e0 = relu(conv0(in)), e1 = relu(conv1(e0))                 G,   6->32->32
//   e2 = relu(conv2(pool(e1))), e3 = relu(conv3(e2))           G/2, 32->64->64
//   e4 = relu(conv4(pool(e3))), e5 = relu(conv5(e4))           G/4, 64->128->128
//   b6 = relu(conv6(pool(e5))), b7 = relu(conv7(b6))           G/8, 128->128->128
//   d8 = relu(conv8(up(b7) + e5))                              G/4, 128->64
//   d9 = relu(conv9(up(d8) + e3))                              G/2, 64->32
//   d10 = relu(conv10(up(d9) + e1)), out = conv11(d10)         G,   32->32->2
// (pool = 2 x 2 mean, up = nearest doubling), 684,642 parameters.  out holds
// 2 L psi (real, imaginary parts) on the grid's points 0 .. G-1 of each
// axis (point G, the far edge, is zero).
//
// Precision: weights and activations are stored in bfloat16; every
// convolution, pooling and reduction accumulates in float; weight gradients,
// activation gradients and the Adam state are float, with a float master
// copy of the weights from which the bfloat16 copy is refreshed after every
// update.
#include <cuda_bf16.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/rotgp.h"
#include "common.cuh"

namespace {

using bf16 = __nv_bfloat16;
using rotgp::splitmix64_unit;

constexpr int kWsCin = 6;
constexpr int kWsLayers = 12;
constexpr int kWsC[kWsLayers][2] = {{kWsCin, 32}, {32, 32},  {32, 64},   {64, 64},
                                    {64, 128},    {128, 128}, {128, 128}, {128, 128},
                                    {128, 64},    {64, 32},   {32, 32},   {32, 2}};
// grid divisor of each layer (G / div)
constexpr int kWsDiv[kWsLayers] = {1, 1, 2, 2, 4, 4, 8, 8, 4, 2, 1, 1};

constexpr int kTile = 16;   // pixels per tile side

// ---------------------------------------------------------------- conv
// What bounds the three convolutions: FP32 FMAs (49 G multiply-adds per step of
// 16 runs of 128^2, 0.66 ms each way at the FP32 rate).  Every sum is taken in
// one fixed order (chunks of 8 input channels, then the 9 taps, then the
// channels; for the weights the points of a run of tiles in raster order),
// because the bfloat16 roundings after it and the sign that Adam's first steps
// take from a gradient turn on the last bit.  So the work is split over outputs
// only, and what limits it is the register bandwidth of shared memory, 128
// bytes a cycle and SM however many lanes read the same word: a thread holds a
// block of outputs (8 points x 8 channels; 3 taps x 2 x 4 channels of weights)
// and products are packed FP32x2.  The next chunk's values are fetched into
// registers while the present one is computed.  GB300, step of 16 runs of
// 128^2, before / after (a pixel x 32 channels and a weight's 9 taps per
// thread; atomic adds): 32 -> 32 channels at 128^2 forward 198 / 95 us, data 238
// / 107, weights 333 / 148; 6 -> 32 weights 237 / 51; 32 -> 2 forward 168 / 24,
// weights 297 / 35; 128 -> 128 at 16^2 forward 138 / 40; the whole step 6.95 /
// 3.13 ms.

// NC consecutive channels of a point, as stored.
template <int NC, class T>
struct chan {
  static constexpr int W = NC * (int)sizeof(T) / 4;
  unsigned w[W];
  __device__ __forceinline__ void load(const T* p) {
    if constexpr (W % 4 == 0) {
#pragma unroll
      for (int i = 0; i < W / 4; ++i) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(p) + i);
        w[4 * i] = t.x;
        w[4 * i + 1] = t.y;
        w[4 * i + 2] = t.z;
        w[4 * i + 3] = t.w;
      }
    } else if constexpr (W % 2 == 0) {
#pragma unroll
      for (int i = 0; i < W / 2; ++i) {
        const uint2 t = __ldg(reinterpret_cast<const uint2*>(p) + i);
        w[2 * i] = t.x;
        w[2 * i + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < W; ++i) w[i] = __ldg(reinterpret_cast<const unsigned*>(p) + i);
    }
  }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = 0u;
  }
  __device__ __forceinline__ float get(int c) const {
    if constexpr (sizeof(T) == 4) return __uint_as_float(w[c]);
    return __uint_as_float(c & 1 ? w[c / 2] & 0xffff0000u : w[c / 2] << 16);
  }
};

// Forward or backward-data convolution of a [B][H][W][Ci] tensor with 3 x 3
// weights.  Forward: out[., co] = sum_{k, ci} in[p + off_k, ci] w[k][ci][co]
// + bias.  Backward data (BWD): the input is the layer's output gradient dY
// (masked by mask > 0 when mask is given: the ReLU of that layer), and
// out[., ci] = sum_{k, co} dZ[p - off_k, co] w[k][ci][co], i.e. the forward
// form with the flipped kernel and swapped channel roles.
//
// A block of two warps takes CO output channels of TH rows, NC input channels
// at a time (8, or all of them where there are fewer); a thread one column and
// Q of the channels.  Its points are packed in pairs of rows r, r + TH / 2, which
// the patch keeps side by side so that every tap reads whole pairs; the weights
// stay bfloat16 in shared memory, a shift or mask making each a pair of equal
// floats for TH / 2 packed FMAs.  CO = 32: 16 columns, four groups of 8 channels.
// CO = 2 (the output layer, which 32 channels would mostly pad): 64 columns.
template <class TIn, class TOut, bool BWD, int NC, int CO, int TH>
__global__ void __launch_bounds__(64) k_conv(const TIn* __restrict__ in,
                                             const bf16* __restrict__ mask,
                                             const bf16* __restrict__ w,
                                             const float* __restrict__ bias, TOut* out, int H,
                                             int W, int Ci, int Co, int relu) {
  static_assert(CO == 32 || CO == 2, "channels per block");
  constexpr int G = CO == 32 ? 4 : 1, Q = CO / G;  // channel groups, channels per thread
  constexpr int TW = 64 / G, PX = TW + 2, PR = TH / 2;
  __shared__ float2 sx[NC][PR + 2][PX];            // rows r and r + PR
  __shared__ __align__(16) unsigned short sw[9][NC][CO];
  const int tiles_x = (W + TW - 1) / TW, tiles_y = (H + TH - 1) / TH;
  const int cob = blockIdx.y * CO, tid = threadIdx.x;
  int t = blockIdx.x;
  const int tx = t % tiles_x;
  t /= tiles_x;
  const int ty = t % tiles_y;
  const int b = t / tiles_y;
  in += (size_t)b * H * W * Ci;
  if (BWD && mask) mask += (size_t)b * H * W * Ci;
  const int cg = tid % G, col = tid / G;
  // the points of the patch (halo of one pixel, zeros outside the image) and
  // the weights that this thread fetches
  constexpr int UI = (PX * (TH + 2) + 63) / 64;
  constexpr int WC = BWD ? NC : CO == 32 ? 8 : 2;                  // channels per weight unit
  constexpr int WN = BWD ? 9 * CO : 9 * NC * (CO / WC), UW = (WN + 63) / 64;
  int off[UI];
#pragma unroll
  for (int i = 0; i < UI; ++i) {
    const int u = tid + 64 * i;
    const int gx = tx * TW + u % PX - 1, gy = ty * TH + u / PX - 1;
    off[i] = u < PX * (TH + 2) && gx >= 0 && gx < W && gy >= 0 && gy < H ? (gy * W + gx) * Ci : -1;
  }
  chan<NC, TIn> rin[UI];
  chan<NC, bf16> rm[BWD ? UI : 1];
  chan<WC, bf16> rw[UW];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int i = 0; i < UI; ++i) {
      if (off[i] >= 0) {
        rin[i].load(in + off[i] + c0);
        if (BWD && mask) rm[i].load(mask + off[i] + c0);
      } else {
        rin[i].zero();
      }
    }
    // forward w[k][ci][co]; backward w[8-k][co][ci], the layer's weight tensor
    // being [9][layer Ci][layer Co]
#pragma unroll
    for (int i = 0; i < UW; ++i) {
      const int u = tid + 64 * i;
      if (u >= WN) continue;
      if (BWD) {
        rw[i].load(w + ((size_t)(8 - u / CO) * Co + cob + u % CO) * Ci + c0);
      } else {
        const int j = u % (CO / WC), r = u / (CO / WC);
        rw[i].load(w + ((size_t)(r / NC) * Ci + c0 + r % NC) * Co + cob + WC * j);
      }
    }
  };
  auto stage = [&] {
#pragma unroll
    for (int i = 0; i < UI; ++i) {
      const int u = tid + 64 * i, qx = u % PX, qy = u / PX;
      if (u >= PX * (TH + 2)) continue;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float v = rin[i].get(c);
        if (BWD && mask && off[i] >= 0 && !(rm[i].get(c) > 0.f)) v = 0.f;
        if (qy < PR + 2) sx[c][qy][qx].x = v;
        if (qy >= PR) sx[c][qy - PR][qx].y = v;
      }
    }
#pragma unroll
    for (int i = 0; i < UW; ++i) {
      const int u = tid + 64 * i;
      if (u >= WN) continue;
      if constexpr (BWD) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
          sw[u / CO][c][u % CO] = (unsigned short)(c & 1 ? rw[i].w[c / 2] >> 16 : rw[i].w[c / 2]);
      } else if constexpr (WC == 8) {
        reinterpret_cast<uint4*>(sw)[u] = make_uint4(rw[i].w[0], rw[i].w[1], rw[i].w[2], rw[i].w[3]);
      } else {
        reinterpret_cast<unsigned*>(sw)[u] = rw[i].w[0];
      }
    }
  };
  float2 acc[PR][Q];
#pragma unroll
  for (int p = 0; p < PR; ++p)
#pragma unroll
    for (int c = 0; c < Q; ++c) acc[p][c] = make_float2(0.f, 0.f);
  fetch(0);
  for (int c0 = 0; c0 < Ci; c0 += NC) {
    __syncthreads();
    stage();
    __syncthreads();
    if (c0 + NC < Ci) fetch(c0 + NC);
#pragma unroll 1
    for (int k = 0; k < 9; ++k) {
      const float2* xr = &sx[0][k / 3][col + k % 3];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float2 v[PR];
#pragma unroll
        for (int p = 0; p < PR; ++p) v[p] = xr[(c * (PR + 2) + p) * PX];
        unsigned wk[Q / 2];
        if constexpr (Q == 8) {
          const uint4 u = *reinterpret_cast<const uint4*>(&sw[k][c][8 * cg]);
          wk[0] = u.x;
          wk[1] = u.y;
          wk[2] = u.z;
          wk[3] = u.w;
        } else {
          wk[0] = *reinterpret_cast<const unsigned*>(&sw[k][c][0]);
        }
#pragma unroll
        for (int j = 0; j < Q / 2; ++j) {
          const float lo = __uint_as_float(wk[j] << 16), hi = __uint_as_float(wk[j] & 0xffff0000u);
#pragma unroll
          for (int p = 0; p < PR; ++p) {
            acc[p][2 * j] = __ffma2_rn(v[p], make_float2(lo, lo), acc[p][2 * j]);
            acc[p][2 * j + 1] = __ffma2_rn(v[p], make_float2(hi, hi), acc[p][2 * j + 1]);
          }
        }
      }
    }
  }
  const int x = tx * TW + col, go = cob + cg * Q;
  if (x >= W) return;
  float bs[Q];
#pragma unroll
  for (int c = 0; c < Q; ++c) bs[c] = bias ? bias[go + c] : 0.f;
#pragma unroll
  for (int r = 0; r < TH; ++r) {
    const int y = ty * TH + r;
    if (y >= H) continue;
    float v[Q];
#pragma unroll
    for (int c = 0; c < Q; ++c) {
      v[c] = (r < PR ? acc[r % PR][c].x : acc[r % PR][c].y) + bs[c];
      if (relu) v[c] = fmaxf(v[c], 0.f);
    }
    TOut* o = out + (((size_t)b * H + y) * W + x) * Co + go;
    if constexpr (sizeof(TOut) == 2) {
      unsigned k[Q / 2];
#pragma unroll
      for (int i = 0; i < Q / 2; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        k[i] = *reinterpret_cast<const unsigned*>(&h);
      }
      *reinterpret_cast<uint4*>(o) = make_uint4(k[0], k[1], k[2], k[3]);
    } else if constexpr (Q == 8) {
      reinterpret_cast<float4*>(o)[0] = make_float4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<float4*>(o)[1] = make_float4(v[4], v[5], v[6], v[7]);
    } else {
      *reinterpret_cast<float2*>(o) = make_float2(v[0], v[1]);
    }
  }
}

// Weight and bias gradients of a convolution: dW[k][ci][co] += sum over
// pixels of X[p + off_k, ci] dZ[p, co], db[co] += sum dZ[p, co], with
// dZ = dY masked by the ReLU of the layer's output.  A block takes CIB input
// x COB output channels and a run of 16 x 16 tiles of one image (where there are
// more runs than slots, several in turn), 8 rows of a tile at a time; its sums
// go to its slot of the partials, [slot][weights, bias], which k_grad_sum adds up
// in a fixed order, so that a training run is the same every time.
// A thread has one row of taps, two input channels and 4 output channels (2
// where the layer has no more): the inputs of three taps slide along the row in
// registers, so a point costs 24 bytes of shared memory for 12 packed FMAs.
// Blocks of the narrow layers keep 128 threads to fetch with.
constexpr int kGradH = 8;
constexpr int kGradSlots = 128;
template <int CIB, int COB>
struct grad_block {
  static constexpr int CG = COB == 32 ? 8 : 1;     // groups of output channels
  static constexpr int WORK = 3 * (CIB / 2) * CG;  // threads with sums
  static constexpr int THREADS = WORK < 128 ? 128 : WORK;
};
template <int CIB, int COB>
__global__ void __launch_bounds__(grad_block<CIB, COB>::THREADS, 3)
    k_conv_wgrad(const bf16* __restrict__ X, const float* __restrict__ dY,
                 const bf16* __restrict__ Yout, int relu, float* part, int B, int H, int W, int Ci,
                 int Co, int tiles_per_block) {
  using block = grad_block<CIB, COB>;
  constexpr int CG = block::CG, V = COB / CG, NT = block::THREADS, CP = CIB / 2;
  constexpr int PX = kTile + 2;
  __shared__ float2 sx[kGradH + 2][PX][CP];
  __shared__ __align__(16) float sz[kGradH * kTile][COB];
  const int tiles_x = (W + kTile - 1) / kTile, tiles_y = (H + kTile - 1) / kTile;
  const int ntiles = tiles_x * tiles_y;
  const int runs = (ntiles + tiles_per_block - 1) / tiles_per_block;
  const int c0 = blockIdx.y * CIB, cob = blockIdx.z * COB;
  float* dW = part + (size_t)blockIdx.x * (9 * Ci + 1) * Co;
  float* db = dW + (size_t)9 * Ci * Co;
  const int cg = threadIdx.x % CG, cp = threadIdx.x / CG % CP, ky = threadIdx.x / (CG * CP);
  const bool works = threadIdx.x < block::WORK;
  const bool has_bias = threadIdx.x < CG && blockIdx.y == 0;  // ky = cp = 0
  float2 acc[3][2][V / 2], bacc[V / 2];
  constexpr int NX = (kGradH + 2) * PX * CP, UX = (NX + NT - 1) / NT;
  constexpr int NZ = kGradH * kTile * CG, UZ = (NZ + NT - 1) / NT;
  chan<2, bf16> rx[UX];
  chan<V, float> rz[UZ];
  chan<V, bf16> rm[UZ];
  const bf16 *Xb = nullptr, *Yb = nullptr;  // of the image
  const float* dYb = nullptr;
  auto fetch = [&](int hh) {  // half tile hh
    const int tt = hh >> 1;
    const int x0 = tt % tiles_x * kTile, y0 = tt / tiles_x * kTile + (hh & 1) * kGradH;
#pragma unroll
    for (int i = 0; i < UX; ++i) {
      const int u = threadIdx.x + NT * i, c = u % CP, q = u / CP;
      const int gx = x0 + q % PX - 1, gy = y0 + q / PX - 1;
      if (u < NX && gx >= 0 && gx < W && gy >= 0 && gy < H && c0 + 2 * c < Ci)
        rx[i].load(Xb + (size_t)(gy * W + gx) * Ci + 2 * c);
      else
        rx[i].zero();
    }
#pragma unroll
    for (int i = 0; i < UZ; ++i) {
      const int u = threadIdx.x + NT * i, c = u % CG, q = u / CG;
      const int gx = x0 + q % kTile, gy = y0 + q / kTile;
      if (u < NZ && gx < W && gy < H) {
        const size_t o = (size_t)(gy * W + gx) * Co + V * c;
        rz[i].load(dYb + o);
        if (relu) rm[i].load(Yb + o);
      } else {
        rz[i].zero();
        rm[i].zero();
      }
    }
  };
  const int items = B * runs, per = (items + (int)gridDim.x - 1) / (int)gridDim.x;
  const int item0 = blockIdx.x * per;
  for (int item = item0; item < min(items, item0 + per); ++item) {
    const int b = item / runs, run = item % runs;
    Xb = X + (size_t)b * H * W * Ci + c0;
    dYb = dY + (size_t)b * H * W * Co + cob;
    if (relu) Yb = Yout + (size_t)b * H * W * Co + cob;
    const int first = 2 * run * tiles_per_block;
    const int last = min(2 * ntiles, first + 2 * tiles_per_block);
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      bacc[i] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[k][0][i] = acc[k][1][i] = make_float2(0.f, 0.f);
    }
    fetch(first);
    for (int hh = first; hh < last; ++hh) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < UX; ++i) {
        const int u = threadIdx.x + NT * i;
        if (u < NX) (&sx[0][0][0])[u] = make_float2(rx[i].get(0), rx[i].get(1));
      }
#pragma unroll
      for (int i = 0; i < UZ; ++i) {
        const int u = threadIdx.x + NT * i;
        if (u >= NZ) continue;
        float* z = &sz[0][0] + V * u;
#pragma unroll
        for (int k = 0; k < V; ++k) z[k] = !relu || rm[i].get(k) > 0.f ? rz[i].get(k) : 0.f;
      }
      __syncthreads();
      if (hh + 1 < last) fetch(hh + 1);
      if (!works) continue;
#pragma unroll 1
      for (int qy = 0; qy < kGradH; ++qy) {
        const float2* xr = &sx[qy + ky][0][cp];
        float2 win[3];
        win[0] = xr[0];
        win[1] = xr[CP];
#pragma unroll
        for (int qx = 0; qx < kTile; ++qx) {
          win[(qx + 2) % 3] = xr[(qx + 2) * CP];
          float2 dz[V / 2];
          const float* zr = &sz[qy * kTile + qx][V * cg];
          if constexpr (V == 4) {
            const float4 z = *reinterpret_cast<const float4*>(zr);
            dz[0] = make_float2(z.x, z.y);
            dz[1] = make_float2(z.z, z.w);
          } else {
            dz[0] = *reinterpret_cast<const float2*>(zr);
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float2 t = win[(qx + k) % 3];
#pragma unroll
            for (int i = 0; i < V / 2; ++i) {
              acc[k][0][i] = __ffma2_rn(make_float2(t.x, t.x), dz[i], acc[k][0][i]);
              acc[k][1][i] = __ffma2_rn(make_float2(t.y, t.y), dz[i], acc[k][1][i]);
            }
          }
          if (has_bias)
#pragma unroll
            for (int i = 0; i < V / 2; ++i) bacc[i] = __fadd2_rn(bacc[i], dz[i]);
        }
      }
    }
    if (!works) continue;
    const bool more = item > item0;  // add to the slot's earlier runs
    auto put = [&](float* d, float2 v) {
      float2* q = reinterpret_cast<float2*>(d);
      if (more) v = __fadd2_rn(*q, v);
      *q = v;
    };
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int gc = c0 + 2 * cp + e;
      if (gc >= Ci) continue;
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < V / 2; ++i)
          put(dW + ((size_t)(3 * ky + k) * Ci + gc) * Co + cob + V * cg + 2 * i, acc[k][e][i]);
    }
    // the bias gradient once, from the blocks of the first input-channel chunk
    if (has_bias)
#pragma unroll
      for (int i = 0; i < V / 2; ++i) put(db + cob + V * cg + 2 * i, bacc[i]);
  }
}

// g[i] = sum of the slots' partials, in eight interleaved sums, the shortest chain
// of the orders tried.  All of them agree with the 64-bit gradients to 6e-7 of
// their scale; but training amplifies last bits (Adam's first steps take a
// gradient's sign), and the median steps to convergence over the 24 held-out runs,
// which tests/test_warmstart.py compares with the analytic start's 173,000, is
// chaotic: 75,500 with this order, 146,500 and 210,000 with two others, 61,500 to
// 232,000 with atomic adds.  A fixed order makes the outcome the same every time;
// it does not make this order's network a better one.
__global__ void k_grad_sum(const float* __restrict__ part, float* g, int slots, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 0.f;
  for (int k = 0; k < slots; k += 8) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] += k + j < slots ? part[(size_t)(k + j) * n + i] : 0.f;
  }
  g[i] = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
}

// ---------------------------------------------------------------- glue
// A thread takes 16 bytes of channels of a point (C is a multiple of 32): with a
// channel a thread the passes waited on the index divisions and narrow loads
// (up-and-add of 16 runs of 128^2 x 32 40 us, pooling 14, its gradient 21).
__device__ __forceinline__ uint4 bf16x8(const float (&v)[8]) {
  unsigned k[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    k[i] = *reinterpret_cast<const unsigned*>(&h);
  }
  return make_uint4(k[0], k[1], k[2], k[3]);
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
// out = mean of each 2 x 2 block of in ([B][2h][2w][C] -> [B][h][w][C])
__global__ void k_pool(const bf16* in, bf16* out, int B, int h, int w, int C) {
  const unsigned n = (unsigned)C / 8;
  const size_t tot = (size_t)B * h * w * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / n, bh = r / w;  // point, image row
    const size_t W2 = 2 * (size_t)w, row = (size_t)W2 * C;
    const bf16* p = in + (2 * bh * W2 + 2 * (r % w)) * C + 8 * (i % n);
    chan<8, bf16> a, b, c, d;
    a.load(p);
    b.load(p + C);
    c.load(p + row);
    d.load(p + row + C);
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = 0.25f * (a.get(k) + b.get(k) + c.get(k) + d.get(k));
    reinterpret_cast<uint4*>(out)[i] = bf16x8(v);
  }
}
// gin[2x2 block] += gout / 4
__global__ void k_pool_bwd(const float* gout, float* gin, int B, int h, int w, int C) {
  const unsigned n = (unsigned)C / 4;
  const size_t tot = (size_t)B * h * w * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / n, bh = r / w, W2 = 2 * (size_t)w, row = W2 * n;
    float4* p = reinterpret_cast<float4*>(gin) + (2 * bh * W2 + 2 * (r % w)) * n + i % n;
    float4 g = reinterpret_cast<const float4*>(gout)[i];
    g = make_float4(0.25f * g.x, 0.25f * g.y, 0.25f * g.z, 0.25f * g.w);
    p[0] = add4(p[0], g);
    p[n] = add4(p[n], g);
    p[row] = add4(p[row], g);
    p[row + n] = add4(p[row + n], g);
  }
}
// out = up(a) + skip ([B][h][w][C] doubled, plus [B][2h][2w][C])
__global__ void k_up_add(const bf16* a, const bf16* skip, bf16* out, int B, int h, int w, int C) {
  const unsigned n = (unsigned)C / 8;
  const size_t tot = (size_t)B * h * w * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / n, bh = r / w, W2 = 2 * (size_t)w, row = W2 * C;
    const size_t o = (2 * bh * W2 + 2 * (r % w)) * C + 8 * (i % n);
    chan<8, bf16> u;
    u.load(a + 8 * i);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const size_t oq = o + (q >> 1) * row + (q & 1) * C;
      chan<8, bf16> s;
      s.load(skip + oq);
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = u.get(k) + s.get(k);
      *reinterpret_cast<uint4*>(out + oq) = bf16x8(v);
    }
  }
}
// ga = sum of each 2 x 2 block of g; gskip = g (the skip's gradient starts here)
__global__ void k_up_add_bwd(const float* g, float* ga, float* gskip, int B, int h, int w, int C) {
  const unsigned n = (unsigned)C / 4;
  const size_t tot = (size_t)B * h * w * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t r = i / n, bh = r / w, W2 = 2 * (size_t)w, row = W2 * n;
    const size_t o = (2 * bh * W2 + 2 * (r % w)) * n + i % n;
    const float4* p = reinterpret_cast<const float4*>(g) + o;
    float4* q = reinterpret_cast<float4*>(gskip) + o;
    const float4 a = p[0], b = p[n], c = p[row], d = p[row + n];
    q[0] = a;
    q[n] = b;
    q[row] = c;
    q[row + n] = d;
    reinterpret_cast<float4*>(ga)[i] = add4(add4(add4(a, b), c), d);
  }
}

// Loss sum((y - t)^2) into per-block partials and its gradient 2 (y - t) / n.
__global__ void k_mse(const float* y, const float* t, float* dy, double* part, size_t n) {
  __shared__ double ws[8];
  double s = 0;
  const float inv = 2.0f / (float)n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    s += (double)d * d;
    dy[i] = inv * d;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += ws[i];
    part[blockIdx.x] = tot;
  }
}

// Adam on the float master weights, then their bfloat16 copy.
__global__ void k_adam(float* p, bf16* pb, const float* g, float* m, float* v, size_t n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = fmaf(b1, m[i], (1.f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = w;
    pb[i] = __float2bfloat16(w);
  }
}

__global__ void k_to_bf16(const float* in, bf16* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = __float2bfloat16(in[i]);
}

// Input planes of run i (Omega, g, nu = prm[3i..3i+2]) on the G x G points
// x_j = -L + j h of both axes (h = 2 L / G): the Thomas-Fermi amplitude of
// the rotating trap, sqrt(max(0, mu - (gx^2 x^2 + gy^2 y^2) / 2) / g) with
// the centrifugally reduced frequencies gx^2 = 1 - Omega^2, gy^2 = nu^2 -
// Omega^2 and mu = sqrt(g gx gy / pi) (unit norm), scaled by 2 L; then x / L,
// y / L, Omega, g / 1000, (nu - 1) / 0.1.
// A block has one row of one run: what the row's points share is computed once
// (a double division or root costs a warp 1,500 cycles; nine of them a point
// took 62 us for 16 runs of 128^2).
__global__ void k_features(const double* prm, bf16* out, int G, double L) {
  __shared__ double c[8];
  const int k = blockIdx.x % G, r = blockIdx.x / G;
  const double h = 2.0 * L / G, y = -L + k * h;
  if (threadIdx.x == 0) {
    const double om = prm[3 * r], g = prm[3 * r + 1], nu = prm[3 * r + 2];
    const double gx2 = fmax(1.0 - om * om, 1e-3), gy2 = fmax(nu * nu - om * om, 1e-3);
    c[0] = sqrt(g * sqrt(gx2 * gy2) / 3.14159265358979323846);
    c[1] = gx2;
    c[2] = gy2;
    c[3] = g;
    c[4] = y / L;
    c[5] = om;
    c[6] = g / 1000.0;
    c[7] = (nu - 1.0) / 0.1;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < G; j += blockDim.x) {
    const double x = -L + j * h;
    const double n_tf = fmax(0.0, c[0] - 0.5 * (c[1] * x * x + c[2] * y * y)) / c[3];
    bf16* o = out + ((size_t)blockIdx.x * G + j) * kWsCin;
    o[0] = __float2bfloat16((float)(2.0 * L * sqrt(n_tf)));
    o[1] = __float2bfloat16((float)(x / L));
    o[2] = __float2bfloat16((float)c[4]);
    o[3] = __float2bfloat16((float)c[5]);
    o[4] = __float2bfloat16((float)c[6]);
    o[5] = __float2bfloat16((float)c[7]);
  }
}

// Network output (2 L psi on G x G points) -> ABI wave function of run i:
// (G+1) x (G+1) complex double, psi = out / (2 L), the far edge zero; with
// rp != 0 multiplied by the random phase exp(2 pi i R) of Eq. fun, R drawn
// from SplitMix64(seed) for point n = k (G + 1) + j as rotgp_init_analytic
// draws it.
__global__ void k_out_to_psi(const float* y, double* psi, int n, int G, double L, int rp,
                             unsigned long long seed) {
  const size_t P = (size_t)(G + 1) * (G + 1), tot = (size_t)n * P;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(i / P);
    const size_t q = i % P;
    const int j = (int)(q % (G + 1)), k = (int)(q / (G + 1));
    double re = 0, im = 0;
    if (j < G && k < G && j > 0 && k > 0) {
      const float* v = y + (((size_t)r * G + k) * G + j) * 2;
      re = v[0] / (2.0 * L);
      im = v[1] / (2.0 * L);
      if (rp) {
        double sn, cs;
        sincos(2.0 * 3.14159265358979323846 * splitmix64_unit(seed, q), &sn, &cs);
        const double a = re * cs - im * sn;
        im = re * sn + im * cs;
        re = a;
      }
    }
    psi[2 * i] = re;
    psi[2 * i + 1] = im;
  }
}

// ABI wave functions ((G+1)^2 complex double) -> targets 2 L psi on G x G.
__global__ void k_psi_to_target(const double* psi, float* t, int n, int G, double L) {
  const size_t tot = (size_t)n * G * G;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < tot;
       i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % G), k = (int)((i / G) % G), r = (int)(i / ((size_t)G * G));
    const double* v = psi + 2 * (((size_t)r * (G + 1) + k) * (G + 1) + j);
    t[2 * i] = (float)(2.0 * L * v[0]);
    t[2 * i + 1] = (float)(2.0 * L * v[1]);
  }
}

int blocks_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 152 * 16); }

}  // namespace

// ---------------------------------------------------------------- context
struct rotgp_ws {
  int G = 0, maxb = 0;
  cudaStream_t s = nullptr;
  size_t np = 0;
  std::vector<size_t> woff, boff;  // offsets of each layer's weights and bias
  float* p = nullptr;              // float master
  bf16* pb = nullptr;              // bfloat16 copy (weights; biases read as float master)
  float *g = nullptr, *m = nullptr, *v = nullptr;
  long long t = 0;                 // Adam step
  double* dprm = nullptr;          // run parameters (3 per run)
  bf16* x = nullptr;               // input planes
  bf16* act[kWsLayers] = {};       // layer outputs (the last one unused)
  bf16 *p1 = nullptr, *p2 = nullptr, *p3 = nullptr;  // pooled
  bf16 *s8 = nullptr, *s9 = nullptr, *s10 = nullptr; // up + skip sums
  float* y = nullptr;              // network output
  float* tgt = nullptr;            // targets
  float *gA = nullptr, *gB = nullptr, *gS1 = nullptr, *gS2 = nullptr, *gS3 = nullptr;
  float* wpart = nullptr;          // partial weight gradients of a layer
  double* part = nullptr;
  double* dpsi = nullptr;          // ABI wave functions (in or out)
  std::string err;
  size_t bytes = 0;
};

namespace {

thread_local std::string g_ws_error;

int wfail(rotgp_ws* w, int code, const char* msg, cudaError_t e = cudaSuccess) {
  std::string m = msg;
  if (e != cudaSuccess) m += std::string(": ") + cudaGetErrorString(e);
  if (w)
    w->err = m;
  else
    g_ws_error = m;
  return code;
}

template <class P>
cudaError_t walloc(rotgp_ws* w, P** p, size_t n) {
  w->bytes += n * sizeof(P);
  return cudaMalloc((void**)p, std::max<size_t>(n, 1) * sizeof(P));
}

size_t plane(const rotgp_ws* w, int layer, int c) {
  const size_t d = (size_t)w->G / kWsDiv[layer];
  return (size_t)w->maxb * d * d * c;
}

template <class TIn, class TOut, bool BWD, int NC, int CO, int TH>
void conv_launch(rotgp_ws* w, const TIn* in, const bf16* mask, int layer, TOut* out, int B,
                 int relu) {
  const int d = w->G / kWsDiv[layer];
  const int Ci = BWD ? kWsC[layer][1] : kWsC[layer][0];
  const int Co = BWD ? kWsC[layer][0] : kWsC[layer][1];
  constexpr int TW = CO == 32 ? 16 : 64;
  const int tiles = ((d + TW - 1) / TW) * ((d + TH - 1) / TH);
  const dim3 grid((unsigned)(tiles * B), (unsigned)(Co / CO));
  const float* bias = BWD ? nullptr : w->p + w->boff[layer];
  k_conv<TIn, TOut, BWD, NC, CO, TH><<<grid, 64, 0, w->s>>>(in, mask, w->pb + w->woff[layer], bias,
                                                            out, d, d, Ci, Co, relu);
}
template <class TIn, class TOut, bool BWD>
cudaError_t conv(rotgp_ws* w, const TIn* in, const bf16* mask, int layer, TOut* out, int B,
                 int relu) {
  // the channels of the first layer's input and of the output layer are their
  // own chunks; every other layer has multiples of 32
  if constexpr (!BWD && sizeof(TOut) == 4) {
    conv_launch<TIn, TOut, BWD, 8, 2, 8>(w, in, mask, layer, out, B, relu);
  } else {
    // planes that would give fewer than two blocks per SM in tiles of 8 rows
    // take tiles of 4 (128 -> 128 at 32^2, 512 blocks: 116 us in 8 rows, 124
    // in 4; at 16^2 128 blocks of 8 rows would leave SMs without one, 40 us in 4)
    const long long d = w->G / kWsDiv[layer];
    const long long blocks = (d + 15) / 16 * ((d + 7) / 8) * B * (kWsC[layer][BWD ? 0 : 1] / 32);
    constexpr int first = BWD ? 2 : kWsCin;
    if (kWsC[layer][BWD ? 1 : 0] == first)
      conv_launch<TIn, TOut, BWD, first, 32, 8>(w, in, mask, layer, out, B, relu);
    else if (blocks < 2 * 152)
      conv_launch<TIn, TOut, BWD, 8, 32, 4>(w, in, mask, layer, out, B, relu);
    else
      conv_launch<TIn, TOut, BWD, 8, 32, 8>(w, in, mask, layer, out, B, relu);
  }
  return cudaGetLastError();
}

// Tiles per run of a weight-gradient block in planes of d x d points, runs per
// image, and slots of partial sums for B images (none of them empty).
int grad_tiles(int d) {
  const int t = (d + kTile - 1) / kTile;
  return std::max(1, std::min(t * t, 8));
}
long long grad_runs(int d, int B) {
  const int t = (d + kTile - 1) / kTile, tpb = grad_tiles(d);
  return (long long)B * ((t * t + tpb - 1) / tpb);
}
int grad_slots(int d, int B) {
  const long long items = grad_runs(d, B), per = (items + kGradSlots - 1) / kGradSlots;
  return (int)((items + per - 1) / per);
}
template <int CIB, int COB>
void wgrad_launch(rotgp_ws* w, const bf16* X, const float* dY, const bf16* Yout, int layer, int B) {
  const int d = w->G / kWsDiv[layer];
  const int Ci = kWsC[layer][0], Co = kWsC[layer][1], n = (9 * Ci + 1) * Co;
  const int slots = grad_slots(d, B);
  const dim3 grid((unsigned)slots, (unsigned)((Ci + CIB - 1) / CIB), (unsigned)(Co / COB));
  k_conv_wgrad<CIB, COB><<<grid, grad_block<CIB, COB>::THREADS, 0, w->s>>>(
      X, dY, Yout, layer < kWsLayers - 1 ? 1 : 0, w->wpart, B, d, d, Ci, Co, grad_tiles(d));
  k_grad_sum<<<(n + 127) / 128, 128, 0, w->s>>>(w->wpart, w->g + w->woff[layer], slots, n);
}
cudaError_t wgrad(rotgp_ws* w, const bf16* X, const float* dY, const bf16* Yout, int layer,
                  int B) {
  if (kWsC[layer][1] == 2)
    wgrad_launch<8, 2>(w, X, dY, Yout, layer, B);
  else if (kWsC[layer][0] == kWsCin)
    wgrad_launch<8, 32>(w, X, dY, Yout, layer, B);
  else
    wgrad_launch<16, 32>(w, X, dY, Yout, layer, B);
  return cudaGetLastError();
}

// Forward pass of B runs whose input planes are in w->x; output in w->y.
cudaError_t forward(rotgp_ws* w, int B) {
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  const int G = w->G;
  chk(conv<bf16, bf16, false>(w, w->x, nullptr, 0, w->act[0], B, 1));
  chk(conv<bf16, bf16, false>(w, w->act[0], nullptr, 1, w->act[1], B, 1));
  k_pool<<<blocks_for(((size_t)B * G * G / 4 * 32) / 8), 256, 0, w->s>>>(w->act[1], w->p1, B, G / 2, G / 2, 32);
  chk(conv<bf16, bf16, false>(w, w->p1, nullptr, 2, w->act[2], B, 1));
  chk(conv<bf16, bf16, false>(w, w->act[2], nullptr, 3, w->act[3], B, 1));
  k_pool<<<blocks_for(((size_t)B * G * G / 16 * 64) / 8), 256, 0, w->s>>>(w->act[3], w->p2, B, G / 4, G / 4, 64);
  chk(conv<bf16, bf16, false>(w, w->p2, nullptr, 4, w->act[4], B, 1));
  chk(conv<bf16, bf16, false>(w, w->act[4], nullptr, 5, w->act[5], B, 1));
  k_pool<<<blocks_for(((size_t)B * G * G / 64 * 128) / 8), 256, 0, w->s>>>(w->act[5], w->p3, B, G / 8, G / 8, 128);
  chk(conv<bf16, bf16, false>(w, w->p3, nullptr, 6, w->act[6], B, 1));
  chk(conv<bf16, bf16, false>(w, w->act[6], nullptr, 7, w->act[7], B, 1));
  k_up_add<<<blocks_for(((size_t)B * G * G / 16 * 128) / 32), 256, 0, w->s>>>(w->act[7], w->act[5], w->s8, B, G / 8, G / 8, 128);
  chk(conv<bf16, bf16, false>(w, w->s8, nullptr, 8, w->act[8], B, 1));
  k_up_add<<<blocks_for(((size_t)B * G * G / 4 * 64) / 32), 256, 0, w->s>>>(w->act[8], w->act[3], w->s9, B, G / 4, G / 4, 64);
  chk(conv<bf16, bf16, false>(w, w->s9, nullptr, 9, w->act[9], B, 1));
  k_up_add<<<blocks_for(((size_t)B * G * G * 32) / 32), 256, 0, w->s>>>(w->act[9], w->act[1], w->s10, B, G / 2, G / 2, 32);
  chk(conv<bf16, bf16, false>(w, w->s10, nullptr, 10, w->act[10], B, 1));
  chk(conv<bf16, float, false>(w, w->act[10], nullptr, 11, w->y, B, 0));
  chk(cudaGetLastError());
  return e;
}

// Backward pass from dL/dy in w->gA (float, [B][G][G][2]); weight gradients
// into w->g.
cudaError_t backward(rotgp_ws* w, int B) {
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  const int G = w->G;
  float *gA = w->gA, *gB = w->gB;
  // layer 11 (linear): dW from d10 and dy; d(d10) = conv^T(dy)
  chk(wgrad(w, w->act[10], gA, nullptr, 11, B));
  chk(conv<float, float, true>(w, gA, nullptr, 11, gB, B, 0));
  // layer 10: input s10 = up(d9) + e1
  chk(wgrad(w, w->s10, gB, w->act[10], 10, B));
  chk(conv<float, float, true>(w, gB, w->act[10], 10, gA, B, 0));  // gA = d(s10)
  k_up_add_bwd<<<blocks_for(((size_t)B * G * G / 4 * 32) / 4), 256, 0, w->s>>>(gA, gB, w->gS1, B, G / 2, G / 2, 32);
  // gB = d(d9); layer 9: input s9 = up(d8) + e3
  chk(wgrad(w, w->s9, gB, w->act[9], 9, B));
  chk(conv<float, float, true>(w, gB, w->act[9], 9, gA, B, 0));    // gA = d(s9)
  k_up_add_bwd<<<blocks_for(((size_t)B * G * G / 16 * 64) / 4), 256, 0, w->s>>>(gA, gB, w->gS2, B, G / 4, G / 4, 64);
  // gB = d(d8); layer 8: input s8 = up(b7) + e5
  chk(wgrad(w, w->s8, gB, w->act[8], 8, B));
  chk(conv<float, float, true>(w, gB, w->act[8], 8, gA, B, 0));    // gA = d(s8)
  k_up_add_bwd<<<blocks_for(((size_t)B * G * G / 64 * 128) / 4), 256, 0, w->s>>>(gA, gB, w->gS3, B, G / 8, G / 8, 128);
  // gB = d(b7); layer 7
  chk(wgrad(w, w->act[6], gB, w->act[7], 7, B));
  chk(conv<float, float, true>(w, gB, w->act[7], 7, gA, B, 0));    // gA = d(b6)
  // layer 6: input pool(e5)
  chk(wgrad(w, w->p3, gA, w->act[6], 6, B));
  chk(conv<float, float, true>(w, gA, w->act[6], 6, gB, B, 0));    // gB = d(p3)
  k_pool_bwd<<<blocks_for(((size_t)B * G * G / 64 * 128) / 4), 256, 0, w->s>>>(gB, w->gS3, B, G / 8, G / 8, 128);
  // gS3 = d(e5); layer 5
  chk(wgrad(w, w->act[4], w->gS3, w->act[5], 5, B));
  chk(conv<float, float, true>(w, w->gS3, w->act[5], 5, gA, B, 0)); // gA = d(e4)
  chk(wgrad(w, w->p2, gA, w->act[4], 4, B));
  chk(conv<float, float, true>(w, gA, w->act[4], 4, gB, B, 0));    // gB = d(p2)
  k_pool_bwd<<<blocks_for(((size_t)B * G * G / 16 * 64) / 4), 256, 0, w->s>>>(gB, w->gS2, B, G / 4, G / 4, 64);
  // gS2 = d(e3); layer 3
  chk(wgrad(w, w->act[2], w->gS2, w->act[3], 3, B));
  chk(conv<float, float, true>(w, w->gS2, w->act[3], 3, gA, B, 0)); // gA = d(e2)
  chk(wgrad(w, w->p1, gA, w->act[2], 2, B));
  chk(conv<float, float, true>(w, gA, w->act[2], 2, gB, B, 0));    // gB = d(p1)
  k_pool_bwd<<<blocks_for(((size_t)B * G * G / 4 * 32) / 4), 256, 0, w->s>>>(gB, w->gS1, B, G / 2, G / 2, 32);
  // gS1 = d(e1); layer 1
  chk(wgrad(w, w->act[0], w->gS1, w->act[1], 1, B));
  chk(conv<float, float, true>(w, w->gS1, w->act[1], 1, gA, B, 0)); // gA = d(e0)
  chk(wgrad(w, w->x, gA, w->act[0], 0, B));
  chk(cudaGetLastError());
  return e;
}

int check_batch(rotgp_ws* w, int n) {
  if (!w) return ROTGP_EINVAL;
  if (n < 1 || n > w->maxb) return wfail(w, ROTGP_EINVAL, "batch size out of range");
  return ROTGP_OK;
}

// parameters of n runs (host, 3 n doubles: Omega, g, nu) -> input planes
int load_features(rotgp_ws* w, int n, const double* prm, double L) {
  cudaError_t e = cudaMemcpyAsync(w->dprm, prm, 3 * n * sizeof(double), cudaMemcpyHostToDevice, w->s);
  if (e != cudaSuccess) return wfail(w, ROTGP_ECUDA, "copy parameters", e);
  k_features<<<(unsigned)(n * w->G), 128, 0, w->s>>>(w->dprm, w->x, w->G, L);
  e = cudaGetLastError();
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "features kernel", e);
}

// targets from n ABI wave functions (host or device, complex double)
int load_targets(rotgp_ws* w, int n, const double* psi, int on_device, double L) {
  const size_t P = (size_t)(w->G + 1) * (w->G + 1) * 2 * n;
  const double* src = psi;
  if (!on_device) {
    cudaError_t e = cudaMemcpyAsync(w->dpsi, psi, P * sizeof(double), cudaMemcpyHostToDevice, w->s);
    if (e != cudaSuccess) return wfail(w, ROTGP_ECUDA, "copy targets", e);
    src = w->dpsi;
  }
  k_psi_to_target<<<blocks_for((size_t)n * w->G * w->G), 256, 0, w->s>>>(src, w->tgt, n, w->G, L);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "target kernel", e);
}

// loss and gradients of n runs (features and targets loaded); loss to host
int loss_and_grad(rotgp_ws* w, int n, double* loss) {
  cudaError_t e = forward(w, n);
  const size_t ny = (size_t)n * w->G * w->G * 2;
  const int nb = 256;
  if (e == cudaSuccess) {
    k_mse<<<nb, 256, 0, w->s>>>(w->y, w->tgt, w->gA, w->part, ny);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = backward(w, n);
  double parts[256];
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(parts, w->part, sizeof parts, cudaMemcpyDeviceToHost, w->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(w->s);
  if (e != cudaSuccess) return wfail(w, ROTGP_ECUDA, "network pass", e);
  double s = 0;
  for (double x : parts) s += x;
  if (loss) *loss = s / (double)ny;
  return ROTGP_OK;
}

}  // namespace

// =============================================================== C ABI
extern "C" {

long long rotgp_ws_param_count(void) {
  long long n = 0;
  for (const auto& c : kWsC) n += 9LL * c[0] * c[1] + c[1];
  return n;
}

const char* rotgp_ws_last_error(const rotgp_ws* w) { return w ? w->err.c_str() : g_ws_error.c_str(); }

void rotgp_ws_destroy(rotgp_ws* w) {
  if (!w) return;
  cudaStreamSynchronize(w->s);
  void* ptrs[] = {w->p, w->pb, w->g, w->m, w->v, w->dprm, w->x, w->p1, w->p2, w->p3, w->s8,
                  w->s9, w->s10, w->y, w->tgt, w->gA, w->gB, w->gS1, w->gS2, w->gS3, w->wpart, w->part,
                  w->dpsi};
  for (void* p : ptrs) cudaFree(p);
  for (auto* a : w->act) cudaFree(a);
  delete w;
}

int rotgp_ws_create(int grid, int max_batch, void* stream, rotgp_ws** out) {
  g_ws_error.clear();
  if (!out) return wfail(nullptr, ROTGP_EINVAL, "null output");
  *out = nullptr;
  if (grid < 16 || grid % 16 != 0 || grid > 1024)
    return wfail(nullptr, ROTGP_EINVAL, "grid must be a multiple of 16 in [16, 1024]");
  if (max_batch < 1 || max_batch > 4096) return wfail(nullptr, ROTGP_EINVAL, "max_batch out of range");
  rotgp_ws* w = new (std::nothrow) rotgp_ws();
  if (!w) return wfail(nullptr, ROTGP_ENOMEM, "host allocation failed");
  w->G = grid;
  w->maxb = max_batch;
  w->s = static_cast<cudaStream_t>(stream);
  size_t off = 0;
  for (const auto& c : kWsC) {
    w->woff.push_back(off);
    off += 9 * (size_t)c[0] * c[1];
    w->boff.push_back(off);
    off += c[1];
  }
  w->np = off;
  const size_t G2 = (size_t)grid * grid * max_batch;
  cudaError_t e = walloc(w, &w->p, w->np);
  if (e == cudaSuccess) e = walloc(w, &w->pb, w->np);
  if (e == cudaSuccess) e = walloc(w, &w->g, w->np);
  if (e == cudaSuccess) e = walloc(w, &w->m, w->np);
  if (e == cudaSuccess) e = walloc(w, &w->v, w->np);
  if (e == cudaSuccess) e = walloc(w, &w->dprm, 3 * (size_t)max_batch);
  if (e == cudaSuccess) e = walloc(w, &w->x, G2 * kWsCin);
  for (int l = 0; l < kWsLayers && e == cudaSuccess; ++l)
    e = walloc(w, &w->act[l], plane(w, l, kWsC[l][1]));
  if (e == cudaSuccess) e = walloc(w, &w->p1, G2 / 4 * 32);
  if (e == cudaSuccess) e = walloc(w, &w->p2, G2 / 16 * 64);
  if (e == cudaSuccess) e = walloc(w, &w->p3, G2 / 64 * 128);
  if (e == cudaSuccess) e = walloc(w, &w->s8, G2 / 16 * 128);
  if (e == cudaSuccess) e = walloc(w, &w->s9, G2 / 4 * 64);
  if (e == cudaSuccess) e = walloc(w, &w->s10, G2 * 32);
  if (e == cudaSuccess) e = walloc(w, &w->y, G2 * 2);
  if (e == cudaSuccess) e = walloc(w, &w->tgt, G2 * 2);
  if (e == cudaSuccess) e = walloc(w, &w->gA, G2 * 32);
  if (e == cudaSuccess) e = walloc(w, &w->gB, G2 * 32);
  if (e == cudaSuccess) e = walloc(w, &w->gS1, G2 * 32);
  if (e == cudaSuccess) e = walloc(w, &w->gS2, G2 / 4 * 64);
  if (e == cudaSuccess) e = walloc(w, &w->gS3, G2 / 16 * 128);
  size_t np = 0;
  for (int l = 0; l < kWsLayers; ++l)
    np = std::max(np, (size_t)std::min<long long>(grad_runs(grid / kWsDiv[l], max_batch), kGradSlots) *
                          (9 * kWsC[l][0] + 1) * kWsC[l][1]);
  if (e == cudaSuccess) e = walloc(w, &w->wpart, np);
  if (e == cudaSuccess) e = walloc(w, &w->part, 256);
  if (e == cudaSuccess) e = walloc(w, &w->dpsi, (size_t)(grid + 1) * (grid + 1) * 2 * max_batch);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->m, 0, w->np * sizeof(float), w->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->v, 0, w->np * sizeof(float), w->s);
  if (e != cudaSuccess) {
    const int rc = wfail(nullptr, e == cudaErrorMemoryAllocation ? ROTGP_ENOMEM : ROTGP_ECUDA,
                         "network buffers", e);
    rotgp_ws_destroy(w);
    return rc;
  }
  *out = w;
  return ROTGP_OK;
}

int rotgp_ws_set_params(rotgp_ws* w, const float* params) {
  if (!w || !params) return w ? wfail(w, ROTGP_EINVAL, "null parameters") : ROTGP_EINVAL;
  cudaError_t e = cudaMemcpyAsync(w->p, params, w->np * sizeof(float), cudaMemcpyHostToDevice, w->s);
  if (e == cudaSuccess) {
    k_to_bf16<<<blocks_for(w->np), 256, 0, w->s>>>(w->p, w->pb, w->np);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(w->m, 0, w->np * sizeof(float), w->s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->v, 0, w->np * sizeof(float), w->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(w->s);
  w->t = 0;
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "set parameters", e);
}

int rotgp_ws_get_params(rotgp_ws* w, float* params) {
  if (!w || !params) return w ? wfail(w, ROTGP_EINVAL, "null parameters") : ROTGP_EINVAL;
  cudaError_t e = cudaMemcpyAsync(params, w->p, w->np * sizeof(float), cudaMemcpyDeviceToHost, w->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(w->s);
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "get parameters", e);
}

int rotgp_ws_propose(rotgp_ws* w, int n, const double* prm, double half_width, int random_phase,
                     unsigned long long seed, void* psi, int psi_on_device) {
  int rc = check_batch(w, n);
  if (rc) return rc;
  if (!prm || !psi || !(half_width > 0)) return wfail(w, ROTGP_EINVAL, "bad arguments");
  if ((rc = load_features(w, n, prm, half_width))) return rc;
  cudaError_t e = forward(w, n);
  double* dst = psi_on_device ? static_cast<double*>(psi) : w->dpsi;
  if (e == cudaSuccess) {
    k_out_to_psi<<<blocks_for((size_t)n * (w->G + 1) * (w->G + 1)), 256, 0, w->s>>>(
        w->y, dst, n, w->G, half_width, random_phase ? 1 : 0, seed);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && !psi_on_device)
    e = cudaMemcpyAsync(psi, w->dpsi, (size_t)n * (w->G + 1) * (w->G + 1) * 2 * sizeof(double),
                        cudaMemcpyDeviceToHost, w->s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(w->s);
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "propose", e);
}

int rotgp_ws_gradients(rotgp_ws* w, int n, const void* inputs, const float* targets, double* loss,
                       float* grads) {
  int rc = check_batch(w, n);
  if (rc) return rc;
  if (!inputs || !targets) return wfail(w, ROTGP_EINVAL, "null inputs or targets");
  const size_t G2 = (size_t)n * w->G * w->G;
  // input planes as float on the host -> bfloat16 on the device
  float* tmp = nullptr;
  cudaError_t e = cudaMalloc((void**)&tmp, G2 * kWsCin * sizeof(float));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(tmp, inputs, G2 * kWsCin * sizeof(float), cudaMemcpyHostToDevice, w->s);
  if (e == cudaSuccess) {
    k_to_bf16<<<blocks_for(G2 * kWsCin), 256, 0, w->s>>>(tmp, w->x, G2 * kWsCin);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(w->tgt, targets, G2 * 2 * sizeof(float), cudaMemcpyHostToDevice, w->s);
  if (e != cudaSuccess) {
    cudaFree(tmp);
    return wfail(w, ROTGP_ECUDA, "gradient inputs", e);
  }
  rc = loss_and_grad(w, n, loss);
  cudaFree(tmp);
  if (rc) return rc;
  if (grads) {
    e = cudaMemcpy(grads, w->g, w->np * sizeof(float), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return wfail(w, ROTGP_ECUDA, "copy gradients", e);
  }
  return ROTGP_OK;
}

int rotgp_ws_train_step(rotgp_ws* w, int n, const double* prm, double half_width,
                        const void* psi, int psi_on_device, float lr, double* loss) {
  int rc = check_batch(w, n);
  if (rc) return rc;
  if (!prm || !psi || !(half_width > 0) || !(lr > 0))
    return wfail(w, ROTGP_EINVAL, "bad arguments");
  if ((rc = load_features(w, n, prm, half_width))) return rc;
  if ((rc = load_targets(w, n, static_cast<const double*>(psi), psi_on_device, half_width)))
    return rc;
  if ((rc = loss_and_grad(w, n, loss))) return rc;
  ++w->t;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)w->t), c2 = 1.f - powf(b2, (float)w->t);
  k_adam<<<blocks_for(w->np), 256, 0, w->s>>>(w->p, w->pb, w->g, w->m, w->v, w->np, lr, b1, b2,
                                              1e-8f, c1, c2);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? ROTGP_OK : wfail(w, ROTGP_ECUDA, "optimiser step", e);
}

}  // extern "C"
