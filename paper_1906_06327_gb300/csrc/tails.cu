// tails.cu -- complex-float sweeps in shared-memory tiles by the two-tail line
// solve (resident.cu): lines whose tails are too long for the chunked TMA
// sweeps (halo above 16 points), and rows that are not 16-byte multiples.
//
// A CTA holds a tile of 32 lines: up to 8 warps of L own points each, and H
// points on both sides.  A lane is a line; a warp runs both tails over the H
// points before and after its own and then its own L points from shared
// memory, with the forward tail of its own points in registers.  The tile is
// read from memory once and written once, nothing waits on another warp
// between load and result (the exact partition solve meets at eight barriers,
// two of them cluster-wide, and was waiting at one 44% of the time), and
// several CTAs per SM overlap their loads and solves.  The ends of a line are
// met by sources in the tile (psi_0 = -b_0, psi_N = -f_N).
//
// What bounds it: instructions, 12 (H + L) / L + 12 a point and the loads of
// both tails, with H1 in x; FMAs that read three registers take 1.7 cycles.
// GB300, one sweep, before / after: 4096^2 (halo 24) x 226 / 92 us, y 178 / 85
// us (exact partition solve in clusters of 8 CTAs, 153 and 160 us with its own
// passes trimmed); 255 x 256 x 128 imaginary time x 74 / 55, y 57 / 54, z 66 / 64
// us, real time x 113 / 60 us.
#include <algorithm>
#include <type_traits>

#include "pairsum.cuh"
#include "tail_solve.cuh"
#include "tails.cuh"

namespace rotgp {

namespace {

constexpr int kTailWarps = 8;

// The end sources of the tile's 32 lines: thread l < 32, line l; P0 - H the
// position of the tile's first point, n its points.
template <class AT>
__device__ __forceinline__ void end_sources(const line_w& k, int first, int n, int N, int H, AT at) {
  const int z0 = -first, zN = N - first;
  float2 b = make_float2(0.f, 0.f), f = b;
  const bool has0 = z0 >= 0, hasN = zN < n;
  if (has0)
    for (int e = min(z0 + H, n - 1); e > z0; --e) b = tail(k.be, at(e), b);
  if (hasN)
    for (int e = max(zN - H, 0); e < zN; ++e) f = tail(k.al, at(e), f);
  if (has0) at(z0) = make_float2(-b.x, -b.y);
  if (hasN) at(zN) = make_float2(-f.x, -f.y);
}

// A warp's L own points of its lane's line: at(e), e = 0 .. 2 H + L - 1, the
// points from H before the own ones; res(i, psi, change).
template <int L, class AT, class RES>
__device__ __forceinline__ void solve_own(const line_w& k, int H, AT at, RES res) {
  float2 f = make_float2(0.f, 0.f), b = f, fo[L];
#pragma unroll 4
  for (int e = 0; e < H; ++e) {
    f = tail(k.al, at(e), f);
    b = tail(k.be, at(2 * H + L - 1 - e), b);
  }
#pragma unroll
  for (int i = 0; i < L; ++i) {
    fo[i] = f;
    f = tail(k.al, at(H + i), f);
  }
#pragma unroll
  for (int i = L - 1; i >= 0; --i) {
    const float2 w = at(H + i);
    fo[i] = res(i, w, change(k, w, fo[i], b));
    b = tail(k.be, w, b);
  }
  res.done(fo);
}

__device__ __forceinline__ line_w line_weights(const float2* tab, int n, int line) {
  return {__ldg(tab + line), __ldg(tab + n + line), __ldg(tab + 2 * (size_t)n + line),
          __ldg(tab + 3 * (size_t)n + line)};
}

// Block sum of a compensated sum, then the last block's total, norm, pending
// scale and flag, as norm_epilogue (sweep_common.cuh), with float pairs up to
// the block's partial.
__device__ __forceinline__ void tail_norm(fpair v, const tail_args& a) {
  __shared__ fpair ws[kTailWarps];
  __shared__ double wd[kTailWarps];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = sum_add(v, sum_xor(v, o));
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    fpair s = ws[0];
    for (int w = 1; w < nw; ++w) s = sum_add(s, ws[w]);
    a.partials[blockIdx.x] = sum_value(s);
    __threadfence();
    last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) s += __ldcg(&a.partials[i]);
  s = warp_sum(s);
  if (lane == 0) wd[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0;
    for (int w = 0; w < nw; ++w) tot += wd[w];
    const double n = tot * a.vol;
    const bool fine = n > 0.0 && isfinite(n);
    *a.norm_out = n;
    if (!fine) atomicOr(a.flags, 1);
    *a.scale_out = fine && a.imag ? 1.0 / sqrt(n) : 1.0;
    *a.counter = 0u;
  }
}

// ---------------------------------------------------------------- columns
template <int L, bool REDUCE, bool IMAG>
__global__ void __launch_bounds__(32 * kTailWarps, 2) k_tail_s(const tail_args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* T = reinterpret_cast<float2*>(smem_raw);  // [point][lane]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x;
  const int H = a.H, N = a.len, own = a.sh.nw * L, n = own + 2 * H;
  const int groups = (a.nx + 31) / 32;
  unsigned b = blockIdx.x;
  const int x0 = (int)(b % groups) * 32;
  b /= groups;
  const int P0 = (int)(b % (unsigned)a.sh.tiles) * own;
  const long long tr = b / (unsigned)a.sh.tiles;
  const long long stride = a.axis == 1 ? a.nx : a.lines;
  const long long base = tr * (a.axis == 1 ? (long long)a.nx * a.len : (long long)a.nx);
  const float2* in = a.in + base + x0;
  if (a.nx % 2 == 0 && x0 + 32 <= a.nx) {
    for (int u = tid; u < n * 16; u += NT) {
      const int e = u >> 4, c = (u & 15) * 2, p = P0 - H + e;
      if (p >= 0 && p < N)
        cp_async<16>(T + e * 32 + c, in + p * stride + c);
      else
        *reinterpret_cast<float4*>(T + e * 32 + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  } else {
    for (int u = tid; u < n * 32; u += NT) {
      const int e = u >> 5, p = P0 - H + e;
      T[u] = p >= 0 && p < N && x0 + lane < a.nx ? in[p * stride + lane] : make_float2(0.f, 0.f);
    }
  }
  const bool act = x0 + lane < a.nx;
  const line_w k = line_weights(a.tab, a.tlines, a.axis == 1 && act ? x0 + lane : 0);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  if (P0 - H <= 0 || P0 - H + n > N) {
    if (warp == 0) end_sources(k, P0 - H, n, N, H, [&](int e) -> float2& { return T[e * 32 + lane]; });
    __syncthreads();
  }
  const int q0 = P0 + warp * L;  // first own position
  float2* out = a.out + base + x0 + lane + q0 * stride;
  const float2* t = T + warp * L * 32 + lane;
  acc_t<float> acc;
  struct result {
    float2* out;
    long long stride;
    acc_t<float>* acc;
    int left;     // own positions inside the line
    bool act, edge;
    __device__ __forceinline__ float2 operator()(int i, float2 w, float2 c) {
      if (i == 0 && edge) return make_float2(0.f, 0.f);
      return IMAG ? make_float2(w.x + c.x, w.y + c.y) : add_dithered(w, c);
    }
    __device__ __forceinline__ void done(const float2 (&o)[L]) {
#pragma unroll
      for (int i = 0; i < L; ++i) {
        if (!act || i >= left) continue;
        out[i * stride] = o[i];
        if (REDUCE) acc->add(fmaf(o[i].x, o[i].x, o[i].y * o[i].y));
      }
    }
  };
  if (q0 < N) {
    result r{out, stride, &acc, N - q0, act, q0 == 0};
    solve_own<L>(k, H, [&](int e) { return t[e * 32]; }, r);
  }
  if (REDUCE) tail_norm({acc.s, -acc.c}, a);
}

// ---------------------------------------------------------------- rows
template <int L, bool IMAG>
__global__ void __launch_bounds__(32 * kTailWarps, 2) k_tail_x(const tail_args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = blockDim.x >> 5;
  const int H = a.H, N = a.len, own = a.sh.nw * L, n = own + 2 * H, W = n | 1, WD = own | 1;
  float2* T = reinterpret_cast<float2*>(smem_raw);  // [row][point]
  float2* D = T + 32 * W;                           // real time: what the rounding of H1 left out
  const long long rows = a.lines;
  const int P0 = (int)(blockIdx.x % (unsigned)a.sh.tiles) * own;
  const long long row0 = (long long)(blockIdx.x / (unsigned)a.sh.tiles) * 32;
  const int first = P0 - H;
  for (int r = warp; r < 32; r += NW) {
    const float2* src = a.in + (row0 + r) * N + first;
    float2* dst = T + r * W;
    const bool ok = row0 + r < rows;
    for (int e = lane; e < n; e += 32) {
      const int p = first + e;
      if (ok && p >= 0 && p < N)
        cp_async<8>(dst + e, src + e);
      else
        dst[e] = make_float2(0.f, 0.f);
    }
  }
  const long long myrow = row0 + lane;
  const int j = myrow < rows ? (int)(myrow % a.ny) : 0;
  const line_w k = line_weights(a.tab, a.tlines, j);
  const float sc = (float)*a.scale, sm1 = (float)(*a.scale - 1.0), gs = IMAG ? a.g * sc * sc : a.g;
  cp_async_commit();
  // the y and z part of the potential of the rows this warp loaded: lane i's row
  // warp + i NW
  float vyz = 0.f;
  {
    const long long r = row0 + warp + lane * NW;
    if (lane * NW + warp < 32 && r < rows) {
      const float y = (float)(a.y0 + (double)(r % a.ny) * a.hy), z = (float)(a.z0 + (double)(r / a.ny) * a.hz);
      vyz = fmaf(a.hnu2 * y, y, a.hlam2 * z * z);
    }
  }
  cp_async_wait<0>();
  __syncwarp();
  // H1 on the points this warp loaded (far from 1, the scale goes first)
  const bool near = sc > 0.5f && sc < 2.f;
  const float pre = near ? 1.f : sc, m1 = near ? sm1 : 0.f;
  for (int r = warp, i = 0; r < 32; r += NW, ++i) {
    const float vy = __shfl_sync(0xffffffffu, vyz, i);
    float2* row = T + r * W;
    for (int e = lane; e < n; e += 32) {
      float2 p = row[e];
      p = make_float2(pre * p.x, pre * p.y);
      const float x = fmaf((float)(first + e), a.hx, a.x0);
      const float pot = fmaf(a.hgam2 * x, x, vy);
      if (IMAG) {
        const float gg = near ? gs : a.g;
        row[e] = damp(p, -a.dt * fmaf(gg, fmaf(p.x, p.x, p.y * p.y), pot), m1);
      } else {
        const float2 v = make_float2(fmaf(m1, p.x, p.x), fmaf(m1, p.y, p.y));
        float2 w, rest;
        rotate_split(v, a.dt * fmaf(a.g, fmaf(v.x, v.x, v.y * v.y), pot), &w, &rest);
        row[e] = w;
        if (e >= H && e < H + own) D[r * WD + e - H] = rest;
      }
    }
  }
  __syncthreads();
  if (first <= 0 || first + n > N) {
    if (warp == 0) end_sources(k, first, n, N, H, [&](int e) -> float2& { return T[lane * W + e]; });
    __syncthreads();
  }
  const float2* t = T + lane * W + warp * L;
  struct result {
    const float2* rest;
    float2* keep;
    bool edge;
    __device__ __forceinline__ float2 operator()(int i, float2 w, float2 c) {
      if (!IMAG) c = make_float2(c.x + rest[i].x, c.y + rest[i].y);
      if (i == 0 && edge) return make_float2(0.f, 0.f);
      return IMAG ? make_float2(w.x + c.x, w.y + c.y) : add_dithered(w, c);
    }
    __device__ __forceinline__ void done(const float2 (&r)[L]) {
      // every warp has read its neighbours' points: the results take their place
      __syncthreads();
#pragma unroll
      for (int i = 0; i < L; ++i) keep[i] = r[i];
    }
  };
  result r{D + lane * WD + warp * L, T + lane * W + H + warp * L, P0 + warp * L == 0};
  solve_own<L>(k, H, [&](int e) { return t[e]; }, r);
  __syncthreads();
  for (int q = warp; q < 32; q += NW) {
    if (row0 + q >= rows) break;
    float2* dst = a.out + (row0 + q) * N + P0;
    const float2* src = T + q * W + H;
    for (int e = lane; e < own && P0 + e < N; e += 32) dst[e] = src[e];
  }
}

}  // namespace

bool tail_plan(int axis, int N, int nx, long long lines, int halo, bool imag, size_t smem_limit,
               tail_shape* s) {
  if (halo >= N) return false;
  // tails cut off after H points leave out the power H + 1 (resident.cu)
  const int H = std::max(1, halo - 2);
  // long tails are run over more own points
  int L = H > 12 ? 32 : 16;
  if (axis == 0 && !imag) L = 16;  // (the rest of H1 takes the room)
  const int tiles = (N + kTailWarps * L - 1) / (kTailWarps * L);
  s->L = L;
  s->nw = std::min(kTailWarps, (N + tiles * L - 1) / (tiles * L));
  s->tiles = (N + s->nw * L - 1) / (s->nw * L);
  const int own = s->nw * L, n = own + 2 * H;
  s->smem = axis == 0 ? 32 * (size_t)((n | 1) + (imag ? 0 : (own | 1))) * 8 : (size_t)n * 32 * 8;
  s->blocks = axis == 0 ? (lines + 31) / 32 * s->tiles
                        : (long long)((nx + 31) / 32) * s->tiles * (lines / nx);
  return s->smem <= smem_limit && s->blocks < (1ll << 31);
}

cudaError_t launch_tail_x(bool imag, const tail_args& a, cudaStream_t s) {
  auto fn = !imag ? k_tail_x<16, false> : a.sh.L == 32 ? k_tail_x<32, true> : k_tail_x<16, true>;
  const cudaError_t e = allow_smem_bytes((const void*)fn, (int)a.sh.smem);
  if (e != cudaSuccess) return e;
  fn<<<(unsigned)a.sh.blocks, 32 * a.sh.nw, a.sh.smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_tail_s(bool reduce, const tail_args& a, cudaStream_t s) {
  auto pick = [&](auto im) {
    constexpr bool IMAG = decltype(im)::value;
    return a.sh.L == 32 ? (reduce ? k_tail_s<32, true, IMAG> : k_tail_s<32, false, IMAG>)
                        : (reduce ? k_tail_s<16, true, IMAG> : k_tail_s<16, false, IMAG>);
  };
  auto fn = a.imag ? pick(std::true_type{}) : pick(std::false_type{});
  const cudaError_t e = allow_smem_bytes((const void*)fn, (int)a.sh.smem);
  if (e != cudaSuccess) return e;
  fn<<<(unsigned)a.sh.blocks, 32 * a.sh.nw, a.sh.smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace rotgp
