// resident.cu -- a block of split steps of one 2D condensate (complex float)
// in one cooperative launch, the state staying in shared memory.
//
// What bounds a small 2D step.  A 512^2 state is 2 MB: its arithmetic and
// traffic take about a microsecond, but a sweep launch takes 6 to 7 us from
// launch to drain, and a step needs two, with the scale of a whole-grid
// reduction between.  Per step on GB300, two sweep launches against this
// kernel: 128^2 11.7 / 3.1 us, 301 x 215 28 / 3.3 us (odd rows: no TMA
// sweeps), 440^2 14.8 / 4.3 us, 512^2 14.8 / 5.0 us; a step of a real-time
// Omega schedule at 512^2 7.5 us.  What is left at 128^2 is the exchange
// (1,560 of 6,400 cycles) and the length of each thread's own path, a lone
// warp of a scheduler issuing about every fourth cycle; at 512^2 the two
// sweeps take half the time.  Here each CTA (one per SM) keeps one tile of the grid
// for the whole block of steps, with halos of H points on all four sides, and
// a step needs ONE grid-wide exchange:
//   fetch the halos and every tile's share of the norm; H1 on the tile and
//   its halos; the x sweep of the tile's columns on its rows and the H rows
//   above and below; the y sweep of the tile's own points; publish the points
//   that lie in other tiles' halos and the tile's share of the norm.
// The work repeated in halos (1.5 to 3 times the points) costs less than a
// second exchange.
//
// Line solve.  Away from its ends a line's system A y = psi has constant
// coefficients, and its inverse is two geometric tails, so that
//   f_p = al (psi_{p-1} + f_{p-1}),  b_p = be (psi_{p+1} + b_{p+1}),
//   psi'_p = 2 y_p - psi_p = psi_p + (gc psi_p + g2 (f_p + b_p)),
// with the converged Thomas multipliers al, be, G = 1/(A0 + A- be + A+ al),
// g2 = 2 G and gc = 2 G - 2.  The two recurrences do not depend on each
// other, unlike a forward sweep and a back substitution, and both are cut
// off H >= `halo` points away (a relative 1e-9, as in the chunked sweeps).
// The ends, y = 0 at positions 0 and N, are met exactly by a source there
// that makes y vanish: psi_0 = -b_0, psi_N = -f_N.  One thread solves a
// segment of L points of one line from registers; the parenthesis is of the
// order of kappa, so psi itself is rounded once, in real time up or down without
// bias (weights near 1 instead
// doubled their rounding every step: on a 301 x 215 state the error after
// 100 steps was 1.5e-6 of psi, against 2e-7).  Thomas segments (forward from
// H points before to H points after, then back) took 53 cycles a point of
// their dependent chain and tables near the ends, twice the time of this
// form.  The x sweep's lanes are consecutive rows, at an odd pitch; the y sweep's
// lanes are consecutive columns.  Scalar FMAs: a packed FP32x2 FMA holds the pipe
// for two cycles, and the packed complex product needs extra additions.
//
// Exchange.  Every tile adds its share of the norm and a count of one to one
// 64-bit word (the count in the low 8 bits, the share above as a scaled
// integer, so that the sum does not depend on the order and every CTA reads
// the same total), and one thread of each CTA polls it: 1,560 cycles for 152
// CTAs, where polling one flag per CTA took 2,600 to 5,000.  The word is
// never reset; a round's sum is the difference from the last round of the
// same word, and two words alternate.  The scale follows the last total; a
// total out of its range is exchanged again with another scale.  Halo points
// carry the tag of their step in the same 8 bytes (re and the tag, im and
// the tag), so they need no fence and no second flag; planes alternate too: a
// tile can be at most one step ahead of a tile that still reads.  Waits are
// bounded (about 2 s of device time).
//
// No double precision inside the loop: one operation of a warp takes 76
// cycles of its scheduler here, a division 1,500.
#include <algorithm>
#include <cmath>

#include "resident.cuh"
#include "tail_solve.cuh"

namespace rotgp {

namespace {

// Threads of a CTA: segments with halos of 14 hold more registers.
__host__ __device__ constexpr int res_threads(int H) { return H <= 8 ? 512 : 384; }

// ---------------------------------------------------------------- norm shares
// 2^n as a float, n within its range
__device__ __forceinline__ float exp2i(int n) { return __uint_as_float((unsigned)(127 + n) << 23); }
// Shares are integers in units of 2^(ex - kShareBits), a total of 2^ex being
// 2^kShareBits; ex stays where the float factors exist.
constexpr int kShareBits = 45, kExMin = -80, kExMax = 170;
constexpr int kShareTries = 32;  // most repeats of an exchange (12 cross all scales)
constexpr long long kShareMax = 1ll << (kShareBits + 2);
// a compensated sum hi + lo (lo small) in those units, as hi 2^23 + lo in 32-bit
// halves (64-bit conversions run in the double pipe); NaN and values out of
// range become the largest share (fminf drops the NaN)
__device__ __forceinline__ int2 share_of(float hi, float lo, int ex) {
  const float up = exp2i(kShareBits - ex);
  const float q = fminf(hi * up, (float)kShareMax);
  const float top = floorf(q * (1.f / 8388608.f));
  const float rest = fmaf(top, -8388608.f, q) + fminf(fmaxf(lo * up, -8e6f), 8e6f);
  return make_int2((int)top, __float2int_rn(rest));
}
// s = 1/sqrt(n) and s - 1 of n = (h + l) (vh + vl), h and l, vh and vl pairs,
// each right to float rounding (one Newton step from the approximate root).
__device__ __forceinline__ float2 inv_sqrt(float h, float l, float vh, float vl) {
  const float p = h * vh;
  const float e = fmaf(h, vh, -p) + fmaf(h, vl, l * vh);
  const float q = rsqrtf(p), q2 = q * q, q2e = fmaf(q, q, -q2);
  const float r = fmaf(-p, q2, 1.f) - fmaf(p, q2e, e * q2);
  return make_float2(fmaf(0.5f * q, r, q), fmaf(0.5f * q, r, q - 1.f));
}

// ---------------------------------------------------------------- exchange
__device__ __forceinline__ unsigned long long tagged(unsigned tag, float v) {
  return ((unsigned long long)tag << 32) | __float_as_uint(v);
}
__device__ __forceinline__ void st_tagged(unsigned long long* p, unsigned tag, float a, float b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(tagged(tag, a)),
               "l"(tagged(tag, b))
               : "memory");
}
__device__ __forceinline__ ulonglong2 ld_words(const unsigned long long* p) {
  ulonglong2 w;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
               : "=l"(w.x), "=l"(w.y)
               : "l"(p)
               : "memory");
  return w;
}
__device__ __forceinline__ bool has_tag(const ulonglong2& w, unsigned tag) {
  return (unsigned)(w.x >> 32) == tag && (unsigned)(w.y >> 32) == tag;
}
__device__ __forceinline__ float2 untagged(const ulonglong2& w) {
  return make_float2(__uint_as_float((unsigned)w.x), __uint_as_float((unsigned)w.y));
}
// Has this wait run too long?  (asked once per round trip)
struct wait_limit {
  long long t0 = 0;
  int it = 0;
  __device__ __forceinline__ bool over() {
    if ((++it & 1023) != 0) return false;
    const long long t = clock64();
    if (t0 == 0) t0 = t;
    return t - t0 > 4000000000LL;
  }
};
// Add a share and a count of one to a round's word.
__device__ __forceinline__ void post_share(unsigned long long* word, long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(word),
               "l"(((unsigned long long)v << 8) | 1ull)
               : "memory");
}
// Wait until all n shares of a round are in the word; `last` is the word after
// its previous round and becomes the word now.  -1 if the wait gave up.
__device__ __forceinline__ long long poll_total(const unsigned long long* word, int n,
                                                unsigned long long* last) {
  wait_limit lim;
  for (;;) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
    const unsigned long long d = w - *last;
    if ((int)(d & 0xff) == n) {
      *last = w;
      return (long long)(d >> 8);
    }
    if (lim.over()) return -1;
  }
}

// The change of the L own points of a segment from its points w (H before,
// L own, H after), p0 the position of w[0] on a line of N points; at(e): w[e]
// for a run-time e.
template <int H, int L, class AT>
__device__ __forceinline__ void solve_segment(const line_w& k, float2 (&w)[2 * H + L], int p0, int N,
                                              AT at, float2 (&c)[L]) {
  const int z0 = -p0, zN = N - p0;
  if (z0 >= 0) {  // position 0 is w[z0], z0 <= H: the source that makes y_0 = 0
    float2 b = make_float2(0.f, 0.f);
    for (int e = z0 + H; e > z0; --e) b = tail(k.be, at(e), b);
#pragma unroll
    for (int e = 0; e <= H; ++e)
      if (e == z0) w[e] = make_float2(-b.x, -b.y);
  }
  if (zN < 2 * H + L) {  // position N is w[zN], zN > H
    float2 f = make_float2(0.f, 0.f);
    for (int e = zN - H; e < zN; ++e) f = tail(k.al, at(e), f);
#pragma unroll
    for (int e = H + 1; e < 2 * H + L; ++e)
      if (e == zN) w[e] = make_float2(-f.x, -f.y);
  }
  float2 f = make_float2(0.f, 0.f), b = f, fo[L];
#pragma unroll
  for (int e = 0; e < H; ++e) {
    f = tail(k.al, w[e], f);
    b = tail(k.be, w[2 * H + L - 1 - e], b);
  }
#pragma unroll
  for (int i = 0; i < L; ++i) {
    fo[i] = f;
    f = tail(k.al, w[H + i], f);
  }
#pragma unroll
  for (int i = L - 1; i >= 0; --i) {
    c[i] = change(k, w[H + i], fo[i], b);
    b = tail(k.be, w[H + i], b);
  }
}
template <bool IMAG, int H, int L>
__global__ void __launch_bounds__(res_threads(H), 1) k_resident(const res_args a) {
  constexpr int NF = kResPlanes, NT = res_threads(H), NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int2 warp_part[NW];
  // the pending scale is s_pre (1 + s_scale): 1 and its difference from 1, or,
  // far from 1, itself and 0
  __shared__ float s_pre, s_scale;
  __shared__ int s_ex;       // scale of the shares
  __shared__ int s_again;    // the total was out of range: another round
  __shared__ int s_fail;     // a wait gave up
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int PA = a.plan.pa, PB = a.plan.pb, RH = a.plan.rows;
  float2* A = reinterpret_cast<float2*>(smem_raw);     // tile with halos, [row][x]
  float2* D = A + (size_t)RH * PA;                     // real time: H1 increments
  float2* B = D + (IMAG ? 0 : (size_t)RH * PA);        // after the x sweep, own columns
  float2* CX = B + (size_t)RH * PB;                    // x weights [f][row]
  float2* CY = CX + (size_t)NF * RH;                   // y weights [f][column]
  float* VY = reinterpret_cast<float*>(CY + (size_t)NF * a.plan.cols);  // y part of V per row

  const int bx = blockIdx.x % a.plan.tiles_x, by = blockIdx.x / a.plan.tiles_x;
  const int nx = a.nx, ny = a.ny;
  // own points: even starts in x (two points per access)
  const int X0 = (int)((long long)bx * nx / a.plan.tiles_x) & ~1;
  const int X1 = bx + 1 == a.plan.tiles_x ? nx : (int)((long long)(bx + 1) * nx / a.plan.tiles_x) & ~1;
  const int Y0 = (int)((long long)by * ny / a.plan.tiles_y);
  const int Y1 = (int)((long long)(by + 1) * ny / a.plan.tiles_y);
  const int TX = X1 - X0, TY = Y1 - Y0;
  const int SX = (TX + L - 1) / L, SY = (TY + L - 1) / L;
  // rows and columns of the tile inside the grid
  const int r0 = max(0, H - Y0), r1 = min(TY + 2 * H, ny - Y0 + H);
  const int c0 = max(0, H - X0), c1 = min(TX + 2 * H, nx - X0 + H);
  const int cols = a.plan.cols;
  const unsigned epoch = *(volatile unsigned*)&a.sync->epoch;

  const int words = RH * PA * (IMAG ? 1 : 2) + RH * PB;
  for (int i = tid; i < words; i += NT) A[i] = make_float2(0.f, 0.f);
  unsigned long long last[2];  // thread 0: the words after their last rounds
  if (tid == 0) {
    s_fail = 0;
    s_ex = a.ex0;
    const double sc = *a.scale;
    const bool near = sc > 0.5 && sc < 2.0;
    s_pre = near ? 1.f : (float)sc;
    s_scale = near ? (float)(sc - 1.0) : 0.f;
    last[0] = *(volatile unsigned long long*)&a.sync->base[0];
    last[1] = *(volatile unsigned long long*)&a.sync->base[1];
  }
  unsigned round = 0;
  __syncthreads();
  for (int r = r0 + warp; r < r1; r += NW) {
    const float2* src = a.in + (long long)(Y0 - H + r) * nx + (X0 - H);
    for (int c = c0 + lane; c < c1; c += 32) A[r * PA + c] = __ldcg(src + c);
  }
  auto load_weights = [&](int step, int first) {  // by the threads from `first` on
    if (tid < first) return;
    const float2* tx = a.tabx + (long long)step * a.step_x;
    const float2* ty = a.taby + (long long)step * a.step_y;
    for (int f = 0; f < NF; ++f) {
      for (int r = r0 + tid - first; r < r1; r += NT - first)
        CX[f * RH + r] = __ldcg(tx + (size_t)f * ny + (Y0 - H + r));
      for (int c = tid - first; c < TX; c += NT - first)
        CY[f * cols + c] = __ldcg(ty + (size_t)f * nx + X0 + c);
    }
  };
  load_weights(0, 0);
  for (int r = tid; r < RH; r += NT) {
    const float y = (float)(a.y0 + (double)(Y0 - H + r) * a.hy);
    VY[r] = a.hnu2 * y * y;
  }
  const float xs = (float)a.x0, hx = (float)a.hx;
  const float vol_h = (float)a.vol, vol_l = (float)(a.vol - (double)vol_h);
  __syncthreads();

  // Own points in pairs, a row's pairs consecutive, and halo points: the rows
  // above and below in full, then the two sides of the own rows.  Quotients
  // by multiplication: i / n is i * (2^32 / n + 1) >> 32 for i n < 2^32.
  const int pw = (TX + 1) / 2, npairs = pw * TY;
  const unsigned pinv = 0xffffffffu / (unsigned)pw + 1u;
  const int tw = c1 - c0, up = H - r0, top = tw * (up + r1 - H - TY);
  const int left = H - c0, sw = left + c1 - H - TX, nhalo = top + sw * TY;
  const unsigned tinv = 0xffffffffu / (unsigned)tw + 1u;
  const unsigned sinv = 0xffffffffu / (unsigned)max(sw, 2) + 1u;
  auto halo_at = [&](int i, int& r, int& c) {
    if (i < top) {
      const int q = tw > 1 ? (int)__umulhi((unsigned)i, tinv) : i;
      r = q < up ? r0 + q : H + TY + q - up;
      c = c0 + i - q * tw;
    } else {
      const int j = i - top, q = sw > 1 ? (int)__umulhi((unsigned)j, sinv) : j, o = j - q * sw;
      r = H + q;
      c = o < left ? c0 + o : H + TX + o - left;
    }
  };
  // the first KH halo points of each thread, the same every step: asked for
  // before the own points are advanced
  constexpr int KH = 3;
  const int words0 = 2 * ((Y0 - H) * nx + (X0 - H));  // word of the tile's corner (ny nx < 2^28)
  int hs[KH];       // place in the tile, -1: none
  int hw[KH];       // word in the exchange plane
  float hx0[KH], hvy[KH];
#pragma unroll
  for (int q = 0; q < KH; ++q) {
    hs[q] = -1;
    if (tid + q * NT >= nhalo) continue;
    int r, c;
    halo_at(tid + q * NT, r, c);
    hs[q] = r * PA + c;
    hw[q] = words0 + 2 * (r * nx + c);
    hx0[q] = fmaf((float)(X0 - H + c), hx, xs);
    hvy[q] = VY[r];
  }
  // and its first pair of own points
  int os = -1;
  float ox = 0.f, ovy = 0.f;
  bool o2 = false;
  if (tid < npairs) {
    const int q = pw > 1 ? (int)__umulhi((unsigned)tid, pinv) : tid, c = 2 * (tid - q * pw);
    os = (H + q) * PA + H + c;
    ox = fmaf((float)(X0 + c), hx, xs);
    ovy = VY[H + q];
    o2 = c + 1 < TX;
  }

  for (int step = 0; step < a.nsteps; ++step) {
    const bool final = step + 1 == a.nsteps;
    const unsigned tag_in = epoch + (unsigned)step, tag = tag_in + 1u;
    // ---- H1 on the tile: own points, while the first halo points arrive from
    // their owners (step 0: all from the state), then the halos
    const float pre = s_pre, sm1 = s_scale, sc = 1.f + sm1, gs = IMAG ? a.g * sc * sc : a.g;
    const unsigned long long* xin = a.xbuf + (size_t)(tag_in & 1) * a.xplane;
    auto h1 = [&](float2 p, int at, float x, float vy) {
      p = make_float2(pre * p.x, pre * p.y);
      if (IMAG) {
        A[at] = damp(p, -a.dt * fmaf(gs, fmaf(p.x, p.x, p.y * p.y), fmaf(a.hgam2 * x, x, vy)),
                     sm1);
      } else {
        // the advanced value rounded, and what the rounding left out (the x
        // sweep adds it to the change of its points)
        const float2 s = make_float2(fmaf(sm1, p.x, p.x), fmaf(sm1, p.y, p.y));
        const float t = a.dt * fmaf(gs, fmaf(s.x, s.x, s.y * s.y), fmaf(a.hgam2 * x, x, vy));
        rotate_split(s, t, &A[at], &D[at]);
      }
    };
    ulonglong2 v[KH];
    if (step > 0) {
#pragma unroll
      for (int q = 0; q < KH; ++q)
        if (hs[q] >= 0) v[q] = ld_words(xin + hw[q]);
    }
    if (os >= 0) {
      const float2 p0 = A[os], p1 = A[os + 1];
      h1(p0, os, ox, ovy);
      if (o2) h1(p1, os + 1, ox + hx, ovy);
    }
#pragma unroll 1
    for (int i = tid + NT; i < npairs; i += NT) {
      const int q = (int)__umulhi((unsigned)i, pinv), c = 2 * (i - q * pw);
      const int at = (H + q) * PA + H + c;
      const float x = fmaf((float)(X0 + c), hx, xs), vy = VY[H + q];
      const float2 p0 = A[at], p1 = A[at + 1];
      h1(p0, at, x, vy);
      if (c + 1 < TX) h1(p1, at + 1, x + hx, vy);
    }
    // the words are looked at only here (a look waits for the load)
    wait_limit lim;
#pragma unroll
    for (int q = 0; q < KH; ++q) {
      if (hs[q] < 0) continue;
      while (step > 0 && !has_tag(v[q], tag_in)) {
        if (lim.over()) {
          s_fail = 1;
          break;
        }
        v[q] = ld_words(xin + hw[q]);
      }
      h1(step > 0 ? untagged(v[q]) : A[hs[q]], hs[q], hx0[q], hvy[q]);
    }
#pragma unroll 1
    for (int i = tid + KH * NT; i < nhalo; i += NT) {
      int r, c;
      halo_at(i, r, c);
      const int at = r * PA + c;
      float2 p = A[at];
      if (step > 0) {
        ulonglong2 w = ld_words(xin + words0 + 2 * (r * nx + c));
        while (!has_tag(w, tag_in)) {
          if (lim.over()) {
            s_fail = 1;
            break;
          }
          w = ld_words(xin + words0 + 2 * (r * nx + c));
        }
        p = untagged(w);
      }
      h1(p, at, fmaf((float)(X0 - H + c), hx, xs), VY[r]);
    }
    __syncthreads();
    if (s_fail) {
      if (tid == 0) atomicOr(a.flags, 8);
      return;
    }

    // ---- the sweeps, one code for both: x, A -> B on rows r0 .. r1 and own
    // columns; y, B -> A's own points and the exchange plane (and the state).
    // The loop body stays within the 32 KB that the instruction cache serves
    // at full rate; the step unrolled (two sweeps with their own code, H1 on
    // eight points at once, the argument reduction of sincosf inlined) took 4
    // to 7 cycles an instruction.
    acc_t<float> acc;
    auto sum_of = [](float2 psi, float2 c) {
      return IMAG ? make_float2(psi.x + c.x, psi.y + c.y) : add_dithered(psi, c);
    };
#pragma unroll 1
    for (int ax = 0; ax < 2; ++ax) {
      const bool y = ax == 1;
      const int nl = y ? TX : r1 - r0, segs = y ? SY : SX;   // lines, segments of each
      const int N = y ? ny : nx, P0 = (y ? Y0 : X0) - H;
      const int es = y ? PB : 1, ls = y ? 1 : PA;            // strides of points, lines
      const float2* src = y ? B : A + r0 * PA;
      const float2* wts = y ? CY : CX + r0;
      const int fs = y ? cols : RH;
      const unsigned ninv = 0xffffffffu / (unsigned)nl + 1u;
#pragma unroll 1
      for (int t = tid; t < nl * segs; t += NT) {
        const int seg = nl > 1 ? (int)__umulhi((unsigned)t, ninv) : t;
        const int l = t - seg * nl, e0 = seg * L;
        const float2* line = src + l * ls + e0 * es;
        const line_w k{wts[l], wts[fs + l], wts[2 * fs + l], wts[3 * fs + l]};
        float2 w[2 * H + L], c[L];
        {
          const float2* q = line;
#pragma unroll
          for (int e = 0; e < 2 * H + L; ++e, q += es) w[e] = *q;
        }
        solve_segment<H, L>(k, w, P0 + e0, N, [&](int e) { return line[e * es]; }, c);
        if (P0 + e0 + H == 0) w[H] = c[0] = make_float2(0.f, 0.f);  // the edge itself
        if (!y) {
          float2* o = B + (r0 + l) * PB + e0;
#pragma unroll
          for (int i = 0; i < L; ++i) {
            if (!IMAG) {
              const float2 r = D[(r0 + l) * PA + e0 + H + i];
              c[i].x += r.x;
              c[i].y += r.y;
            }
            o[i] = sum_of(w[H + i], c[i]);
          }
          continue;
        }
        float2* own = A + (H + e0) * PA + H + l;
        size_t g = (size_t)(Y0 + e0) * nx + X0 + l;
        unsigned long long* xout = a.xbuf + (size_t)(tag & 1) * a.xplane;
        const bool side = l < H || l >= TX - H;
        const int n = TY - e0;
#pragma unroll
        for (int i = 0; i < L; ++i, own += PA, g += nx) {
          const float2 o = sum_of(w[H + i], c[i]);
          const bool in = i < n;
          acc.add(in ? fmaf(o.x, o.x, o.y * o.y) : 0.f);
          if (in) *own = o;
          if (in && (side || e0 + i < H || i >= n - H))  // some tile's halo
            st_tagged(xout + 2 * g, tag, o.x, o.y);
          if (in && final) a.out[g] = o;
        }
      }
      if (!y) __syncthreads();
    }
    // ---- the norm: this tile's share, then the total and the pending scale
    for (int tries = 0;; ++tries) {
      int2 v = share_of(acc.s, -acc.c, s_ex);
      v.x = __reduce_add_sync(0xffffffffu, v.x);
      v.y = __reduce_add_sync(0xffffffffu, v.y);
      if (lane == 0) warp_part[warp] = v;
      __syncthreads();
      if (tid == 0) {
        // (a warp's sums stay below 2^30, those of 512 threads pass 2^31)
        long long hi = 0, lo = 0;
#pragma unroll
        for (int i = 0; i < NW; ++i) hi += warp_part[i].x, lo += warp_part[i].y;
        long long t = max(0ll, (hi << 23) + lo);
        unsigned long long* word = &a.sync->word[round & 1][0];
        post_share(word, min(t, kShareMax));
        t = poll_total(word, gridDim.x, &last[round & 1]);
        if (t < 0) {
          s_fail = 1;
          t = 1ll << kShareBits;
        }
        const int ex = s_ex, bits = 64 - __clzll(t);
        // the scale that this total asks for
        const int next = t == 0 ? ex - 40 : t >= kShareMax ? ex + 24 : ex + bits - kShareBits - 1;
        s_ex = max(kExMin, min(kExMax, next));
        s_again = (t < (1ll << (kShareBits - 9)) || t >= kShareMax) && s_ex != ex &&
                  tries < kShareTries;
        const float h = (float)(int)(t >> 24) * 16777216.f, l = (float)(int)(t & 0xffffff);
        const float dn = exp2i(ex - kShareBits);
        const float2 sc = inv_sqrt(h * dn, l * dn, vol_h, vol_l);
        const bool use = IMAG && t > 0 && isfinite(sc.x), near = sc.x > 0.5f && sc.x < 2.f;
        s_pre = use && !near ? sc.x : 1.f;
        s_scale = use && near ? sc.y : 0.f;
        if (final && blockIdx.x == 0 && !s_again && !s_fail) {
          const double n = ldexp((double)t, ex - kShareBits) * a.vol;
          const bool fine = t > 0 && t < kShareMax;
          *a.norm = fine ? n : nan("");
          *a.scale = IMAG && fine ? 1.0 / sqrt(n) : 1.0;
          if (!fine) atomicOr(a.flags, 1);
          // every CTA has posted its last round: all have read these
          a.sync->epoch = tag;
          a.sync->base[0] = last[0];
          a.sync->base[1] = last[1];
        }
      }
      if (a.step_x && !final) load_weights(step + 1, 32);  // a schedule's next tables
      __syncthreads();
      ++round;
      if (!s_again || s_fail) break;
    }
    if (s_fail) {
      if (tid == 0) atomicOr(a.flags, 8);
      return;
    }
  }
}

template <bool IMAG, int H, int L>
cudaError_t launch_r(const res_args& a, cudaStream_t s) {
  auto fn = k_resident<IMAG, H, L>;
  cudaError_t e = allow_smem_bytes((const void*)fn, (int)a.plan.smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<res_args*>(&a)};
  return cudaLaunchCooperativeKernel((const void*)fn, dim3(a.plan.tiles_x * a.plan.tiles_y),
                                     dim3(res_threads(H)), args, a.plan.smem, s);
}

// The weights of one line per thread: the converged multiplier m of the Thomas
// recursion, the root of A- A+ m^2 - A0 m + 1 = 0 near 1/A0, in float and
// then by one Newton step to double rounding (the step's division in float is
// enough); G = 1/(A0 - 2 A- A+ m) likewise.  Divisions in double would take
// 1,500 cycles each.
struct dc {
  double x, y;
};
__device__ __forceinline__ dc dmul(dc a, dc b) {
  return {fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x)};
}
__device__ __forceinline__ float2 fmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 finv(float2 a) {
  const float r = 1.f / fmaf(a.x, a.x, a.y * a.y);
  return make_float2(a.x * r, -a.y * r);
}
__device__ __forceinline__ float2 tof(dc a) { return make_float2((float)a.x, (float)a.y); }

__global__ void __launch_bounds__(32) k_res_tables(float2* tab, int nlines, int iters, axis_coef co,
                                                   res_omegas om) {
  const int l = blockIdx.x * 32 + threadIdx.x;
  if (l >= nlines) return;
  tab += (size_t)blockIdx.y * kResPlanes * nlines + l;
  const double u = (co.u0 + (double)l * co.du) * om.v[blockIdx.y];
  const dc kap{co.kap_re, co.kap_im}, tau{co.tau_re * u, co.tau_im * u};
  const dc a0{1.0 + 2.0 * kap.x, 2.0 * kap.y};
  const dc am{tau.x - kap.x, tau.y - kap.y}, ap{-kap.x - tau.x, -kap.y - tau.y};
  const dc aa = dmul(am, ap);
  const float2 a0f = tof(a0), aaf = tof(aa);
  float2 mf = finv(a0f);
  for (int i = 0; i < iters; ++i) {
    const float2 t = fmul(aaf, mf);
    mf = finv(make_float2(a0f.x - t.x, a0f.y - t.y));
  }
  dc m{mf.x, mf.y};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const dc am2 = dmul(aa, m);                      // A- A+ m
    const dc q{am2.x - a0.x, am2.y - a0.y}, r = dmul(q, m);
    const float2 res = make_float2((float)(r.x + 1.0), (float)r.y);
    const float2 slope = make_float2((float)(am2.x + q.x), (float)(am2.y + q.y));
    const float2 dm = fmul(res, finv(slope));
    m.x -= dm.x;
    m.y -= dm.y;
  }
  const dc al = dmul(am, m), be = dmul(ap, m), t = dmul(aa, m);
  const dc D{a0.x - 2.0 * t.x, a0.y - 2.0 * t.y};
  const float2 gf = finv(tof(D));
  dc g{gf.x, gf.y};
  const dc e = dmul(D, g);                           // g (2 - D g)
  g = dmul(g, {2.0 - e.x, -e.y});
  tab[0] = make_float2((float)-al.x, (float)-al.y);
  tab[(size_t)nlines] = make_float2((float)-be.x, (float)-be.y);
  tab[(size_t)2 * nlines] = make_float2((float)(2.0 * g.x), (float)(2.0 * g.y));
  tab[(size_t)3 * nlines] = make_float2((float)(2.0 * g.x - 2.0), (float)(2.0 * g.y));
}

}  // namespace

bool res_make_plan(int nx, int ny, int halo, bool imag, int sm_count, size_t smem_limit,
                   res_plan* best) {
  // tails cut off after H points leave out the power H + 1 of the decay; the
  // chunked sweeps' halo is the power that is below 1e-9, plus one
  const int H = halo <= 6 ? 4 : halo <= 8 ? 6 : 14;
  // the ends' sources want the ends further apart than a tail reaches
  if (halo > 16 || nx < 2 * H + 2 || ny < 2 * H + 2 || (long long)nx * ny > (1 << 28)) return false;
  const int most = std::min(sm_count, kResMaxCtas), NF = kResPlanes;
  double best_cost = 0;
  bool found = false;
  for (int L : {4, 8})
    for (int tx = 1; tx <= most && tx <= nx / (H + 2); ++tx)
      for (int ty = 1; tx * ty <= most && ty <= ny / H; ++ty) {
        // largest tile (starts rounded down to even in x)
        const int TX = (nx + tx - 1) / tx + 1, TY = (ny + ty - 1) / ty;
        const int SX = (TX + L - 1) / L, SY = (TY + L - 1) / L;
        auto pitch = [](int w) { return w | 1; };  // odd: rows on distinct banks
        res_plan p;
        p.H = H;
        p.L = L;
        p.tiles_x = tx;
        p.tiles_y = ty;
        p.pa = pitch(SX * L + 2 * H + 1);
        p.pb = pitch(SX * L);
        p.rows = SY * L + 2 * H;
        p.cols = TX;
        p.smem = ((size_t)p.rows * p.pa * (imag ? 1 : 2) + (size_t)p.rows * p.pb +
                  (size_t)NF * (p.rows + TX)) * 8 + (size_t)p.rows * 4;
        if (p.smem > smem_limit || (TX + 2 * H + 1) / 2 * (TY + 2 * H) >= 32768) continue;
        // cycles of the busiest tile: instructions over what its warps issue
        // (a lone warp of a scheduler issues every fourth cycle)
        const double seg = 12.0 * (H + L) + 24.0 * L + 2.0 * H + 40.0;
        auto phase = [&](double tasks) {
          const double warps = std::ceil(tasks / 32.0), at_once = std::min(warps, res_threads(H) / 32.0);
          return warps * seg / std::min(2.8, at_once / 4.0 * 0.7 + 0.3);
        };
        const double cost = (TX + 2.0 * H) * (TY + 2.0 * H) * (imag ? 0.45 : 0.6) +
                            0.25 * (phase((TY + 2.0 * H) * SX) + phase((double)TX * SY));
        if (!found || cost < best_cost) {
          found = true;
          best_cost = cost;
          *best = p;
        }
      }
  return found;
}

cudaError_t launch_resident(bool imag, const res_args& a, cudaStream_t s) {
  const int H = a.plan.H, L = a.plan.L;
  if (H == 4 && L == 4) return imag ? launch_r<true, 4, 4>(a, s) : launch_r<false, 4, 4>(a, s);
  if (H == 4 && L == 8) return imag ? launch_r<true, 4, 8>(a, s) : launch_r<false, 4, 8>(a, s);
  if (H == 6 && L == 4) return imag ? launch_r<true, 6, 4>(a, s) : launch_r<false, 6, 4>(a, s);
  if (H == 6 && L == 8) return imag ? launch_r<true, 6, 8>(a, s) : launch_r<false, 6, 8>(a, s);
  if (H == 14 && L == 4) return imag ? launch_r<true, 14, 4>(a, s) : launch_r<false, 14, 4>(a, s);
  if (H == 14 && L == 8) return imag ? launch_r<true, 14, 8>(a, s) : launch_r<false, 14, 8>(a, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_res_tables(float2* tab, int nlines, int iters, const axis_coef& co,
                              const res_omegas& om, int nsteps, cudaStream_t s) {
  const dim3 grid((unsigned)((nlines + 31) / 32), (unsigned)nsteps);
  k_res_tables<<<grid, 32, 0, s>>>(tab, nlines, iters, co, om);
  return cudaGetLastError();
}

}  // namespace rotgp
