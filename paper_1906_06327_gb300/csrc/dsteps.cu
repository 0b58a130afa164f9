// dsteps.cu -- imaginary-time steps in complex double.
//
// What bounds them.  The double pipe: a warp's fused multiply-add holds its
// scheduler's for 64 to 76 cycles whether its neighbours depend on it or not,
// 1/64 of the float rate, so the time of a sweep is its double operations
// over the schedulers that have a warp, and latency, memory and occupancy
// hardly matter.  The chunked sweeps (sweep_x.cu, sweep_s.cu) spend 24
// operations a point, more in halos, and gave their work to as many warps as
// there are groups of 32 lines: 4 of 608 schedulers busy on a 128^2 state,
// 256 on 256 x 256 x 32.
//
// Line solve, 18 operations a point.  Away from the start of a line the
// Thomas factors are constant, m = 1 + mu the multiplier, al = -m A-, be = -m
// A+; with the multiplier taken out of both recurrences,
//   t_p = al e_{p-1},  e_p = psi_p + t_p           (forward)
//   c_p = t_p + be u_{p+1},  u_p = psi_p + c_p     (back)
//   psi'_p = 2 m u_p - psi_p = psi_p + 2 (c_p + mu u_p).
// t, c and mu u are of the order of kappa, so psi itself is rounded once (2 m
// u - psi as it stands takes 12 operations and three times the rounding error
// of the four-term form of the chunked sweeps).  The end of the line is exact
// as it stands (u_N = 0).  At its start the recurrences solve the line
// continued to the left; subtracting u_0 al^p, the solution of the homogeneous
// system that does so, makes the value at position 0 vanish (lines longer
// than a tail).  Tails are cut off at the halo of the chunked sweeps (1e-17).
//
// Rows (x): the points of a line are spread over the lanes, P consecutive
// ones each, and the carries follow from a truncated scan over the lanes (two
// passes of each recurrence: 30 operations a point, but no halo in which H1
// would be repeated).  Columns (y, z): a lane walks its own line, one segment
// with its halos.  H1: the exponential is a Taylor series of degree 9 where
// the step's exponent is below 1/16.
//
// A 2D state (of up to 512 points in x, 1,024 in y) runs a whole block of steps in one
// cooperative launch, a line at a time on all four schedulers of an SM, with a
// grid-wide exchange after each sweep (one 64-bit word pair that takes every CTA's count and
// share of the norm, as in resident.cu, here in 85-bit integers).
//
// GB300, before / after: 128^2 step 134 / 11.9 us; 256 x 256 x 32 step 1,120 /
// 494 us (x 474 / 235, y 249 / 134, z 390 / 125); distance from 64-bit values
// of another program after 100 steps at 128^2 4.5e-15 / 3.6e-15.
#include <algorithm>

#include "dsteps.cuh"
#include "sweep_common.cuh"

namespace rotgp {

namespace {

typedef double2 dz;
__device__ __forceinline__ dz zero2d() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ dz zmul(dz k, dz b) {
  return make_double2(fma(k.x, b.x, -(k.y * b.y)), fma(k.x, b.y, k.y * b.x));
}
__device__ __forceinline__ dz zadd(dz a, dz b) { return make_double2(a.x + b.x, a.y + b.y); }
// a + k b
__device__ __forceinline__ dz zfma(dz k, dz b, dz a) {
  return make_double2(fma(k.x, b.x, fma(-k.y, b.y, a.x)), fma(k.x, b.y, fma(k.y, b.x, a.y)));
}
// psi + 2 (c + mu u)
__device__ __forceinline__ dz zout(dz psi, dz c, dz mu, dz u) {
  const dz w = zfma(mu, u, c);
  return make_double2(fma(2.0, w.x, psi.x), fma(2.0, w.y, psi.y));
}
__device__ __forceinline__ dz shfl_d(dz v, int src, bool use) {
  const dz r = make_double2(__shfl_sync(0xffffffffu, v.x, src & 31),
                            __shfl_sync(0xffffffffu, v.y, src & 31));
  return use ? r : zero2d();
}

// e^u
__device__ __noinline__ double exp_far(double u) { return exp(u); }
__device__ __forceinline__ double exp_near(double u) {
  double p = fma(u, 1.0 / 362880.0, 1.0 / 40320.0);
  p = fma(u, p, 1.0 / 5040.0);
  p = fma(u, p, 1.0 / 720.0);
  p = fma(u, p, 1.0 / 120.0);
  p = fma(u, p, 1.0 / 24.0);
  p = fma(u, p, 1.0 / 6.0);
  p = fma(u, p, 0.5);
  p = fma(u, p, 1.0);
  return fma(u, p, 1.0);
}
// (a float test: a double comparison is one more operation of the double pipe)
__device__ __forceinline__ double exp_d(double u) {
  const float big = __uint_as_float((unsigned)(__double_as_longlong(u) >> 32) & 0x7fffffffu);
  const float lim = __uint_as_float(0x3fb00000u);  // the high word of 1/16
  return __all_sync(0xffffffffu, big < lim) ? exp_near(u) : exp_far(u);
}

// The weights of one line as a lane of solve_line needs them, asked for
// together and ahead of their use.
constexpr int kDLevels = 5;
template <int P>
struct dweights {
  dz al, be, mu;
  dz ka[kDLevels], kb[kDLevels];  // al^(P 2^l), be^(P 2^l) of the scan
  dz ca, cb;                      // al^(P lane), be^(P (31 - lane)) of the carry
  dz pa[P];                       // al^p of the lane's points (first warp)
};
__device__ __forceinline__ dz dpow(const dz* tab, int nlines, int line, int first, int n) {
  return n < kDPow ? __ldg(tab + (size_t)(first + n) * nlines + line) : zero2d();
}
template <int P, int NW>
__device__ __forceinline__ void dload(dweights<P>& k, const dz* tab, int nlines, int line, int q0,
                                      int levels) {
  const int lane = threadIdx.x & 31;
  k.al = __ldg(tab + line);
  k.be = __ldg(tab + (size_t)nlines + line);
  k.mu = __ldg(tab + (size_t)2 * nlines + line);
#pragma unroll
  for (int l = 0; l < kDLevels; ++l) {
    if (l >= levels) break;
    k.ka[l] = dpow(tab, nlines, line, 3, P << l);
    k.kb[l] = dpow(tab, nlines, line, 3 + kDPow, P << l);
  }
  if (NW > 1) {
    k.ca = dpow(tab, nlines, line, 3, P * lane);
    k.cb = dpow(tab, nlines, line, 3 + kDPow, P * (31 - lane));
  }
  if (NW == 1 || threadIdx.x < 32) {
#pragma unroll
    for (int i = 0; i < P; ++i) k.pa[i] = dpow(tab, nlines, line, 3, q0 + i);
  }
}
// levels of the scan: P 2^levels points reach over the halo
__device__ __forceinline__ int scan_levels(int P, int halo) {
  int l = 0;
  while ((P << l) < halo && l < kDLevels) ++l;
  return l;
}

// One line of N points over NW warps, P points a lane: psi -> psi'.  q0: the
// position of this lane's first point; carry: shared exchange of the warps'
// end values (two sets of NW, for NW > 1; `set` alternates from line to line).
template <int P, int NW>
__device__ __forceinline__ void solve_line(const dweights<P>& k, dz (&psi)[P], int q0, int N,
                                           int levels, dz (*carry)[2][NW]) {
  const int lane = threadIdx.x & 31, w = NW > 1 ? (int)(threadIdx.x >> 5) : 0;
  // forward: the lane's end value from a zero carry, then over the lanes
  dz E = psi[0];
#pragma unroll
  for (int i = 1; i < P; ++i) E = zfma(k.al, E, psi[i]);
#pragma unroll
  for (int l = 0; l < kDLevels; ++l) {
    if (l >= levels) break;
    E = zfma(k.ka[l], shfl_d(E, lane - (1 << l), lane >= (1 << l)), E);
  }
  dz X = shfl_d(E, lane - 1, lane >= 1);
  if (NW > 1) {
    if (lane == 31) (*carry)[0][w] = E;
    __syncthreads();
    if (w > 0) X = zfma(k.ca, (*carry)[0][w - 1], X);
  }
  dz t[P];  // t, then c
#pragma unroll
  for (int i = 0; i < P; ++i) {
    t[i] = zmul(k.al, X);
    X = zadd(psi[i], t[i]);
    if (q0 + i >= N) t[i] = X = zero2d();
  }
  // back (psi is zero past the end, so that e = psi + t is there as well)
  dz U = X;
#pragma unroll
  for (int i = P - 2; i >= 0; --i) U = zfma(k.be, U, zadd(psi[i], t[i]));
#pragma unroll
  for (int l = 0; l < kDLevels; ++l) {
    if (l >= levels) break;
    U = zfma(k.kb[l], shfl_d(U, lane + (1 << l), lane + (1 << l) < 32), U);
  }
  dz Y = shfl_d(U, lane + 1, lane < 31);
  if (NW > 1) {
    if (lane == 0) (*carry)[1][w] = U;
    __syncthreads();
    if (w + 1 < NW) Y = zfma(k.cb, (*carry)[1][w + 1], Y);
  }
#pragma unroll
  for (int i = P - 1; i >= 0; --i) {
    t[i] = zfma(k.be, Y, t[i]);
    Y = zadd(psi[i], t[i]);
  }
  // the start: no value at position 0 (where c_0 is u_0)
  if (w == 0) {
    const dz u0 = shfl_d(Y, 0, true), n0 = make_double2(-u0.x, -u0.y);
#pragma unroll
    for (int i = 0; i < P; ++i) t[i] = zfma(k.pa[i], n0, t[i]);
  }
#pragma unroll
  for (int i = 0; i < P; ++i) psi[i] = zout(psi[i], t[i], k.mu, zadd(psi[i], t[i]));
}

// H1 in imaginary time with the pending scale: psi <- s exp(u) psi, u = cr
// |psi|^2 + vx + vy of the unscaled psi (cr = -dt g s^2, v = -dt V).
__device__ __forceinline__ dz h1_d(dz v, double s, double cr, double pot) {
  const double f = s * exp_d(fma(cr, fma(v.x, v.x, v.y * v.y), pot));
  return make_double2(f * v.x, f * v.y);
}

// ---------------------------------------------------------------- rows
template <int P>
__global__ void __launch_bounds__(128) k_drows(const dline_args a) {
  const int lane = threadIdx.x & 31, N = a.len, q0 = lane * P;
  const double s = *a.scale, cr = -a.dt * a.g * s * s;
  const int levels = scan_levels(P, a.halo);
  double vx[P];
#pragma unroll
  for (int i = 0; i < P; ++i) {
    const double x = fma((double)(q0 + i), a.hx, a.x0);
    vx[i] = q0 + i < N ? -a.dt * (a.hgam2 * x * x) : 0.0;
  }
  const long long warps = (long long)gridDim.x * 4;
  for (long long r = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); r < a.lines; r += warps) {
    const int kz = (int)(r / a.ny), j = (int)(r - (long long)kz * a.ny);
    const double y = fma((double)j, a.hy, a.y0), z = fma((double)kz, a.hz, a.z0);
    const double vyz = -a.dt * fma(a.hnu2 * y, y, a.hlam2 * z * z);
    dweights<P> k;
    dload<P, 1>(k, a.tab, a.tlines, j, q0, levels);
    const dz* row = a.in + r * N;
    dz psi[P];
#pragma unroll
    for (int i = 0; i < P; ++i) psi[i] = q0 + i < N ? row[q0 + i] : zero2d();
#pragma unroll
    for (int i = 0; i < P; ++i) psi[i] = h1_d(psi[i], s, cr, vx[i] + vyz);
    solve_line<P, 1>(k, psi, q0, N, levels, (dz(*)[2][1]) nullptr);
    dz* out = a.out + r * N;
#pragma unroll
    for (int i = 0; i < P; ++i)
      if (q0 + i < N) out[q0 + i] = psi[i];
  }
}

// ---------------------------------------------------------------- columns
// A warp owns 32 consecutive x at one transverse position and a segment of
// a.seg points with halos; t of the segment in shared memory, psi read again
// on the way back.
template <bool REDUCE>
__global__ void __launch_bounds__(32) k_dcols(const dline_args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  dz* ts = reinterpret_cast<dz*>(smem_raw) + threadIdx.x;  // t, [position][lane]
  const int N = a.len, H = a.halo, L = a.seg;
  const int groups = (a.nx + 31) / 32, segs = (N + L - 1) / L;
  long long t = blockIdx.x;
  const int sg = (int)(t % segs);
  t /= segs;
  const int x = (int)(t % groups) * 32 + threadIdx.x;
  const long long tr = t / groups;
  const bool act = x < a.nx;
  const long long stride = a.axis == 1 ? a.nx : (long long)a.nx * a.ny;
  const long long off = (a.axis == 1 ? tr * a.nx * a.ny : tr * a.nx) + (act ? x : 0);
  const dz* in = a.in + off;
  dz* out = a.out + off;
  const int line = a.axis == 1 && act ? x : 0;
  const dz al = __ldg(a.tab + line), be = __ldg(a.tab + (size_t)a.tlines + line);
  const dz mu = __ldg(a.tab + (size_t)2 * a.tlines + line);
  const int p0 = sg * L, p1 = min(N, p0 + L), pe = min(N, p1 + H);
  // forward, four loads ahead
  {
    dz E = zero2d(), v[4];
    int p = max(0, p0 - H);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = p + i < pe ? in[(p + i) * stride] : zero2d();
    for (; p < pe; p += 4) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (p + i >= pe) break;
        const dz t = zmul(al, E);
        E = zadd(v[i], t);
        if (p + i >= p0) ts[(p + i - p0) * 32] = t;
        v[i] = p + 4 + i < pe ? in[(p + 4 + i) * stride] : zero2d();
      }
    }
  }
  // back, four loads ahead: psi a second time
  acc_t<double> acc;
  dz u = zero2d(), v[4];
  int p = pe - 1;
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = p - i >= p0 ? in[(p - i) * stride] : zero2d();
  // the first positions of a line wait for u_0: c stays in place of t
  const int head = sg == 0 ? min(H, p1) : p0;  // (H <= L)
  for (; p >= p0; p -= 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int q = p - i;
      if (q < p0) break;
      const dz psi = v[i], c = zfma(be, u, ts[(q - p0) * 32]);
      v[i] = q - 4 >= p0 ? in[(q - 4) * stride] : zero2d();
      u = zadd(psi, c);
      if (q >= p1) continue;
      if (q < head) {
        ts[(q - p0) * 32] = c;
        continue;
      }
      const dz o = zout(psi, c, mu, u);
      if (REDUCE && act) acc.add(fma(o.x, o.x, o.y * o.y));
      if (act) out[q * stride] = o;
    }
  }
  if (sg == 0) {
    const dz n0 = make_double2(-u.x, -u.y);
    for (int q = head - 1; q >= 0; --q) {
      const dz psi = in[q * stride], c = zfma(dpow(a.tab, a.tlines, line, 3, q), n0, ts[q * 32]);
      const dz o = zout(psi, c, mu, zadd(psi, c));
      if (REDUCE && act) acc.add(fma(o.x, o.x, o.y * o.y));
      if (act) out[q * stride] = o;
    }
  }
  if (REDUCE) norm_epilogue(acc.value(), a);
}

// ---------------------------------------------------------------- 2D steps
constexpr int kDBits = 45, kDFrac = 40;
constexpr int kDTries = 64;  // most repeats of an exchange (48 cross all scales)

// v in units of 2^(ex - kDBits - kDFrac) as hi 2^kDFrac + lo; what is too
// large, negative or NaN becomes the largest share
__device__ __forceinline__ void dshare(double v, int ex, unsigned long long* hi,
                                       unsigned long long* lo) {
  const unsigned long long b = __double_as_longlong(v), one = 1ull << 52;
  const int e = (int)(b >> 52) - 1023;                 // (negative and NaN: large)
  const int s = e - 52 + kDBits + kDFrac - ex;
  unsigned __int128 w = (b & (one - 1)) | one;
  if (e == -1023 || s < -64)
    w = 0;
  else if (e > ex + 1)
    w = (unsigned __int128)1 << (kDBits + kDFrac + 1);
  else
    w = s >= 0 ? w << s : w >> -s;
  *hi = (unsigned long long)(w >> kDFrac);
  *lo = (unsigned long long)w & ((1ull << kDFrac) - 1);
}
__device__ __forceinline__ unsigned long long warp_sum_u(unsigned long long v) {
  const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0xffffff));
  const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 24));
  return ((unsigned long long)b << 24) + a;
}

template <int PX, int PY>
__global__ void __launch_bounds__(128) k_dsteps(const dstep_args a) {
  __shared__ dz carry[2][2][4];
  __shared__ unsigned long long parts[4][2];
  __shared__ double s_scale;
  __shared__ int s_ex, s_again, s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nx = a.nx, ny = a.ny;
  unsigned long long last[2][2];
  if (tid == 0) {
    s_scale = *a.scale;
    s_ex = a.ex0;
    s_fail = s_again = 0;
    for (int i = 0; i < 4; ++i)
      last[i >> 1][i & 1] = *(volatile unsigned long long*)&a.sync->base[i >> 1][i & 1];
  }
  double vx[PX];
#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const double x = fma((double)(tid * PX + i), a.hx, a.x0);
    vx[i] = tid * PX + i < nx ? -a.dt * (a.hgam2 * x * x) : 0.0;
  }
  const int lx = scan_levels(PX, a.halo), ly = scan_levels(PY, a.halo);
  // a sweep's first weights are asked for before the exchange that it waits for
  dweights<PX> kx;
  dweights<PY> ky;
  if (blockIdx.x < ny) dload<PX, 4>(kx, a.tabx, ny, blockIdx.x, tid * PX, lx);
  __syncthreads();
  int set = 0;
  // Meet every CTA: thread 0 adds (hi, lo) and a count of one to the round's
  // words and waits for all; false if the wait gave up.  Everything that the
  // CTAs stored before is visible after.
  auto meet = [&](int word, unsigned long long* hi, unsigned long long* lo) -> bool {
    unsigned long long* w = a.sync->word[word];
    __threadfence();
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"((*hi << 8) | 1ull) : "memory");
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(w + 1), "l"((*lo << 8) | 1ull) : "memory");
    long long t0 = 0;
    for (int it = 1;; ++it) {
      unsigned long long p, q;
      asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(p), "=l"(q) : "l"(w) : "memory");
      const unsigned long long dp = p - last[word][0], dq = q - last[word][1];
      if ((dp & 0xff) == gridDim.x && (dq & 0xff) == gridDim.x) {
        last[word][0] = p;
        last[word][1] = q;
        *hi = dp >> 8;
        *lo = dq >> 8;
        __threadfence();
        return true;
      }
      if ((it & 1023) == 0) {
        const long long t = clock64();
        if (t0 == 0) t0 = t;
        if (t - t0 > 4000000000LL) return false;
      }
    }
  };
  for (int step = 0; step < a.nsteps; ++step) {
    const double s = s_scale, cr = -a.dt * a.g * s * s;
    for (int j = blockIdx.x; j < ny; j += gridDim.x, set ^= 1) {
      const double y = fma((double)j, a.hy, a.y0), vy = -a.dt * (a.hnu2 * y * y);
      if (j != (int)blockIdx.x) dload<PX, 4>(kx, a.tabx, ny, j, tid * PX, lx);
      const dz* row = a.psi[0] + (long long)j * nx;
      const int q0 = tid * PX;
      dz psi[PX];
#pragma unroll
      for (int i = 0; i < PX; ++i) psi[i] = q0 + i < nx ? __ldcg(row + q0 + i) : zero2d();
#pragma unroll
      for (int i = 0; i < PX; ++i) psi[i] = h1_d(psi[i], s, cr, vx[i] + vy);
      solve_line<PX, 4>(kx, psi, q0, nx, lx, &carry[set]);
      dz* out = a.psi[1] + (long long)j * nx;
#pragma unroll
      for (int i = 0; i < PX; ++i)
        if (q0 + i < nx) __stcg(out + q0 + i, psi[i]);
    }
    if (blockIdx.x < nx) dload<PY, 4>(ky, a.taby, nx, blockIdx.x, tid * PY, ly);
    __syncthreads();
    if (tid == 0) {
      unsigned long long z0 = 0, z1 = 0;
      if (!meet(0, &z0, &z1)) s_fail = 1;
    }
    __syncthreads();
    if (s_fail) break;
    double sum = 0.0;
    for (int i = blockIdx.x; i < nx; i += gridDim.x, set ^= 1) {
      if (i != (int)blockIdx.x) dload<PY, 4>(ky, a.taby, nx, i, tid * PY, ly);
      const int q0 = tid * PY;
      dz psi[PY];
#pragma unroll
      for (int u = 0; u < PY; ++u)
        psi[u] = q0 + u < ny ? __ldcg(a.psi[1] + (long long)(q0 + u) * nx + i) : zero2d();
      solve_line<PY, 4>(ky, psi, q0, ny, ly, &carry[set]);
#pragma unroll
      for (int u = 0; u < PY; ++u) {
        if (q0 + u >= ny) continue;
        sum = fma(psi[u].x, psi[u].x, fma(psi[u].y, psi[u].y, sum));
        __stcg(a.psi[0] + (long long)(q0 + u) * nx + i, psi[u]);
      }
    }
    if (blockIdx.x < ny) dload<PX, 4>(kx, a.tabx, ny, blockIdx.x, tid * PX, lx);
    for (int tries = 0;; ++tries) {
      unsigned long long hi, lo;
      dshare(sum, s_ex, &hi, &lo);
      hi = warp_sum_u(hi);
      lo = warp_sum_u(lo);
      if (lane == 0) {
        parts[warp][0] = hi;
        parts[warp][1] = lo;
      }
      __syncthreads();
      if (tid == 0) {
        const unsigned long long most = 1ull << (kDBits + 2);
        hi = min(parts[0][0] + parts[1][0] + parts[2][0] + parts[3][0], most);
        lo = parts[0][1] + parts[1][1] + parts[2][1] + parts[3][1];
        // (a repeated exchange takes the x sweep's word in turn, so that a
        // round never meets the round before it on the same word)
        if (tries > 0) {
          unsigned long long z0 = 0, z1 = 0;
          if (!meet(0, &z0, &z1)) s_fail = 1;
        }
        if (!s_fail && !meet(1, &hi, &lo)) s_fail = 1;
        // The scale that this total asks for, from the bits of the whole total:
        // a sum of many shares below one unit of hi lies in lo alone, and taken
        // for nothing it would lower the scale until the shares are out of
        // range again, and so on for ever.  With all bits a repeat leads to a
        // total in range, or on in one direction to the end of the scales.
        hi += lo >> kDFrac;
        lo &= (1ull << kDFrac) - 1;
        const int ex = s_ex, bits = hi ? kDFrac + 64 - __clzll(hi) : 64 - __clzll(lo);
        const int next = hi >= most  ? ex + 40
                         : bits == 0 ? ex - 40
                                     : ex + bits - kDFrac - kDBits - 1;
        s_ex = max(-900, min(1000, next));
        s_again = !s_fail && (hi < (1ull << (kDBits - 9)) || hi >= most) && s_ex != ex &&
                  tries < kDTries;
        if (!s_again && !s_fail) {
          const double n = ldexp((double)hi + ldexp((double)lo, -kDFrac), ex - kDBits) * a.vol;
          const bool fine = hi > 0 && hi < most;
          // 1/sqrt(n): two Newton steps from the float root (n scaled to [1, 4))
          const int half = ilogb(n) >> 1;
          const double m = ldexp(n, -2 * half);
          double q = (double)rsqrtf((float)m);
          q = q * fma(-0.5 * m * q, q, 1.5);
          q = q * fma(-0.5 * m * q, q, 1.5);
          s_scale = fine ? ldexp(q, -half) : 1.0;
          if (step + 1 == a.nsteps && blockIdx.x == 0) {
            *a.norm = fine ? n : nan("");
            *a.scale = fine ? 1.0 / sqrt(n) : 1.0;
            if (!fine) atomicOr(a.flags, 1);
            for (int i = 0; i < 4; ++i) a.sync->base[i >> 1][i & 1] = last[i >> 1][i & 1];
          }
        }
      }
      __syncthreads();
      if (!s_again || s_fail) break;
    }
    if (s_fail) break;
  }
  if (s_fail && tid == 0) atomicOr(a.flags, 8);
}

// ---------------------------------------------------------------- tables
__global__ void __launch_bounds__(32) k_dtables(dz* tab, int nlines, int halo, axis_coef co) {
  const int l = blockIdx.x * 32 + threadIdx.x;
  if (l >= nlines) return;
  tab += l;
  const double u = co.u0 + (double)l * co.du;
  const dz kap = make_double2(co.kap_re, co.kap_im), tau = make_double2(co.tau_re * u, co.tau_im * u);
  const dz a0 = make_double2(1.0 + 2.0 * kap.x, 2.0 * kap.y);
  const dz am = make_double2(tau.x - kap.x, tau.y - kap.y);
  const dz ap = make_double2(-kap.x - tau.x, -kap.y - tau.y);
  const dz aa = zfma(am, ap, zero2d());
  // the multiplier: the root of A- A+ m^2 - A0 m + 1 = 0 near 1/A0, by
  // iterating m = 1/(A0 - A- A+ m) in float and three Newton steps in double
  // whose quotient is taken in float
  float2 mf = make_float2(1.f, 0.f);
  for (int i = 0; i < 64; ++i) {
    const float tx = (float)aa.x * mf.x - (float)aa.y * mf.y, ty = (float)aa.x * mf.y + (float)aa.y * mf.x;
    const float qx = (float)a0.x - tx, qy = (float)a0.y - ty, r = 1.f / (qx * qx + qy * qy);
    mf = make_float2(qx * r, -qy * r);
  }
  dz m = make_double2(mf.x, mf.y);
  for (int i = 0; i < 3; ++i) {
    const dz t = zfma(aa, m, zero2d());
    const dz q = make_double2(t.x - a0.x, t.y - a0.y), r = zfma(q, m, make_double2(1.0, 0.0));
    const float sx = (float)(t.x + q.x), sy = (float)(t.y + q.y), i2 = 1.f / (sx * sx + sy * sy);
    const float rx = (float)r.x, ry = (float)r.y;
    m.x -= (double)((rx * sx + ry * sy) * i2);
    m.y -= (double)((ry * sx - rx * sy) * i2);
  }
  dz al = zfma(m, am, zero2d()), be = zfma(m, ap, zero2d());
  al = make_double2(-al.x, -al.y);
  be = make_double2(-be.x, -be.y);
  tab[0] = al;
  tab[(size_t)nlines] = be;
  tab[(size_t)2 * nlines] = make_double2(m.x - 1.0, m.y);
  dz pa = make_double2(1.0, 0.0), pb = pa;
  for (int p = 0; p < kDPow; ++p) {
    tab[(size_t)(3 + p) * nlines] = p < halo ? pa : zero2d();
    tab[(size_t)(3 + kDPow + p) * nlines] = p < halo ? pb : zero2d();
    if (p < halo) {
      pa = zfma(pa, al, zero2d());
      pb = zfma(pb, be, zero2d());
    }
  }
}

int points_per_lane(int N, int warps) {
  for (int P : {1, 2, 4, 8, 16})
    if (32 * warps * P >= N) return P;
  return 0;
}

template <int PX>
cudaError_t launch_2d(const dstep_args& a, int PY, int blocks, cudaStream_t s) {
  const void* fn = PY == 1   ? (const void*)k_dsteps<PX, 1>
                   : PY == 2 ? (const void*)k_dsteps<PX, 2>
                   : PY == 4 ? (const void*)k_dsteps<PX, 4>
                             : (const void*)k_dsteps<PX, 8>;
  void* args[] = {const_cast<dstep_args*>(&a)};
  return cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(128), args, 0, s);
}

}  // namespace

cudaError_t launch_dtables(double2* tab, int nlines, int halo, const axis_coef& co, cudaStream_t s) {
  k_dtables<<<(nlines + 31) / 32, 32, 0, s>>>(tab, nlines, halo, co);
  return cudaGetLastError();
}

int drow_points(int N, int halo) {
  const int P = points_per_lane(N, 1);
  return halo <= kDPow && halo <= 32 * P && halo < N ? P : 0;
}

cudaError_t launch_drows(const dline_args& a, int P, cudaStream_t s) {
  const unsigned blocks = (unsigned)std::min<long long>((a.lines + 3) / 4, 152 * 16);
  switch (P) {
    case 1: k_drows<1><<<blocks, 128, 0, s>>>(a); break;
    case 2: k_drows<2><<<blocks, 128, 0, s>>>(a); break;
    case 4: k_drows<4><<<blocks, 128, 0, s>>>(a); break;
    case 8: k_drows<8><<<blocks, 128, 0, s>>>(a); break;
    case 16: k_drows<16><<<blocks, 128, 0, s>>>(a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The segment length with the least double operations of the busiest
// scheduler: 18 a point, 6 and 12 in the halos, rounds of one warp per
// scheduler.  At least a halo, at most 96 points with the halo (48 KB of
// shared memory a warp).
int dcol_segment(int N, long long lines, int halo, int sm_count) {
  if (halo >= N) return 0;
  const long long groups = (lines + 31) / 32;
  double best = 0;
  int seg = 0;
  for (int segs = 1; segs <= N; ++segs) {
    const int L = (N + segs - 1) / segs;
    if (L + std::min(halo, N - L) > 96) continue;
    if (L < halo && L < N) break;
    const long long warps = groups * ((N + L - 1) / L);
    const double rounds = (double)((warps + 4LL * sm_count - 1) / (4LL * sm_count));
    const double cost = rounds * (18.0 * L + (L < N ? 18.0 * halo : 0.0) + 20.0);
    if (!seg || cost < best) {
      best = cost;
      seg = L;
    }
  }
  return seg;
}
long long dcol_blocks(int nx, long long lines, int len, int seg) {
  return (long long)((nx + 31) / 32) * (lines / nx) * ((len + seg - 1) / seg);
}

cudaError_t launch_dcols(bool reduce, const dline_args& a, cudaStream_t s) {
  const size_t smem = (size_t)(a.seg + std::min(a.halo, a.len - a.seg)) * 32 * sizeof(double2);
  const void* fn = reduce ? (const void*)k_dcols<true> : (const void*)k_dcols<false>;
  const cudaError_t e = allow_smem_bytes(fn, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)dcol_blocks(a.nx, a.lines, a.len, a.seg);
  if (reduce)
    k_dcols<true><<<blocks, 32, smem, s>>>(a);
  else
    k_dcols<false><<<blocks, 32, smem, s>>>(a);
  return cudaGetLastError();
}

bool dstep_fits(int nx, int ny, int halo) {
  const int px = points_per_lane(nx, 4), py = points_per_lane(ny, 4);
  return px >= 1 && px <= 4 && py >= 1 && py <= 8 && halo <= 32 * std::min(px, py) &&
         halo < std::min(nx, ny);
}

cudaError_t launch_dsteps(const dstep_args& a, int sm_count, cudaStream_t s) {
  const int px = points_per_lane(a.nx, 4), py = points_per_lane(a.ny, 4);
  const int blocks = std::min(std::min(sm_count, 250), std::max(a.nx, a.ny));
  switch (px) {
    case 1: return launch_2d<1>(a, py, blocks, s);
    case 2: return launch_2d<2>(a, py, blocks, s);
    case 4: return launch_2d<4>(a, py, blocks, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace rotgp
