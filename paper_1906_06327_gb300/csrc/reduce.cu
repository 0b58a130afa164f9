// reduce.cu -- the read-only reductions over a state: the observables of
// Sec. 2 (norm, real-part mu and E of Eqs. e2dr/e3dr, complex forms of
// Eqs. e2d/e3d, rms sizes), the vortex count diagnostic, and the plain norm
// used after loading a state.
//
// Every reduction is one pass over the state: each thread accumulates its
// sites in registers, blocks reduce with warp shuffles and write one partial
// per block, and the last block to finish (atomic ticket) combines the
// partials in a fixed order, so results are deterministic run to run.  The
// pending imaginary-time scale is applied as the state is read.
#include <algorithm>

#include "observe.cuh"
#include "pairsum.cuh"

namespace rotgp {

// ------------------------------------------------------------ observables
// One pass over the state.  A warp owns 28 columns along the march (z in 3D,
// y in 2D; lanes 2 .. 29, the outer lanes hold the neighbours in x) and walks
// a chunk of it with the five points around the current one in registers, so
// the differences along the march need no memory, those in x are shuffles,
// and only those in y of a 3D state are further loads, of rows that the
// neighbouring warps of the block load as well (L1).  No shared memory and no
// barrier inside the walk: the tiles of 32 x 8 columns staged plane by plane
// that this replaces met at a barrier per plane.
//
// What bounds it: instructions (about 170 a site, of which 32 are the eight
// compensated sums; the FMAs, with three registers read each, take 1.7 cycles),
// not the one read of the state: three blocks per SM instead of two were
// slower (spills; 256 x 256 x 128 152 us against 117).  Sums that follow from
// others are not kept: |psi|^2 = psi_R^2 + psi_I^2, the complex-form energy is
// the sum of the two real-part ones, and the squares of the coordinates that
// are constant along the march multiply a column's sum once.  The sums meet in
// float pairs (pairsum.cuh), and the ratios and roots are left to the host:
// they and the sums of 14 doubles through shuffles were most of the time on a
// small state.  GB300, before / after, whole rotgp_observables call (with the
// vortex count): 128^2 72 / 31 us, 440^2 153 / 39 us, 4096^2 1,880 / 310 us,
// 256 x 256 x 128 261 / 135 us.
__device__ __forceinline__ float fmat(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmat(double a, double b, double c) { return fma(a, b, c); }
template <class T>
__device__ __forceinline__ cpx<T> shfl_to(cpx<T> v, int d) {  // of the lane d to the right
  const int src = ((int)threadIdx.x + d) & 31;
  return mk<T>(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
constexpr int kObsCols = 28, kObsWarps = 8;

template <class T, bool D3>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1) k_observe(const observe_args a) {
  using C = cpx<T>;
  using S = typename run_sum<T>::sum;
  const C* psi = static_cast<const C*>(a.psi);
  const int nx = a.nx, ny = a.ny, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nm = D3 ? a.nz : ny;                      // points of a march
  const long long ms = D3 ? (long long)nx * ny : nx;  // its stride
  const T s = (T)(*a.scale);
  const T ihx2 = (T)(1.0 / (a.hx * a.hx)), ihy2 = (T)(1.0 / (a.hy * a.hy));
  const T ihz2 = D3 ? (T)(1.0 / (a.hz * a.hz)) : (T)0;
  const T i2hx = (T)(0.5 / a.hx), i2hy = (T)(0.5 / a.hy), om = (T)a.omega;
  const T c12x = ihx2 / (T)12, c12y = ihy2 / (T)12, c12z = ihz2 / (T)12;
  const T i12hx = i2hx / (T)6, i12hy = i2hy / (T)6;
  const T x0 = (T)a.x0, y0 = (T)a.y0, z0 = (T)a.z0, hx = (T)a.hx, hy = (T)a.hy, hz = (T)a.hz;
  const T hgam2 = (T)a.hgam2, hnu2 = (T)a.hnu2, hlam2 = (T)a.hlam2;
  const T l0 = (T)2 * (ihx2 + ihy2 + ihz2), l04 = (T)30 * (c12x + c12y + c12z);
  const int groups = (nx + kObsCols - 1) / kObsCols;
  const int parts = (nm + a.chunk - 1) / a.chunk;
  // a block's warps: neighbouring rows (3D), neighbouring column groups (2D)
  const int wide = D3 ? (ny + kObsWarps - 1) / kObsWarps : (groups + kObsWarps - 1) / kObsWarps;
  const int items = D3 ? wide * groups * parts : wide * parts;
  run_sum<T> lr, li, nr, ni, l4, m2s;
  S tot[OS_COUNT];
#pragma unroll
  for (int v = 0; v < OS_COUNT; ++v) tot[v] = sum_zero((S*)nullptr);
  T dmax = 0;
  for (int it = blockIdx.x; it < items; it += gridDim.x) {
    const int wi = it % wide, rest = it / wide;
    const int grp = D3 ? rest % groups : wi * kObsWarps + warp;
    const int part = D3 ? rest / groups : rest;
    const int j0 = D3 ? wi * kObsWarps + warp : 0;    // row of the column (3D)
    const int i = grp * kObsCols + lane - 2;
    if (grp >= groups || (D3 && j0 >= ny)) continue;  // whole warps
    const int k0 = part * a.chunk, k1 = min(nm, k0 + a.chunk);
    const bool col = i >= 0 && i < nx;
    const C* base = psi + (D3 ? (long long)j0 * nx : 0) + i;
    auto raw = [&](int k, int dj) -> C {              // unscaled, zero outside
      if (!col || k < 0 || k >= nm || (D3 && (j0 + dj < 0 || j0 + dj >= ny))) return mk<T>(0, 0);
      return base[k * ms + (D3 ? (long long)dj * nx : 0)];
    };
    const bool own = lane >= 2 && lane < 2 + kObsCols && i >= 1 && i < nx && (!D3 || j0 >= 1);
    const T x = x0 + (T)i * hx, yc = y0 + (T)j0 * hy;
    const T vc = D3 ? fmat(hgam2 * x, x, hnu2 * yc * yc) : hgam2 * x * x;
    const T xh = x * i2hy, x12 = x * i12hy;
    C w[5], ahead = raw(k0 + 3, 0), side[4] = {};
#pragma unroll
    for (int d = 0; d < 5; ++d) w[d] = s * raw(k0 - 2 + d, 0);
    if (D3) {
      side[0] = raw(k0, -2), side[1] = raw(k0, -1), side[2] = raw(k0, 1), side[3] = raw(k0, 2);
    }
    run_sum<T> cr, ci;  // this column's psi_R^2 and psi_I^2
    T mf = (T)k0;
    for (int k = k0; k < k1; ++k) {
      const C next = raw(k + 4, 0);
      C sd[4];
#pragma unroll
      for (int d = 0; d < 4; ++d) sd[d] = s * side[d];
      if (D3 && k + 1 < k1) {
        side[0] = raw(k + 1, -2), side[1] = raw(k + 1, -1);
        side[2] = raw(k + 1, 1), side[3] = raw(k + 1, 2);
      }
      const C c = w[2];
      const C xm2 = shfl_to(c, -2), xm = shfl_to(c, -1), xp = shfl_to(c, 1), xp2 = shfl_to(c, 2);
      const C ym2 = D3 ? sd[0] : w[0], ym = D3 ? sd[1] : w[1];
      const C yp = D3 ? sd[2] : w[3], yp2 = D3 ? sd[3] : w[4];
      const T m = D3 ? z0 + mf * hz : y0 + mf * hy;   // the march's coordinate
      const T y = D3 ? yc : m;
      const T V = D3 ? fmat(hlam2 * m, m, vc) : fmat(hnu2 * m, m, vc);
      if (own && k >= 1) {
        const C sx = xp + xm, sy = yp + ym, ex = xp2 + xm2, ey = yp2 + ym2;
        const C dx = xp - xm, dy = yp - ym, fx = xp2 - xm2, fy = yp2 - ym2;
        C sz = mk<T>(0, 0), ez = sz;
        if (D3) {
          sz = w[3] + w[1];
          ez = w[4] + w[0];
        }
        const T re = c.x, im = c.y, r2 = re * re, i2 = im * im, dens = fmat(re, re, i2);
        // -lap/2 + V and the rotation term, 3-point and 5-point forms;
        // L_z psi / i = y D_x psi - x D_y psi
        const T yh = y * i2hx, y12 = y * i12hx;
        const T lapr = fmat(ihx2, sx.x, fmat(ihy2, sy.x, fmat(ihz2, sz.x, -l0 * re)));
        const T lapi = fmat(ihx2, sx.y, fmat(ihy2, sy.y, fmat(ihz2, sz.y, -l0 * im)));
        const T lzr = fmat(yh, dx.x, -xh * dy.x), lzi = fmat(yh, dx.y, -xh * dy.y);
        const T hr = fmat((T)-0.5, lapr, fmat(V, re, om * lzi));
        const T hi = fmat((T)-0.5, lapi, fmat(V, im, -om * lzr));
        const T l4r = fmat(c12x, fmat((T)16, sx.x, -ex.x),
                           fmat(c12y, fmat((T)16, sy.x, -ey.x),
                                fmat(c12z, fmat((T)16, sz.x, -ez.x), -l04 * re)));
        const T l4i = fmat(c12x, fmat((T)16, sx.y, -ex.y),
                           fmat(c12y, fmat((T)16, sy.y, -ey.y),
                                fmat(c12z, fmat((T)16, sz.y, -ez.y), -l04 * im)));
        const T z4r = fmat(y12, fmat((T)8, dx.x, -fx.x), -x12 * fmat((T)8, dy.x, -fy.x));
        const T z4i = fmat(y12, fmat((T)8, dx.y, -fx.y), -x12 * fmat((T)8, dy.y, -fy.y));
        const T h4r = fmat((T)-0.5, l4r, fmat(V, re, om * z4i));
        const T h4i = fmat((T)-0.5, l4i, fmat(V, im, -om * z4r));
        cr.add(r2);
        ci.add(i2);
        lr.add(re * hr);
        li.add(im * hi);
        nr.add(dens * r2);
        ni.add(dens * i2);
        m2s.add(m * m * dens);
        l4.add(fmat(re, h4r, im * h4i));
        dmax = dmax > dens ? dmax : dens;
        if (D3 && k == a.kplane) {
          run_sum<T> d;
          d.add(dens);
          tot[OS_P0] = sum_add(tot[OS_P0], d.value());
          tot[OS_PX2] = sum_add(tot[OS_PX2], sum_scale(x * x, d.value()));
          tot[OS_PY2] = sum_add(tot[OS_PY2], sum_scale(yc * yc, d.value()));
        }
      }
#pragma unroll
      for (int d = 0; d < 4; ++d) w[d] = w[d + 1];
      w[4] = s * ahead;
      ahead = next;
      mf += (T)1;
    }
    const S dc = sum_add(cr.value(), ci.value());
    tot[OS_RE2] = sum_add(tot[OS_RE2], cr.value());
    tot[OS_IM2] = sum_add(tot[OS_IM2], ci.value());
    tot[OS_X2] = sum_add(tot[OS_X2], sum_scale(x * x, dc));
    if (D3) tot[OS_Y2] = sum_add(tot[OS_Y2], sum_scale(yc * yc, dc));
  }
  tot[OS_LR] = lr.value();
  tot[OS_LI] = li.value();
  tot[OS_NR] = nr.value();
  tot[OS_NI] = ni.value();
  tot[OS_L4] = l4.value();
  tot[D3 ? OS_Z2 : OS_Y2] = m2s.value();
  __shared__ double fin[OS_COUNT];
  if (!grid_sums16<true>(tot, (double)dmax, a.partials, a.counter, fin)) return;
  if (threadIdx.x < OS_COUNT) a.sums[threadIdx.x] = fin[threadIdx.x];
  if (threadIdx.x < 2) {
    // the ellipse of the vortex count, a lane per axis (the division is 1,500
    // cycles; in the counting kernel every thread paid it)
    const double s0 = D3 ? fin[OS_P0] : fin[OS_RE2] + fin[OS_IM2];
    const double m = fin[(D3 ? OS_PX2 : OS_X2) + threadIdx.x];
    const double r2 = s0 > 0 ? 6.0 * m / s0 : 0.0;
    a.ellipse->r2[threadIdx.x] = r2;
    a.ellipse->inv[threadIdx.x] = r2 > 0 ? 1.f / (float)r2 : 0.f;
  }
  if (threadIdx.x == 0) *a.count = 0;
}

// ------------------------------------------------------------ vortex count
// Plaquettes (i,j)..(i+1,j+1) of the plane k = kplane that touch no edge and
// are centred inside 0.9 of the ellipse R_x^2 = 6 <x^2>, R_y^2 = 6 <y^2> of
// the plane's density: winding = round(sum of arg(psi_b conj(psi_a)) around
// the loop / 2 pi), computed in T.
//
// The centre is tested in float and only within 1e-5 of the line in double
// (two divisions, 3,000 cycles of a warp).  Four phase steps that are each
// well inside a right angle cannot add up to a full turn, so the arc tangents
// are left to the few plaquettes with a larger step.
__device__ __forceinline__ float atan2_t(float y, float x) { return atan2f(y, x); }
__device__ __forceinline__ double atan2_t(double y, double x) { return atan2(y, x); }
__device__ __forceinline__ int round_half_away(float v) { return (int)roundf(v); }
__device__ __forceinline__ int round_half_away(double v) { return (int)round(v); }

template <class T>
__global__ void __launch_bounds__(256) k_vort_count(const observe_args a) {
  using C = cpx<T>;
  const C* pl = static_cast<const C*>(a.psi) + (size_t)a.kplane * a.nx * a.ny;
  const float irx2 = a.ellipse->inv[0], iry2 = a.ellipse->inv[1];
  if (!(irx2 > 0.f && iry2 > 0.f)) return;
  const float fx0 = a.fx0, fy0 = a.fy0, fhx = a.fhx, fhy = a.fhy;
  int cnt = 0;
  for (int j = 1 + blockIdx.y; j + 1 < a.ny; j += gridDim.y) {
    const float yc = fmaf((float)j, fhy, fy0), ey = yc * yc * iry2;
    for (int i = 1 + blockIdx.x * 256 + threadIdx.x; i + 1 < a.nx; i += gridDim.x * 256) {
      const float xc = fmaf((float)i, fhx, fx0), e = fmaf(xc * xc, irx2, ey) - 0.81f;
      if (e > 1e-5f) continue;
      if (e > -1e-5f) {
        const double rx2 = a.ellipse->r2[0], ry2 = a.ellipse->r2[1];
        const double xd = a.x0 + i * a.hx + 0.5 * a.hx, yd = a.y0 + j * a.hy + 0.5 * a.hy;
        if (!(xd * xd / rx2 + yd * yd / ry2 < 0.81)) continue;
      }
      const C* p = pl + (size_t)j * a.nx + i;
      const C q[4] = {p[0], p[1], p[1 + a.nx], p[a.nx]};
      T pr[4], pi[4];
      bool small = true;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const C u = q[(t + 1) & 3], v = q[t];
        pr[t] = u.x * v.x + u.y * v.y;
        pi[t] = u.y * v.x - u.x * v.y;
        small = small && pr[t] > (T)0.125 * fabs(pi[t]);
      }
      if (small) continue;
      T w = 0;
#pragma unroll
      for (int t = 0; t < 4; ++t) w += atan2_t(pi[t], pr[t]);
      const int wn = round_half_away(w / (T)6.28318530717958647692);
      cnt += wn < 0 ? -wn : wn;
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(a.count, cnt);
}

// ------------------------------------------------------------ plain norm
template <class T>
__global__ void __launch_bounds__(256) k_norm(const void* psi_v, long long n, double vol,
                                              int imag_scale, double* partials,
                                              unsigned* counter, double* scale_out,
                                              double* norm_out, int* flags) {
  using S = typename run_sum<T>::sum;
  const cpx<T>* psi = static_cast<const cpx<T>*>(psi_v);
  run_sum<T> q;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x)
    q.add(abs2(psi[idx]));
  S v[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = sum_zero((S*)nullptr);
  v[0] = q.value();
  __shared__ double fin[16];
  if (!grid_sums16<false>(v, 0.0, partials, counter, fin)) return;
  if (threadIdx.x == 0) {
    const double nrm = fin[0] * vol;
    *norm_out = nrm;
    if (!(nrm > 0.0) || !isfinite(nrm)) {
      atomicOr(flags, 1);
      *scale_out = 1.0;
    } else {
      *scale_out = imag_scale ? 1.0 / sqrt(nrm) : 1.0;
    }
  }
}

// ------------------------------------------------------------ launchers
// The march split so that the blocks' rounds of work items, each with its five
// points to fill the window, come out shortest.
void observe_shape(int nx, int ny, int nz, int dim, int sm_count, int* chunk, int* blocks) {
  const int groups = (nx + kObsCols - 1) / kObsCols, nm = dim == 3 ? nz : ny;
  const long long wide = dim == 3 ? (long long)((ny + kObsWarps - 1) / kObsWarps) * groups
                                  : (groups + kObsWarps - 1) / kObsWarps;
  const long long most = (long long)kObserveBlocksPerSm * sm_count;
  double best = 0;
  for (int parts = 1; parts <= nm && parts <= 512; ++parts) {
    const int len = (nm + parts - 1) / parts, np = (nm + len - 1) / len;
    const double cost = (double)((wide * np + most - 1) / most) * (len + 6.0);
    if (parts == 1 || cost < best) {
      best = cost;
      *chunk = len;
      *blocks = (int)std::min(most, wide * np);
    }
  }
}

cudaError_t launch_observe(bool fp64, const observe_args& a, int blocks, cudaStream_t s) {
  if (a.dim == 3) {
    if (fp64)
      k_observe<double, true><<<blocks, 256, 0, s>>>(a);
    else
      k_observe<float, true><<<blocks, 256, 0, s>>>(a);
  } else {
    if (fp64)
      k_observe<double, false><<<blocks, 256, 0, s>>>(a);
    else
      k_observe<float, false><<<blocks, 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t launch_vortex_count(bool fp64, const observe_args& a, cudaStream_t s) {
  const dim3 grid((unsigned)std::min(16, (a.nx + 255) / 256), (unsigned)std::min(512, a.ny));
  if (fp64)
    k_vort_count<double><<<grid, 256, 0, s>>>(a);
  else
    k_vort_count<float><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_norm(bool fp64, const void* psi, long long nsites, double vol, int imag_scale,
                        double* partials, unsigned int* counter, double* scale_out,
                        double* norm_out, int* flags, int blocks, int threads, cudaStream_t s) {
  if (fp64)
    k_norm<double><<<blocks, threads, 0, s>>>(psi, nsites, vol, imag_scale, partials, counter,
                                              scale_out, norm_out, flags);
  else
    k_norm<float><<<blocks, threads, 0, s>>>(psi, nsites, vol, imag_scale, partials, counter,
                                             scale_out, norm_out, flags);
  return cudaGetLastError();
}

}  // namespace rotgp
