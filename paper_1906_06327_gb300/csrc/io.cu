// io.cu -- states in and out of a context: the analytic initial state of
// Eq. fun, and conversion between the ABI layout ((N+1)^d points with both
// edges, float or double) and the device layout (N^d points, index 0 edge
// stored as zero, index N edge implicit) with the pending scale applied.
#include <algorithm>

#include "common.cuh"
#include "observe.cuh"
#include "pairsum.cuh"

namespace rotgp {

// Eq. fun: psi = (x + i y)/sqrt(pi d^2) exp(-(x^2+y^2)/(2 d^2)) e^{2 pi i R}
// [3D: * (pi d_z^2)^(-1/4) exp(-z^2/(2 d_z^2))]; function 0: (x + i y) -> 1.
// Evaluated in double, stored in T.  R(x_i, y_j) is the number of the point
// n = j (N_x + 1) + i of the (N_x+1)(N_y+1) plane: read from the table R
// (phase_mode 1) or drawn from SplitMix64(seed) (phase_mode 2); phase_mode 0
// leaves the phase out.
template <class T>
__global__ void k_init_analytic(cpx<T>* psi, int nx, int ny, int nz, int dim, double x0,
                                double hx, double y0, double hy, double z0, double hz,
                                int function, int phase_mode, const double* R,
                                unsigned long long seed, double d_xy, double d_z) {
  const long long n = (long long)nx * ny * nz;
  const double kPi = 3.14159265358979323846;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(idx % nx), j = (int)((idx / nx) % ny), k = (int)(idx / ((long long)nx * ny));
    if (i == 0 || j == 0 || (dim == 3 && k == 0)) {
      psi[idx] = mk<T>(0, 0);
      continue;
    }
    const double x = x0 + i * hx, y = y0 + j * hy;
    double pr = 1.0, pi = 0.0;
    if (function) {
      pr = x;
      pi = y;
    }
    double amp = exp(-(x * x + y * y) / (2.0 * d_xy * d_xy)) / sqrt(kPi * d_xy * d_xy);
    if (dim == 3) {
      const double z = z0 + k * hz;
      amp *= pow(kPi * d_z * d_z, -0.25) * exp(-z * z / (2.0 * d_z * d_z));
    }
    double sn = 0.0, cs = 1.0;
    const unsigned long long pn = (unsigned long long)j * (nx + 1) + i;
    if (phase_mode == 1) sincos(2.0 * kPi * R[pn], &sn, &cs);
    if (phase_mode == 2) sincos(2.0 * kPi * splitmix64_unit(seed, pn), &sn, &cs);
    psi[idx] = mk<T>((T)(amp * (pr * cs - pi * sn)), (T)(amp * (pr * sn + pi * cs)));
  }
}

// Between complex float and complex float, both layouts are copied row by row: a
// warp takes 256 points of a row, so no index is divided per point and every
// lane has eight loads in flight.  Nothing is converted to double there (three or
// six operations of the double pipe per point made whole calls on a 4096^2 state
// take 222 us in and 202 us out; 79 and 66 us now, 256 x 256 x 128 130 and 115 us,
// now 55 and 42).  The norm of a loaded state is summed as it is written.
//
// Where either side is double, and on rows of a few points, a thread takes one
// point at a time from the whole grid: the double pipe is what bounds those
// copies, and a lane outside the row costs it as much as one inside (into complex
// double, rows against points: 20 x 300 x 300 177 / 21 us, 256 x 256 x 128 133 / 70; from it, 99 / 25 and 51 / 68).
constexpr int kRowPart = 256;
template <class TS, class TD>
constexpr bool row_copy() { return sizeof(TS) + sizeof(TD) == 8; }
constexpr int kRowLeast = 16;  // points of a row

// Coordinates of point idx of an a x b x ... grid.
__device__ __forceinline__ void grid_point(long long idx, int a, int b, int* i, int* j, int* k) {
  if (idx <= 0xffffffffll) {
    const unsigned u = (unsigned)idx, r = u / (unsigned)a;
    *i = (int)(u - r * (unsigned)a);
    *k = (int)(r / (unsigned)b);
    *j = (int)(r - (unsigned)*k * (unsigned)b);
  } else {
    const long long r = idx / a;
    *i = (int)(idx - r * a);
    *k = (int)(r / b);
    *j = (int)(r - (long long)*k * b);
  }
}

// ABI layout -> device layout, with the norm of the loaded state in the same
// pass (NORM) and from it the pending scale; otherwise the scale is 1.
template <class TS, class TD, bool NORM, bool ROWS>
__global__ void __launch_bounds__(256) k_load(const cpx<TS>* __restrict__ src,
                                              cpx<TD>* __restrict__ psi, int nx, int ny, int nz,
                                              int dim, double vol, double* partials,
                                              unsigned* counter, double* scale, double* norm,
                                              int* flags) {
  using S = typename run_sum<TD>::sum;
  run_sum<TD> q;
  if constexpr (!ROWS) {
    const long long n = (long long)nx * ny * nz;
    for (long long idx = (long long)blockIdx.x * 256 + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * 256) {
      int i, j, k;
      grid_point(idx, nx, ny, &i, &j, &k);
      cpx<TD> w = mk<TD>(0, 0);
      if (i != 0 && j != 0 && !(dim == 3 && k == 0)) {
        const cpx<TS> v = src[((long long)k * (ny + 1) + j) * (nx + 1) + i];
        w = mk<TD>((TD)v.x, (TD)v.y);
      }
      psi[idx] = w;
      if (NORM) q.add(abs2(w));
    }
  } else {
    const int lane = threadIdx.x & 31, parts = (nx + kRowPart - 1) / kRowPart;
    const long long tasks = (long long)ny * nz * parts;
    for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < tasks;
         t += (long long)gridDim.x * 8) {
      const long long row = t / parts;
      const int i0 = (int)(t - row * parts) * kRowPart + lane;
      const int k = (int)(row / ny), j = (int)(row - (long long)k * ny);
      const bool zero = j == 0 || (dim == 3 && k == 0);
      const cpx<TS>* from = src + ((long long)k * (ny + 1) + j) * (nx + 1);
      cpx<TS> v[kRowPart / 32];
#pragma unroll
      for (int u = 0; u < kRowPart / 32; ++u) {
        const int i = i0 + 32 * u;
        v[u] = !zero && i > 0 && i < nx ? from[i] : mk<TS>(0, 0);
      }
#pragma unroll
      for (int u = 0; u < kRowPart / 32; ++u) {
        const int i = i0 + 32 * u;
        if (i - lane >= nx) break;
        if (i >= nx) continue;
        const cpx<TD> w = mk<TD>((TD)v[u].x, (TD)v[u].y);
        psi[row * nx + i] = w;
        if (NORM) q.add(abs2(w));
      }
    }
  }
  if (!NORM) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale = 1.0;
    return;
  }
  S s[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) s[i] = sum_zero((S*)nullptr);
  s[0] = q.value();
  __shared__ double fin[16];
  if (!grid_sums16<false>(s, 0.0, partials, counter, fin)) return;
  if (threadIdx.x == 0) {
    const double n = fin[0] * vol;
    const bool fine = n > 0.0 && isfinite(n);
    *norm = n;
    *scale = fine ? 1.0 / sqrt(n) : 1.0;
    if (!fine) atomicOr(flags, 1);
  }
}

// s v rounded once, s = sh + sl.  The second part of an infinity (NaN, or of the
// other sign) is left out; taking such values through double instead, in a
// branch, made reading back 256 x 256 x 128 100 us slower.
__device__ __forceinline__ float scaled(double s, float sh, float sl, float v, float) {
  const float p = sl * v;
  return fmaf(sh, v, fabsf(p) < __int_as_float(0x7f800000) ? p : 0.f);
}
template <class TS, class TD>
__device__ __forceinline__ TD scaled(double s, float, float, TS v, TD) {
  return (TD)(s * (double)v);
}

// Device layout -> ABI layout, multiplying by the pending scale and writing
// zeros on both edges of every axis.
template <class TS, class TD, bool ROWS>
__global__ void __launch_bounds__(256) k_store(const cpx<TS>* __restrict__ psi,
                                               cpx<TD>* __restrict__ dst, int nx, int ny, int nz,
                                               int dim, const double* scale) {
  const double s = *scale;
  const float sh = (float)s, sl = (float)(s - (double)sh);
  if constexpr (!ROWS) {
    const long long n = (long long)(nx + 1) * (ny + 1) * (dim == 3 ? nz + 1 : 1);
    for (long long idx = (long long)blockIdx.x * 256 + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * 256) {
      int i, j, k;
      grid_point(idx, nx + 1, ny + 1, &i, &j, &k);
      const bool edge = i == 0 || i == nx || j == 0 || j == ny || (dim == 3 && (k == 0 || k == nz));
      cpx<TD> w = mk<TD>(0, 0);
      if (!edge) {
        const cpx<TS> v = psi[((long long)k * ny + j) * nx + i];
        w = mk<TD>(scaled(s, sh, sl, v.x, (TD)0), scaled(s, sh, sl, v.y, (TD)0));
      }
      dst[idx] = w;
    }
  } else {
    const int lane = threadIdx.x & 31, parts = (nx + 1 + kRowPart - 1) / kRowPart;
    const long long tasks = (long long)(ny + 1) * (dim == 3 ? nz + 1 : 1) * parts;
    for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < tasks;
         t += (long long)gridDim.x * 8) {
      const long long row = t / parts;
      const int i0 = (int)(t - row * parts) * kRowPart + lane;
      const int k = (int)(row / (ny + 1)), j = (int)(row - (long long)k * (ny + 1));
      const bool zero = j == 0 || j == ny || (dim == 3 && (k == 0 || k == nz));
      const cpx<TS>* from = psi + ((long long)k * ny + j) * nx;
      cpx<TS> v[kRowPart / 32];
#pragma unroll
      for (int u = 0; u < kRowPart / 32; ++u) {
        const int i = i0 + 32 * u;
        v[u] = !zero && i > 0 && i < nx ? from[i] : mk<TS>(0, 0);
      }
#pragma unroll
      for (int u = 0; u < kRowPart / 32; ++u) {
        const int i = i0 + 32 * u;
        if (i - lane > nx) break;
        if (i <= nx)
          dst[row * (nx + 1) + i] = mk<TD>(scaled(s, sh, sl, v[u].x, (TD)0), scaled(s, sh, sl, v[u].y, (TD)0));
      }
    }
  }
}

__global__ void k_set_scalar(double* p, double v) { *p = v; }

// The density integrated along z (the paper's reduced 2D density of a 3D
// state, Sec. 3): out[j][i] = h_z sum_k |s psi(i, j, k)|^2 on the
// (N_x+1)(N_y+1) plane, edges zero; in 2D the density itself.
template <class T>
__global__ void k_column_density(const cpx<T>* psi, double* out, int nx, int ny, int nz,
                                 double hz, const double* scale) {
  const long long px = nx + 1, n = px * (ny + 1);
  const double s2 = (*scale) * (*scale);
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long i = idx % px, j = idx / px;
    double acc = 0.0;
    if (i > 0 && i < nx && j > 0 && j < ny)
      for (int k = 0; k < nz; ++k) {
        const cpx<T> v = psi[((long long)k * ny + j) * nx + i];
        acc += (double)v.x * v.x + (double)v.y * v.y;
      }
    out[idx] = s2 * acc * hz;
  }
}

static int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 65536) b = 65536;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t launch_init_analytic(bool fp64, void* psi, int nx, int ny, int nz, int dim,
                                 double x0, double hx, double y0, double hy, double z0,
                                 double hz, int function, int phase_mode, const double* R,
                                 unsigned long long seed, double d_xy, double d_z,
                                 cudaStream_t s) {
  const int threads = 256, blocks = grid_for((long long)nx * ny * nz, threads);
  if (fp64)
    k_init_analytic<double><<<blocks, threads, 0, s>>>(static_cast<cpx<double>*>(psi), nx, ny,
                                                       nz, dim, x0, hx, y0, hy, z0, hz,
                                                       function, phase_mode, R, seed, d_xy, d_z);
  else
    k_init_analytic<float><<<blocks, threads, 0, s>>>(static_cast<cpx<float>*>(psi), nx, ny, nz,
                                                      dim, x0, hx, y0, hy, z0, hz, function,
                                                      phase_mode, R, seed, d_xy, d_z);
  return cudaGetLastError();
}

static long long row_tasks(long long rows, int points) {
  return rows * ((points + kRowPart - 1) / kRowPart);
}

cudaError_t launch_load(bool fp64_store, bool fp64_src, const void* src, void* psi, int nx, int ny,
                        int nz, int dim, double vol, bool normalise, double* partials,
                        unsigned* counter, double* scale, double* norm, int* flags, int blocks,
                        cudaStream_t s) {
#define ROTGP_LD(TS, TD)                                                                       \
  do {                                                                                         \
    const bool rows = row_copy<TS, TD>() && nx >= kRowLeast;                                   \
    const long long work = rows ? (row_tasks((long long)ny * nz, nx) + 7) / 8                  \
                                : ((long long)nx * ny * nz + 255) / 256;                       \
    auto fn = rows ? (normalise ? k_load<TS, TD, true, row_copy<TS, TD>()>                     \
                                : k_load<TS, TD, false, row_copy<TS, TD>()>)                   \
                   : (normalise ? k_load<TS, TD, true, false> : k_load<TS, TD, false, false>); \
    fn<<<(int)std::min<long long>(blocks, work), 256, 0, s>>>(                                 \
        static_cast<const cpx<TS>*>(src), static_cast<cpx<TD>*>(psi), nx, ny, nz, dim, vol,    \
        partials, counter, scale, norm, flags);                                                \
  } while (0)
  if (fp64_src) {
    if (fp64_store) ROTGP_LD(double, double); else ROTGP_LD(double, float);
  } else {
    if (fp64_store) ROTGP_LD(float, double); else ROTGP_LD(float, float);
  }
#undef ROTGP_LD
  return cudaGetLastError();
}

cudaError_t launch_unpack(bool fp64_store, bool fp64_dst, const void* psi, void* dst, int nx,
                          int ny, int nz, int dim, const double* scale, cudaStream_t s) {
  const long long rows_out = (long long)(ny + 1) * (dim == 3 ? nz + 1 : 1);
#define ROTGP_UP(TS, TD)                                                                       \
  do {                                                                                         \
    const bool rows = row_copy<TS, TD>() && nx >= kRowLeast;                                   \
    const long long work = rows ? (row_tasks(rows_out, nx + 1) + 7) / 8                        \
                                : (rows_out * (nx + 1) + 255) / 256;                           \
    auto fn = rows ? k_store<TS, TD, row_copy<TS, TD>()> : k_store<TS, TD, false>;             \
    fn<<<(int)std::min<long long>(rows ? 152 * 8 : 65536, work), 256, 0, s>>>(                 \
        static_cast<const cpx<TS>*>(psi), static_cast<cpx<TD>*>(dst), nx, ny, nz, dim, scale); \
  } while (0)
  if (fp64_store) {
    if (fp64_dst) ROTGP_UP(double, double); else ROTGP_UP(double, float);
  } else {
    if (fp64_dst) ROTGP_UP(float, double); else ROTGP_UP(float, float);
  }
#undef ROTGP_UP
  return cudaGetLastError();
}

cudaError_t launch_column_density(bool fp64, const void* psi, double* out, int nx, int ny,
                                  int nz, double hz, const double* scale, cudaStream_t s) {
  const int threads = 256, blocks = grid_for((long long)(nx + 1) * (ny + 1), threads);
  if (fp64)
    k_column_density<double><<<blocks, threads, 0, s>>>(static_cast<const cpx<double>*>(psi), out,
                                                        nx, ny, nz, hz, scale);
  else
    k_column_density<float><<<blocks, threads, 0, s>>>(static_cast<const cpx<float>*>(psi), out,
                                                       nx, ny, nz, hz, scale);
  return cudaGetLastError();
}

cudaError_t launch_set_scalar(double* p, double v, cudaStream_t s) {
  k_set_scalar<<<1, 1, 0, s>>>(p, v);
  return cudaGetLastError();
}

}  // namespace rotgp
