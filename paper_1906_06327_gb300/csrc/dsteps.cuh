// dsteps.cuh -- imaginary-time steps in complex double (dsteps.cu).
#pragma once

#include "common.cuh"

namespace rotgp {

constexpr int kDPow = 64;  // powers of the tails kept per line (the largest halo)

// Weights of the lines of one axis, planes of double2 [f][line]: al, be, mu =
// m - 1 (m the converged Thomas multiplier), then al^0 .. al^(kDPow - 1), then the
// powers of be; powers past the halo are zero.
constexpr int kDPlanes = 3 + 2 * kDPow;
cudaError_t launch_dtables(double2* tab, int nlines, int halo, const axis_coef& co, cudaStream_t s);

struct dline_args {
  const double2* in;
  double2* out;
  const double2* tab;
  int tlines;            // lines of the table (z: 1)
  int nx, ny, nz;
  int axis, len, halo;
  long long lines;       // lines of the sweep
  int seg;               // columns: own points of a segment
  // H1 substep and pending scale (rows of the x sweep)
  double dt, g, hgam2, hnu2, hlam2, x0, hx, y0, hy, z0, hz;
  // norm of the last sweep (as norm_epilogue wants it)
  double vol;
  int imag;
  double* partials;
  unsigned* counter;
  double* scale_out;
  double* norm_out;
  int* flags;
  const double* scale;
};

// Rows (x sweep with H1): points per lane for lines of N points, at most 16 (512
// points); 0 if none.
int drow_points(int N, int halo);
cudaError_t launch_drows(const dline_args& a, int P, cudaStream_t s);
// Columns (y and z sweeps): own points of a segment (0: none, lines of more than
// 96 points with a halo above 48), and the blocks.
int dcol_segment(int N, long long lines, int halo, int sm_count);
long long dcol_blocks(int nx, long long lines, int len, int seg);
cudaError_t launch_dcols(bool reduce, const dline_args& a, cudaStream_t s);

// A block of 2D steps in one cooperative launch.
struct dsync {
  unsigned long long word[2][16];  // exchange words of alternate rounds: hi, lo
  unsigned long long base[2][2];   // their values after the last launch
};
struct dstep_args {
  double2* psi[2];                 // the state, and the state after the x sweep
  const double2* tabx;
  const double2* taby;
  int nx, ny, halo, nsteps, ex0;
  double dt, g, hgam2, hnu2, x0, hx, y0, hy, vol;
  double* scale;
  double* norm;
  int* flags;
  dsync* sync;
};
// Can lines of nx (at most 512) and ny (1,024) points with this halo run there?
bool dstep_fits(int nx, int ny, int halo);
cudaError_t launch_dsteps(const dstep_args& a, int sm_count, cudaStream_t s);

}  // namespace rotgp
