// tails.cuh -- complex-float sweeps by two geometric tails per line, in
// shared-memory tiles (tails.cu).
#pragma once

#include "common.cuh"

namespace rotgp {

// Tile of 32 lines: warps of L own points each along the line.
struct tail_shape {
  int L = 0, nw = 0, tiles = 0;
  size_t smem = 0;
  long long blocks = 0;
};
// For `lines` lines of N points (x: rows, else columns of nx); false if the
// form does not serve them (a line no longer than the halo).
bool tail_plan(int axis, int N, int nx, long long lines, int halo, bool imag, size_t smem_limit,
               tail_shape* s);

struct tail_args {
  const float2* in;
  float2* out;
  const float2* tab;    // weights [al, be, g2, gc][line] (launch_res_tables)
  int tlines;
  int nx, ny, axis, len, H;
  tail_shape sh;
  long long lines;
  // H1 (x): as stream_args
  float dt, g, hgam2, hnu2, hlam2, x0, hx;
  double y0, hy, z0, hz;
  const double* scale;
  // norm of the last sweep
  double vol;
  int imag;
  double* partials;
  unsigned* counter;
  double* scale_out;
  double* norm_out;
  int* flags;
};
cudaError_t launch_tail_x(bool imag, const tail_args& a, cudaStream_t s);
cudaError_t launch_tail_s(bool reduce, const tail_args& a, cudaStream_t s);

}  // namespace rotgp
