// resident.cuh -- the on-chip 2D stepper (resident.cu): one cooperative launch
// for a block of split steps of one condensate whose tiles stay in the shared
// memory of the SMs.
#pragma once

#include "common.cuh"

namespace rotgp {

// Most CTAs of a launch (one per SM; at most 255), and steps per table build of a schedule.
constexpr int kResMaxCtas = 160;
constexpr int kResSchedule = 32;
constexpr int kResPlanes = 4;  // weights of a line: al, be, g2, gc

// Tiles of a launch: tiles_x x tiles_y CTAs, each a tile of about
// nx / tiles_x x ny / tiles_y points with halos of H points.
struct res_plan {
  int H = 0, L = 0;          // halo; own points of a segment
  int tiles_x = 0, tiles_y = 0;
  int pa = 0, pb = 0;        // shared-memory pitches (points) of the two tiles
  int rows = 0;              // rows of a tile with its halos
  int cols = 0;              // most own columns of a tile
  size_t smem = 0;           // dynamic shared memory of a CTA
};

// Exchange of the norm: two words that take the shares of alternate rounds,
// their values after the last rounds of the last launch, and the number of
// steps so far (the tags of the halo points go on from launch to launch).
struct res_sync {
  unsigned long long word[2][16];
  unsigned long long base[2];
  unsigned epoch;
};

struct res_args {
  const float2* in;          // state buffers, pitch nx
  float2* out;
  // two planes through which tiles exchange halos: a point is two words
  // (re, im) that carry the tag of their step
  unsigned long long* xbuf;
  size_t xplane;             // words of a plane
  const float2* tabx;        // weight planes [f][line] of the x and y lines
  const float2* taby;
  long long step_x, step_y;  // from one step's tables to the next (0: the same)
  int nx, ny;
  res_plan plan;
  float dt, g, hgam2, hnu2;
  double x0, hx, y0, hy, vol;
  double* scale;             // pending scale in, scale and norm out
  double* norm;
  int* flags;                // bit 0 non-finite norm, bit 3 a wait gave up
  res_sync* sync;
  int ex0;                   // scale of the first shares: 2^ex0 near 1/vol
  int nsteps;
};

// Tile plan for an nx x ny state whose truncated carries need `halo` points;
// false when it has none (halo above 16, or tiles beyond the shared memory).
bool res_make_plan(int nx, int ny, int halo, bool imag, int sm_count, size_t smem_limit,
                   res_plan* p);
cudaError_t launch_resident(bool imag, const res_args& a, cudaStream_t s);

// Weights [al, be, g2, gc][line] of one axis (resident.cu) for nsteps rotation
// frequencies in turn; co holds tau per unit of omega.  iters: steps after
// which the multiplier recursion has converged.
struct res_omegas {
  double v[kResSchedule];
};
cudaError_t launch_res_tables(float2* tab, int nlines, int iters, const axis_coef& co,
                              const res_omegas& om, int nsteps, cudaStream_t s);

// Does a step of this mode of the context run in the on-chip stepper?
bool ctx_resident(const rotgp_ctx* c, bool imag);
// Its time per step of a block of n: alone, one launch over the whole chip; or
// in launches of its own beside other instances', what it adds to them, and the
// least time of a step.
struct ctx_cost {
  double alone, beside, least;
};
ctx_cost ctx_step_cost(const rotgp_ctx* c, bool imag, long long n);
// Build what steps of this mode would build first (a capture would record it).
int ctx_prepare(rotgp_ctx* c, bool imag);
// Steps from here on beside other instances' (no launch over the whole chip).
void ctx_set_beside(rotgp_ctx* c, bool on);
// Points over which a line carry of the context stays above the rounding of
// the exact partition solve (hybrid.cuh).
int ctx_carry_reach(const rotgp_ctx* c);

}  // namespace rotgp
