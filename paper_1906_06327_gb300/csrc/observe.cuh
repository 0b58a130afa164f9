// observe.cuh -- observables and vortex count of a context's state (reduce.cu)
// and its loading (io.cu): the parts that share block sums.
#pragma once

#include "../../include/rotgp.h"
#include "common.cuh"

namespace rotgp {

// The sums of one pass over the state (scaled by the pending renormalisation),
// in this order; V is the trap potential, lap the three-point Laplacian, D
// the central differences, _4 the fourth-order forms.
enum {
  OS_RE2,   // psi_R^2
  OS_IM2,   // psi_I^2
  OS_LR,    // psi_R (-lap psi_R/2 + V psi_R + Omega (y D_x psi_I - x D_y psi_I))
  OS_LI,    // the same for the state rotated by -i (R <- I, I <- -R)
  OS_NR,    // |psi|^2 psi_R^2
  OS_NI,    // |psi|^2 psi_I^2
  OS_X2,    // x^2 |psi|^2
  OS_Y2,
  OS_Z2,
  OS_L4,    // Re psi^* (-lap_4/2 + V - Omega L_z4) psi
  OS_P0,    // |psi|^2, x^2 |psi|^2, y^2 |psi|^2 of the plane of the vortex count
  OS_PX2,
  OS_PY2,
  OS_MAX = 15,  // largest |psi|^2
  OS_COUNT = 16
};

// R^2 of the vortex count's ellipse per axis, and 1/R^2 in float
struct observe_ellipse {
  double r2[2];
  float inv[2];
};

struct observe_args {
  const void* psi;
  int nx, ny, nz, dim, kplane;
  double hx, hy, hz, x0, y0, z0;
  double hgam2, hnu2, hlam2, omega;
  const double* scale;
  int chunk;            // points of a march (z in 3D, y in 2D) per work item
  double* partials;     // OS_COUNT per block
  unsigned* counter;
  double* sums;         // OS_COUNT doubles
  int* count;           // vortices
  observe_ellipse* ellipse;
  float fx0, fy0, fhx, fhy;  // centre of plaquette (0, 0), spacings
};

// Work split: points per march and blocks for a state on this many SMs.
void observe_shape(int nx, int ny, int nz, int dim, int sm_count, int* chunk, int* blocks);
constexpr int kObserveBlocksPerSm = 2;  // most blocks: this times the SMs
cudaError_t launch_observe(bool fp64, const observe_args& a, int blocks, cudaStream_t s);
// The vortices in the ellipse that launch_observe left.
cudaError_t launch_vortex_count(bool fp64, const observe_args& a, cudaStream_t s);

// ABI layout -> device layout, the norm of the loaded state, and from it the
// pending scale (normalise) or 1; flags bit 0 as the step reductions set it.
// blocks: at most as many as partials has room for OS_COUNT each.
cudaError_t launch_load(bool fp64_store, bool fp64_src, const void* src, void* psi, int nx, int ny,
                        int nz, int dim, double vol, bool normalise, double* partials,
                        unsigned* counter, double* scale, double* norm, int* flags, int blocks,
                        cudaStream_t s);

// rotgp_observables in two parts (rotgp.cu): enqueue, then wait and form the
// results, so that many contexts' evaluations can be in flight together.
int ctx_observe(rotgp_ctx* c);
int ctx_observed(rotgp_ctx* c, rotgp_obs* out);

}  // namespace rotgp
