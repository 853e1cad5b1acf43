// Parameter blocks and launchers of the solver and element-wise kernels (krylov.cu).
#pragma once

#include "common.cuh"
#include "passes.cuh"

namespace lsgpu {

enum ScalarPhase : int { PH_RESID = 0, PH_ALPHA = 1, PH_OMEGA = 2, PH_RHO = 3 };

// debug build: the index-check record of krylov.cu (debug_bounds.cuh)
unsigned bounds_site_krylov(bool clear);

struct UpdParams {
  SlotSel sel;
  size_t n, vstride;
  float2* r;                // the field is read from the slot's x and written to its xo
  const float2 *p, *s, *t, *rh;
  double* partials;
  int maxparts = 0;   // partial-sum blocks allocated per slot (0: not checked)
};

struct ScalarParams {
  SlotDev* slots;
  unsigned mask;
  int phase;
  const double* partials;   // [slot][nparts][4]
  int nparts;
  size_t n;                 // voxels per slot
};

// States of the slots of one operator call: each reads x and writes xo.  The vectors come by value, so that the
// launch holds all it needs: an upload from host memory would be repeated from there by a captured graph.
struct OperatorSlots {
  static constexpr int kMax = 128;   // views per launch (2 KB of parameters)
  SlotDev* slots;           // of the launch's first view
  int n;
  const float* f;
  int adjoint;
  const float2* x[kMax];
  float2* xo[kMax];
};

struct PlaneWaveParams {
  int nx, ny, nz;
  double h;
  const double* k;          // device, 3 per view
  float2* const* out;       // device array of device pointers
  float2* tables = nullptr; // per-view 1-D phase factors (allocated by the launcher)
};

struct PadParams {
  SlotSel sel;
  int nx, ny, mx, my, ox, oy;
  const float2* const* src;   // device array of per-slot detector arrays
  float2* dst; size_t dst_stride;
};

struct GradParams {
  size_t n;
  int nslots;
  const float2* const* u;     // device array of forward fields
  const SlotDev* slots;       // the adjoint fields w_s = slots[s].x
  const float* c;             // device, per-slot weights
  float* grad;
};

struct ResidualParams {
  size_t count;
  const float2* const* pred;
  const float2* const* meas;
  float2* const* res;
  double* partials;           // [view][nblocks][4]
};

void launch_operator_slots(const OperatorSlots& a, size_t voxels, cudaStream_t st);
void launch_update(const UpdParams& a, int nblocks, int nslots, cudaStream_t st);
void launch_scalar(const ScalarParams& a, int nslots, cudaStream_t st);
void launch_zero_shadow(const SlotDev* slots, int slot, float2* rh, size_t n, cudaStream_t st);
void launch_inner(const ResidualParams& a, int nblocks, int nviews, cudaStream_t st);
cudaError_t launch_plane_waves(const PlaneWaveParams& a, int nviews, cudaStream_t st);
void launch_potential(const float* dn, size_t count, double eta_b, double kb, float* f, cudaStream_t st);
void launch_far_reduce(const FarPassParams& a, int nslots, cudaStream_t st);
void launch_pad_detector(const PadParams& a, int nslots, cudaStream_t st);
void launch_gradient(const GradParams& a, cudaStream_t st);
void launch_residual(const ResidualParams& a, int nblocks, int nviews, cudaStream_t st);

}  // namespace lsgpu
