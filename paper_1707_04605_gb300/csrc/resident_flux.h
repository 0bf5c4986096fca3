// Resident kernels of the first-order flux system (mixed.cu): the pressures of a
// patch's rows and halo rows and the fluxes of every cell that touches an own
// row stay in shared memory for many steps.  A cell on the border is advanced
// by each patch that needs it, with the same operations on the same values, so
// that only border pressures travel (resident_common.cuh's exchange).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "kernels.cuh"
#include "mg_internal.h"
#include "resident.h"

namespace mg {

// Per patch: own rows (border rows first; slot = position), halo rows, cells
// (those without a halo row first), and per own row its incidences in the mesh's
// order as {cell of the patch, weights}.
struct HostFluxPatches {
  int B = 0;
  std::vector<int32_t> own_off, border, halo_off, x_off, cell_off, inner, inc_off;
  std::vector<int32_t> row, row_inc;        // per own row: row, first | count << kIncShift
  std::vector<int32_t> halo, halo_x;
  std::vector<int32_t> cell;                // cell, or ~cell where another patch owns it
  std::vector<int32_t> cell_slot;           // [cells][4] slots of its rows
  std::vector<int4> inc;
  int max_own = 0, max_halo = 0, max_slots = 0, max_cells = 0, max_inc = 0;
};
constexpr int kIncShift = 20;
// geo_inc: {cell, weights} per incidence of hm.nc_ptr.  MG_ERR_UNSUPPORTED when
// the mesh cannot be cut so.
int build_flux_patches(const HostMesh& hm, int B, const std::vector<int4>& geo_inc,
                       HostFluxPatches& out);

struct DevFluxPatches {
  int32_t B, n_x, max_own, max_halo, max_slots, max_cells, max_inc;
  const int32_t *own_off, *border, *halo_off, *x_off, *cell_off, *inner, *inc_off;
  const int32_t *row, *row_inc, *halo, *halo_x, *cell, *cell_slot;
  const int4* inc;
};

struct ResidentFluxArgs {
  DevFluxPatches P;
  DevEvents ev;
  const float2* coef;
  const float4* cell;       // packed cells (mixed.cu)
  const float* keep;
  const float* fl;
  float* traces;
  int32_t nt, step0, steps, ld, col0;
  int64_t m;
  float dt;
  const float *p, *q;       // p_l, q_{l-1/2} at step0, or null: zero
  float *out_p, *out_q;     // those after the last step, or null
  float* hist;              // p_{l+1} of step step0 + j at hist + j * state, or null
  int64_t state;
  uint4* xbuf;
  int* status;
  long long budget;
};

// Reverse steps k, k - 1, ... (`steps` of them) on the shot columns [col0, col0 +
// 4 lpr), a whole group of the node adjoint's sum over the shots.
struct ResidentFluxAdjArgs {
  DevFluxPatches P;
  DevEvents ev;
  const float2* coef;
  const float4* cell;
  const float* keep;
  const float* w;           // [n_traces][nt] trace weights
  int32_t nt, k, steps, ld, col0, nseg;
  int64_t m;
  float dt;
  const float* p;           // p_k; p_{k+1} state floats after it, p_{k-j} before it
  int64_t state;
  float *tp, *Qt;           // adjoint states, read (not at step nt - 1) and written
  double* hacc;             // [n][nseg]
  uint4* xbuf;
  int* status;
  long long budget;
};

// Lanes per row (4 columns each) whose patches fit smem_max bytes and whose
// launches take the least time by the estimate; us: that of a step of ld4 float4
// columns.  shape.lpr = 0: none fits.
void resident_flux_shape(const DevFluxPatches& P, int d, int ld4, int smem_max,
                         ResidentShape& shape, double& us);
// The same for reverse steps, whose lanes are given: min(32, ld4).
void resident_flux_adj_shape(const DevFluxPatches& P, int d, int ld4, int smem_max,
                             ResidentShape& shape, double& us);
int launch_resident_flux(const ResidentFluxArgs& a, int d, const ResidentShape& s,
                         cudaStream_t st);
int launch_resident_flux_adj(const ResidentFluxAdjArgs& a, int d, const ResidentShape& s,
                             cudaStream_t st);

}  // namespace mg
