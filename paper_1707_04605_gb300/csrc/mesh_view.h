// Read-only view of a mesh handle's resident data, for entry points that
// live outside capi.cu.
#pragma once

#include <cstdint>
#include <mutex>
#include <vector>

#include "../../include/mgwave.h"
#include "kernels.cuh"
#include "resident_flux.h"

namespace mg {

struct MeshView {
  int device;
  int bc;
  int64_t n;                 // rows
  int64_t m;                 // finest cells
  DevEll K;                  // sliced-ELL stiffness
  CoefArgs coef_base;        // incidence arrays for the coefficients (eps, dt, outputs unset)
  const double* row_abs;     // sum_j |K_ij| per row (device)
  const int32_t* perm_host;  // caller node -> row (host, [n])
  int64_t* launches;         // the handle's launch counter
  int batch;                 // gather batch of the untiled kernels
};

int mesh_view(mg_mesh* mesh, MeshView* out);

// Padded shot count (row stride of the states) of a batch of S shots.
int padded_shots(int S);

// Loads the module of mg_forward_noalloc's fixed device array and its
// kernels on device `dev` (current) and caches the array's address there.
int noalloc_prepare(int dev);

struct HostMesh;
// Host image of a handle's mesh (read-only), its device, and a way to count
// launches made on its behalf by entry points outside capi.cu.
const HostMesh* host_mesh(const mg_mesh* mesh);
int mesh_device(const mg_mesh* mesh);
int mesh_graph_chunk(const mg_mesh* mesh);   // steps per CUDA-graph chunk (0: off)
void add_launches(mg_mesh* mesh, int64_t n);
// Outputs that the handle's calls have set to NaN so far because a device wait
// ran out; synchronises with the stream.
int mesh_poisoned(mg_mesh* mesh, cudaStream_t st, int* count);

// Work buffers of the flux path's calls: taken from the handle for a call, and
// left on it again (false: it holds a set already).
struct FluxBuffer {
  void* p;
  size_t bytes;
};
void mesh_take_scratch(mg_mesh* mesh, std::vector<FluxBuffer>& bufs);
bool mesh_keep_scratch(mg_mesh* mesh, std::vector<FluxBuffer>& bufs);

// Packed geometry of the flux path, kept on the handle.
struct FluxGeometry {
  const float4* cell = nullptr;      // per cell: rows, gradients
  const int32_t* inc_ptr = nullptr;  // [n + 1]
  const int4* inc = nullptr;         // per node and incident cell: {cell, weights}
  const int32_t* cells = nullptr;    // [m][d + 1] rows
  DevFluxPatches patches{};          // B = 0: no resident kernel for this mesh
};
std::mutex& mesh_flux_mutex(mg_mesh* mesh);   // held around the next two
bool mesh_flux_geometry(mg_mesh* mesh, FluxGeometry* out);   // false: not built yet
int mesh_set_flux_geometry(mg_mesh* mesh, const std::vector<float>& cell,
                           const std::vector<int32_t>& inc_ptr, const std::vector<int4>& inc,
                           const HostFluxPatches& patches, FluxGeometry* out);
long long mesh_wait_budget(const mg_mesh* mesh);   // clock cycles of one device wait

// One problem of a multi-instance batch, prepared on its own handle: device
// inputs staged, coefficients and FP32 wavelet computed, event lists built,
// and the handle's state / checkpoint / accumulator buffers sized.
struct InstanceView {
  DevEll K;
  DevEvents ev;
  const float4* coef;
  const float* wavelet;
  const double* eps;        // device copy or caller pointer
  int S, S_pad, tiles;
  int64_t R, n;
  float* A; float* B; float* C; float* D;  // n * S_pad floats each
  float* ckpt;              // [nck][2][n][S_pad] when requested
  float* seg;               // [K+2][n][S_pad] when requested
  float* tr;                // [R][nt] internal trace buffer
  float* G;                 // [4][tiles][n] Kahan accumulators when requested
  const float* w;           // [R][nt] staged weights when given
  int64_t* launches;
};

// ckpt_every > 0 sizes checkpoint and segment buffers; w (device or host
// per flags) is staged when non-null.
int prepare_instance(mg_mesh* mesh, const double* eps, const mg_shots* shots,
                     const double* wavelet, double dt, int nt, int flags, void* stream,
                     int ckpt_every, const float* w, InstanceView* out);

// FP64 per-cell gradient from the instance's accumulators, restricted to
// `level` into g (device pointer, or host pointer with MG_HOST_PTRS).
int finish_gradient(mg_mesh* mesh, int level, const double* eps_dev, double dt, int tiles,
                    double* g, int flags, void* stream);

}  // namespace mg
