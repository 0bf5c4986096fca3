// Resident kernels (resident_common.cuh): the states of a group of shots stay
// on chip for many steps, each CTA holding one patch of the mesh.  Host tables
// (resident_plan.cpp) and the launch interface.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>
#include <new>
#include <vector>

#include "kernels.cuh"
#include "mg_internal.h"

namespace mg {

// A thread's marks over all rows or cells while it works on one patch: zero
// pages of which a patch touches few.
struct Stamps {
  int32_t* p;
  explicit Stamps(int64_t n) : p(static_cast<int32_t*>(std::calloc(n, sizeof(int32_t)))) {}
  void need() const {
    if (!p) throw std::bad_alloc();
  }
  ~Stamps() { std::free(p); }
  Stamps(const Stamps&) = delete;
  Stamps& operator=(const Stamps&) = delete;
  int32_t& operator[](int64_t i) { return p[i]; }
};

// Runs one iteration of a parallel loop, which no exception may leave: memory
// that it does not get is counted.
template <class F>
void no_throw(int& oom, F&& body) {
  try {
    body();
  } catch (const std::bad_alloc&) {
    ++oom;
  }
}

// Rows cut into B patches: a patch's border rows (coupled to rows of other
// patches) first, then its inner rows.
struct HostPatches {
  int B = 0;
  std::vector<int32_t> part;       // [n] patch of each row
  std::vector<int32_t> own_off;    // [B + 1] into row
  std::vector<int32_t> n_border;   // [B]
  std::vector<int32_t> row;
  std::vector<std::vector<int32_t>> halo;   // per patch: rows of others that it reads
};
// MG_ERR_UNSUPPORTED when the coupling of two patches is not mutual, MG_ERR_OOM
// when the host's memory runs out.
int build_patches(const HostMesh& hm, int B, HostPatches& out);

// The rows in groups of rpw that a warp advances together (rpw = 32 / lanes
// per row), border and inner rows apart, each kind padded to whole groups.  A
// patch's slots: row k of group g at g rpw + k, then its halo rows.  A row's
// off-diagonal entries go in pairs p at first + p rpw + k of its group.
// Border slots are exchange rows in order.
constexpr int kPairShift = 20, kPairMask = 0x7ff;
constexpr int kEventBit = (int)0x80000000;   // set on the device: sources or receivers
struct HostGroups {
  struct Pair {
    int32_t slot[2];
    float val[2];
  };
  std::vector<int32_t> grp_off, border, pair_off, halo_off, x_off;   // per patch
  std::vector<int32_t> hdr;          // per group: first pair (of the patch) | pairs << kPairShift
  std::vector<int32_t> row;          // per own slot: row or -1
  std::vector<float> diag;
  std::vector<Pair> pair;
  std::vector<int32_t> halo, halo_x; // rows and exchange rows of the halo slots
  int uniform = 0;                   // pairs of every row when all are alike, else 0
  int max_pairs = 0, max_groups = 0, max_halo = 0, max_slots = 0;                 // of a patch
};
void group_rows(const HostMesh& hm, const HostPatches& P, int rpw, HostGroups& out);

// Device image of the groups.
struct DevPatches {
  int32_t B, n_x, uniform;   // patches, exchange rows
  int32_t max_pairs, max_groups, max_halo, max_slots;
  const int32_t *grp_off, *border, *pair_off, *halo_off, *x_off, *hdr, *row, *halo, *halo_x;
  const float* diag;
  const int4* pair;
};

// Launch shape: lpr lanes per row (4 lpr columns).
constexpr int kResidentThreads = 1024;
struct ResidentShape {
  int lpr = 0, warps = 0, smem = 0;
};

struct ResidentArgs {
  DevPatches P;
  DevEvents ev;
  const float4* coef;
  const float* wavelet;
  float* traces;            // [n_traces][nt] or null
  const float2* tcoef;      // tangent: its coefficients and the traces of dp
  float* dtraces;
  int32_t nt, step0, steps; // steps step0 .. step0 + steps - 1
  int32_t ld, col0;         // shot columns [col0, col0 + 4 lpr) of rows of ld floats
  const float *p, *pm;      // p_l, p_{l-1} at step0, or null: zero
  float *out_p, *out_pm;    // the last two states, or null
  float* hist;              // p_{l+1} of step step0 + j at hist + j * state, or null
  int64_t state;
  uint4* xbuf;              // exchange rows, [2][n_x][lpr][2], zeroed before the launch
  int* status;
  long long budget;         // SM clock cycles one wait may take
};

// Reverse steps k, k - 1, ... (`steps` of them) on the source tile of shot
// columns [col0, col0 + 4 lpr).
struct ResidentAdjArgs {
  DevPatches P;
  DevEvents ev;
  const float4* coef;
  const float* w;           // [n_traces][nt] trace weights
  int32_t nt, k, steps, ld, col0;
  float *mu, *mu1;          // mu_k, mu_{k+1}; then those after the last step
  const float* pk;          // p_k; p_{k-j} is j * state floats before it
  int64_t state;
  float *G, *Gc, *H, *Hc;   // [n] sums of the tile
  uint4* xbuf;
  int* status;
  long long budget;
};

// Shape of lpr lanes per row with row_bytes more bytes of shared memory per
// own row; MG_ERR_UNSUPPORTED when a patch does not fit smem_max bytes.
int resident_fit(const DevPatches& D, int lpr, int row_bytes, int smem_max, ResidentShape& s);
// Raises the dynamic shared memory limit of a kernel on the current device.
int resident_smem_limit(const void* kern, int smem);
int launch_resident_step(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st);
// p and dp of 2 lpr shots, from rest.
int launch_resident_tangent(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st);
int launch_resident_adjoint(const ResidentAdjArgs& a, const ResidentShape& s, cudaStream_t st);
// *kept <- *status (null: 0).  A copy of 4 bytes between two kernels in its place
// took about 20 us of a call of 620.
int launch_note_kept(const int* status, int* kept, cudaStream_t st);
// x[0..n) <- NaN, *status <- 1 and *count + 1 if *a or *b is not 0 (each may be
// null): results of a launch whose wait ran out.
int launch_poison(float* x, int64_t n, const int* a, const int* b, int* status, int* count,
                  cudaStream_t st);

}  // namespace mg
