// Host side of the resident kernels (shapes, limits) and the forward kernel's
// instances.
#include <algorithm>
#include <map>
#include <mutex>

#include "resident_step.cuh"

namespace mg {
namespace {

__global__ void k_note_kept(const int* status, int* kept) { *kept = status ? *status : 0; }

// (a may be status: every block finds it set, whoever comes first)
__global__ void k_poison(float* x, int64_t n, const int* a, const int* b, int* status,
                         int* count) {
  if (!(a && *a) && !(b && *b)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *status = 1;
    ++*count;
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = __int_as_float(0x7fffffff);
}

}  // namespace

int resident_smem_limit(const void* kern, int smem) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int> done;   // (kernel, device) -> limit set
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MG_ERR_CUDA;
  std::lock_guard<std::mutex> lock(mu);
  int& have = done[{kern, dev}];
  if (have >= smem) return MG_OK;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess) {
    cudaGetLastError();
    return MG_ERR_UNSUPPORTED;
  }
  have = smem;
  return MG_OK;
}

int resident_fit(const DevPatches& D, int lpr, int row_bytes, int smem_max, ResidentShape& s) {
  const int rpw = 32 / lpr;
  s.lpr = lpr;
  s.smem = 2 * D.max_slots * 16 * lpr + 16 * D.max_pairs +
           (16 + 4 + row_bytes) * D.max_groups * rpw + 4 * (D.max_halo + D.max_groups + 4);
  if (s.smem > smem_max) return MG_ERR_UNSUPPORTED;
  // a warp for each group, and at least one of each kind
  s.warps = std::min(kResidentThreads / 32, D.max_groups + 1);
  return MG_OK;
}

int launch_resident_step(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st) {
  switch (s.lpr) {
    case 1: return launch_lpr<1, false>(a, s, st);
    case 2: return launch_lpr<2, false>(a, s, st);
    case 4: return launch_lpr<4, false>(a, s, st);
    case 8: return launch_lpr<8, false>(a, s, st);
    case 16: return launch_lpr<16, false>(a, s, st);
    case 32: return launch_lpr<32, false>(a, s, st);
  }
  return MG_ERR_ARG;
}

int launch_note_kept(const int* status, int* kept, cudaStream_t st) {
  k_note_kept<<<1, 1, 0, st>>>(status, kept);
  return check_launch();
}

int launch_poison(float* x, int64_t n, const int* a, const int* b, int* status, int* count,
                  cudaStream_t st) {
  if (n <= 0) return MG_OK;
  k_poison<<<(unsigned)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, st>>>(x, n, a, b, status,
                                                                               count);
  return check_launch();
}

}  // namespace mg
