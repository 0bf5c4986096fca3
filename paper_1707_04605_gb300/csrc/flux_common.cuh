// Device parts shared by the flux path's kernels (mixed.cu, resident_flux.cu).
#pragma once

#include <cuda_runtime.h>

#include "kernels.cuh"

namespace mg {
namespace {

__device__ __forceinline__ float4 fma4f(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
// Sources [s0, s1) of a row's shots 4 c4 .. 4 c4 + 3.
__device__ __forceinline__ void add_source(const DevEvents& ev, int s0, int s1, int c4, float f,
                                           float4& rhs) {
  for (int s = s0; s < s1; ++s) {
    const int d = __ldg(ev.src_shot + s) - 4 * c4;
    if (d == 0) rhs.x += f;
    if (d == 1) rhs.y += f;
    if (d == 2) rhs.z += f;
    if (d == 3) rhs.w += f;
  }
}
// Receivers [r0, r1) of a row's shots: sample l of their traces.
__device__ __forceinline__ void record(const DevEvents& ev, int r0, int r1, int c4, float* traces,
                                       int nt, int l, const float4& pv) {
  for (int r = r0; r < r1; ++r) {
    const int d = __ldg(ev.rec_shot + r) - 4 * c4;
    if (d < 0 || d > 3) continue;
    const float v = d == 0 ? pv.x : d == 1 ? pv.y : d == 2 ? pv.z : pv.w;
    traces[(int64_t)__ldg(ev.rec_trace + r) * nt + l] = v;
  }
}

// Geometry packed so that a warp reads a cell's constants with a few 16-byte
// loads: cell e, kCellW<D> float4: its D + 1 rows, then the gradients [a][k].
template <int D>
constexpr int kCellW = ((D + 1) * (D + 1) + 3) / 4;

}  // namespace
}  // namespace mg
