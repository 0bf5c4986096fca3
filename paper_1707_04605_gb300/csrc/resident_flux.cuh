// Device parts shared by the resident kernels of the flux system
// (resident_flux.h): the patch's tables in shared memory and a step's cells.
#pragma once

#include "flux_common.cuh"
#include "resident_common.cuh"
#include "resident_flux.h"

namespace mg {
namespace {

// Constants in shared memory.  Three dimensions: a cell's slots (byte offsets),
// gradients and damping factors in 5 float4, an incidence {offset of the cell,
// weights}.  Two dimensions, smaller (36 bytes per cell and 12 per incidence
// instead of 48 and 16: 62,641 nodes then fit 4 lanes per row, not 2): gradients
// and factors in two planes of float4, the slots packed; {offset, weight}, and a
// plane of the other weight.
constexpr int kSlotBits = 10;
template <int D>
constexpr int kRecW = D == 2 ? 2 : 5;                 // float4 per cell
template <int D>
constexpr int kIncBytes = D == 2 ? 8 : 16;
template <int D>
constexpr int kCellMore = D == 2 ? 4 : 0;             // bytes in the other planes
template <int D>
constexpr int kIncMore = D == 2 ? 4 : 0;

// Advances the patch's cells [c0, c1), thread t of `threads` taking every
// threads-th float4: q <- keep q + dt sum g p, SIGN < 0: q <- keep q - sum g p.
template <int D, int LPR, int SIGN>
__device__ __forceinline__ void step_cells(unsigned cell0, unsigned slots, int max_cells,
                                           unsigned p0, unsigned q0, unsigned qk,
                                           int c0, int c1, int t, int threads, float dt) {
#pragma unroll 1
  for (int i = c0 * LPR + t; i < c1 * LPR; i += threads) {
    const int e = i / LPR;
    float w[4 * 5];   // slots, gradients, factors
    if (D == 2) {
      const float4 x = lds4(cell0 + e * 16), y = lds4(cell0 + (max_cells + e) * 16);
      const int v = lds1(slots + e * 4);
#pragma unroll
      for (int a = 0; a <= D; ++a)
        w[a] = __int_as_float((v >> (a * kSlotBits) & ((1 << kSlotBits) - 1)) * (16 * LPR));
      w[3] = x.x;
      w[4] = x.y;
      w[5] = x.z;
      w[6] = x.w;
      w[7] = y.x;
      w[8] = y.y;
      w[9] = y.z;
      w[10] = y.w;
    } else {
#pragma unroll
      for (int j = 0; j < kRecW<D>; ++j) {
        const float4 x = lds4(cell0 + e * (16 * kRecW<D>) + 16 * j);
        w[4 * j] = x.x;
        w[4 * j + 1] = x.y;
        w[4 * j + 2] = x.z;
        w[4 * j + 3] = x.w;
      }
    }
    float4 pv[D + 1], o[D];
#pragma unroll
    for (int a = 0; a <= D; ++a) pv[a] = lds4(p0 + __float_as_uint(w[a]));
    const unsigned q = q0 + e * (16 * LPR);
#pragma unroll
    for (int k = 0; k < D; ++k) o[k] = lds4(q + k * qk);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int a = 0; a <= D; ++a) acc = fma4f(w[D + 1 + a * D + k], pv[a], acc);
      const float kp = w[(D + 1) * (D + 1) + k];
      sts4(q + k * qk,
           SIGN > 0 ? make_float4(fmaf(kp, o[k].x, dt * acc.x), fmaf(kp, o[k].y, dt * acc.y),
                                  fmaf(kp, o[k].z, dt * acc.z), fmaf(kp, o[k].w, dt * acc.w))
                    : make_float4(fmaf(kp, o[k].x, -acc.x), fmaf(kp, o[k].y, -acc.y),
                                  fmaf(kp, o[k].z, -acc.z), fmaf(kp, o[k].w, -acc.w)));
    }
  }
}

// The patch's parts and its constants in shared memory: cells, incidences
// {offset of the cell, weights}, rows {coefficients, incidences, row | event},
// exchange rows of the halo.
struct FluxPatch {
  int r0, own, h0, halo, e0, cells, border, inner, x0;
  float4* cell;
  int4* row;
  unsigned char* inc;
  double* sums;         // per own row, when asked for
  int *slots, *halo_x;
  float* w1;
};

template <int D, int LPR>
__device__ __forceinline__ FluxPatch fill_flux(const DevFluxPatches& P, const DevEvents& ev,
                                               const float4* __restrict__ geo,
                                               const float* __restrict__ keep,
                                               const float2* __restrict__ coef, void* at,
                                               bool sums) {
  constexpr int SLOT = 16 * LPR;
  const int b = blockIdx.x, tid = threadIdx.x, threads = blockDim.x;
  FluxPatch t;
  t.r0 = __ldg(P.own_off + b);
  t.own = __ldg(P.own_off + b + 1) - t.r0;
  t.h0 = __ldg(P.halo_off + b);
  t.halo = __ldg(P.halo_off + b + 1) - t.h0;
  t.e0 = __ldg(P.cell_off + b);
  t.cells = __ldg(P.cell_off + b + 1) - t.e0;
  t.border = __ldg(P.border + b);
  t.inner = __ldg(P.inner + b);
  t.x0 = __ldg(P.x_off + b);
  t.cell = static_cast<float4*>(at);
  t.row = reinterpret_cast<int4*>(t.cell + P.max_cells * kRecW<D>);
  t.inc = reinterpret_cast<unsigned char*>(t.row + P.max_own);
  t.sums = reinterpret_cast<double*>(t.inc + (size_t)P.max_inc * kIncBytes<D>);
  t.slots = reinterpret_cast<int*>(t.sums + (sums ? P.max_own : 0));
  t.w1 = reinterpret_cast<float*>(t.slots + P.max_cells * (kCellMore<D> / 4));
  t.halo_x = reinterpret_cast<int*>(t.w1 + P.max_inc * (kIncMore<D> / 4));
  const int i0 = __ldg(P.inc_off + b), incs = __ldg(P.inc_off + b + 1) - i0;
  for (int i = tid; i < t.cells; i += threads) {
    int e = __ldg(P.cell + t.e0 + i);
    if (e < 0) e = ~e;
    float w[4 * 5] = {}, c[4 * kCellW<D>];   // gradients and factors, the packed cell
    for (int j = 0; j < kCellW<D>; ++j) {
      const float4 x = __ldg(geo + (int64_t)e * kCellW<D> + j);
      c[4 * j] = x.x;
      c[4 * j + 1] = x.y;
      c[4 * j + 2] = x.z;
      c[4 * j + 3] = x.w;
    }
    constexpr int G = D == 2 ? 0 : D + 1;
    int packed = 0;
    for (int j = 0; j <= D; ++j) {
      const int v = __ldg(P.cell_slot + (size_t)(t.e0 + i) * 4 + j);
      if (D == 2) packed |= v << (j * kSlotBits);
      else w[j] = __int_as_float(v * SLOT);
    }
    for (int j = 0; j < (D + 1) * D; ++j) w[G + j] = c[D + 1 + j];
    for (int k = 0; k < D; ++k) w[G + (D + 1) * D + k] = __ldg(keep + (int64_t)e * D + k);
    for (int j = 0; j < kRecW<D>; ++j)
      t.cell[D == 2 ? j * P.max_cells + i : i * kRecW<D> + j] =
          make_float4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    if (D == 2) t.slots[i] = packed;
  }
  for (int i = tid; i < incs; i += threads) {
    int4 q = __ldg(P.inc + i0 + i);
    q.x *= SLOT;
    if (D == 2) {
      reinterpret_cast<int2*>(t.inc)[i] = make_int2(q.x, q.y);
      t.w1[i] = __int_as_float(q.z);
    } else {
      reinterpret_cast<int4*>(t.inc)[i] = q;
    }
  }
  for (int i = tid; i < t.own; i += threads) {
    int r = __ldg(P.row + t.r0 + i);
    const float2 c = __ldg(coef + r);
    if (__ldg(ev.src_ptr + r) != __ldg(ev.src_ptr + r + 1) ||
        __ldg(ev.rec_ptr + r) != __ldg(ev.rec_ptr + r + 1))
      r |= kEventBit;
    t.row[i] = make_int4(__float_as_int(c.x), __float_as_int(c.y), __ldg(P.row_inc + t.r0 + i), r);
  }
  for (int i = tid; i < t.halo; i += threads) t.halo_x[i] = __ldg(P.halo_x + t.h0 + i);
  return t;
}

// Fluxes [k][m][ld] of the patch's cells into shared memory (q null: zero), and
// those that the patch owns back.
template <int D, int LPR>
__device__ __forceinline__ void load_fluxes(const DevFluxPatches& P, const FluxPatch& t,
                                            const float* q, int64_t m, int ld4, int c4, unsigned qs,
                                            unsigned qk) {
  for (int i = threadIdx.x; i < t.cells * LPR; i += blockDim.x) {
    int e = __ldg(P.cell + t.e0 + i / LPR);
    if (e < 0) e = ~e;
    for (int k = 0; k < D; ++k)
      sts4(qs + k * qk + i * 16, q && c4 < ld4 ? *(reinterpret_cast<const float4*>(q) +
                                                   ((int64_t)k * m + e) * ld4 + c4)
                                               : make_float4(0.f, 0.f, 0.f, 0.f));
  }
}
template <int D, int LPR>
__device__ __forceinline__ void store_fluxes(const DevFluxPatches& P, const FluxPatch& t, float* q,
                                             int64_t m, int ld4, int c4, unsigned qs, unsigned qk) {
  for (int i = threadIdx.x; i < t.cells * LPR; i += blockDim.x) {
    const int e = __ldg(P.cell + t.e0 + i / LPR);
    if (e < 0 || c4 >= ld4) continue;
    for (int k = 0; k < D; ++k)
      reinterpret_cast<float4*>(q)[((int64_t)k * m + e) * ld4 + c4] = lds4(qs + k * qk + i * 16);
  }
}

// sum_k w[e,i,k] q^(k)_e over a row's incidences `inc`, in their order.
template <int D>
__device__ __forceinline__ float4 row_fluxes(int inc, unsigned inc0, unsigned w1, unsigned ql,
                                             unsigned qk) {
  float4 bt = make_float4(0.f, 0.f, 0.f, 0.f);
  int s = inc & ((1 << kIncShift) - 1);
  const int end = s + (inc >> kIncShift);
#pragma unroll 2
  for (; s < end; ++s) {
    if (D == 2) {
      const int2 w = lds2(inc0 + s * 8);
      const float v = __int_as_float(lds1(w1 + s * 4));
      const unsigned q = ql + w.x;
      bt = fma4f(__int_as_float(w.y), lds4(q), bt);
      bt = fma4f(v, lds4(q + qk), bt);
    } else {
      const float4 w = lds4(inc0 + s * 16);
      const unsigned q = ql + __float_as_uint(w.x);
#pragma unroll
      for (int k = 0; k < D; ++k)
        bt = fma4f(k == 0 ? w.y : k == 1 ? w.z : w.w, lds4(q + k * qk), bt);
    }
  }
  return bt;
}

// Threads that copy the halo: all units in flight at once, an eighth of the
// warps at most.
__device__ __forceinline__ int copy_threads(int units) {
  return 32 * min(max(1, (int)blockDim.x / 256), (units + 32 * kFetch - 1) / (32 * kFetch));
}

}  // namespace
}  // namespace mg
