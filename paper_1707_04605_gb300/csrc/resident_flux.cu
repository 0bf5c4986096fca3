// Resident kernel of the flux system's forward steps: one cooperative launch
// advances the patches (resident_flux.h) for 4 LPR shots.
//
// Bound by shared memory: a cell reads D + 1 pressures and reads and writes D
// fluxes, a row reads D fluxes per incident cell (42 accesses of 16 bytes per
// row and 4 columns in two dimensions), against two launches per step whose
// gathers go through L2.  Us per step, launches -> resident (lanes per row that
// fit): 62,641 nodes, 128 shots 91.6 -> 59.8 (2), 4 shots 9.8 -> 2.8 (1);
// 15,769 nodes, 32 shots 8.1 -> 3.1 (8), 128 shots 17.1 -> 11.5 (16); 3,997
// nodes, 10 shots 5.9 -> 2.1 (4), 256 shots 11.2 -> 10.4 (32); 4,199 nodes of
// tetrahedra, 64 shots 29.8 -> 18.3 (4).
//
// A step: the last warps copy the halo pressures while the others advance the
// cells without halo rows; the cells with halo rows; the rows, border rows
// first, whose new pressures go out at once.  Three barriers, one state: a
// pressure is overwritten only after every cell has read it.
#include <algorithm>

#include "flux_common.cuh"
#include "resident_common.cuh"
#include "resident_flux.h"

namespace mg {
namespace {

// A cell in shared memory: slots (byte offsets), gradients, damping factors.
template <int D>
constexpr int kRecW = ((D + 1) * (D + 1) + D + 3) / 4;   // float4: 3, 5

// Advances the patch's cells [c0, c1): group i of 32 / LPR cells of warp w of nw.
template <int D, int LPR>
__device__ __forceinline__ void step_cells(unsigned cell0, unsigned p0, unsigned q0, unsigned qk,
                                           int c0, int c1, int t, int threads, float dt) {
#pragma unroll 1
  for (int i = c0 * LPR + t; i < c1 * LPR; i += threads) {
    const int e = i / LPR;
    float w[4 * kRecW<D>];
#pragma unroll
    for (int j = 0; j < kRecW<D>; ++j) {
      const float4 x = lds4(cell0 + e * (16 * kRecW<D>) + 16 * j);
      w[4 * j] = x.x;
      w[4 * j + 1] = x.y;
      w[4 * j + 2] = x.z;
      w[4 * j + 3] = x.w;
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
      sts4(q + k * qk, make_float4(fmaf(kp, o[k].x, dt * acc.x), fmaf(kp, o[k].y, dt * acc.y),
                                   fmaf(kp, o[k].z, dt * acc.z), fmaf(kp, o[k].w, dt * acc.w)));
    }
  }
}

template <int D, int LPR>
__global__ void __launch_bounds__(kResidentThreads, 1) k_resident_flux(ResidentFluxArgs a) {
  constexpr int SLOT = 16 * LPR;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int failed;
  const int b = blockIdx.x, tid = threadIdx.x, threads = blockDim.x;
  const DevFluxPatches& P = a.P;
  const int r0 = __ldg(P.own_off + b), own = __ldg(P.own_off + b + 1) - r0;
  const int h0 = __ldg(P.halo_off + b), halo = __ldg(P.halo_off + b + 1) - h0;
  const int e0 = __ldg(P.cell_off + b), cells = __ldg(P.cell_off + b + 1) - e0;
  const int i0 = __ldg(P.inc_off + b), incs = __ldg(P.inc_off + b + 1) - i0;
  const int border = __ldg(P.border + b), inner = __ldg(P.inner + b), x0 = __ldg(P.x_off + b);
  // states, cells, incidences, rows {coef, incidences, row | event}, halo rows
  const unsigned ps = smem_u32(sm), qs = ps + P.max_slots * SLOT;
  const unsigned qk = P.max_cells * SLOT;
  float4* const cell_s = reinterpret_cast<float4*>(sm + (size_t)(P.max_slots + D * P.max_cells) * SLOT);
  int4* const inc_s = reinterpret_cast<int4*>(cell_s + P.max_cells * kRecW<D>);
  int4* const row_s = inc_s + P.max_inc;
  int* const halo_s = reinterpret_cast<int*>(row_s + P.max_own);
  if (tid == 0) failed = 0;
  for (int i = tid; i < cells; i += threads) {
    int e = __ldg(P.cell + e0 + i);
    if (e < 0) e = ~e;
    float w[4 * kRecW<D>] = {}, c[4 * kCellW<D>];
    for (int j = 0; j < kCellW<D>; ++j) {
      const float4 x = __ldg(a.cell + (int64_t)e * kCellW<D> + j);
      c[4 * j] = x.x;
      c[4 * j + 1] = x.y;
      c[4 * j + 2] = x.z;
      c[4 * j + 3] = x.w;
    }
    for (int j = 0; j <= D; ++j)
      w[j] = __int_as_float(__ldg(P.cell_slot + (size_t)(e0 + i) * 4 + j) * SLOT);
    for (int j = D + 1; j < (D + 1) * (D + 1); ++j) w[j] = c[j];
    for (int k = 0; k < D; ++k) w[(D + 1) * (D + 1) + k] = __ldg(a.keep + (int64_t)e * D + k);
    for (int j = 0; j < kRecW<D>; ++j)
      cell_s[i * kRecW<D> + j] = make_float4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  }
  for (int i = tid; i < incs; i += threads) {
    int4 q = __ldg(P.inc + i0 + i);
    q.x *= SLOT;
    inc_s[i] = q;
  }
  for (int i = tid; i < own; i += threads) {
    int r = __ldg(P.row + r0 + i);
    const float2 c = __ldg(a.coef + r);
    if (__ldg(a.ev.src_ptr + r) != __ldg(a.ev.src_ptr + r + 1) ||
        __ldg(a.ev.rec_ptr + r) != __ldg(a.ev.rec_ptr + r + 1))
      r |= kEventBit;
    row_s[i] = make_int4(__float_as_int(c.x), __float_as_int(c.y), __ldg(P.row_inc + r0 + i), r);
  }
  for (int i = tid; i < halo; i += threads) halo_s[i] = __ldg(P.halo_x + h0 + i);
  const int ld4 = a.ld / 4;
  for (int i = tid; i < (own + halo) * LPR; i += threads) {
    const int s = i / LPR, c4 = a.col0 / 4 + i % LPR;
    const int r = s < own ? __ldg(P.row + r0 + s) : __ldg(P.halo + h0 + s - own);
    sts4(ps + i * 16, a.p && c4 < ld4 ? __ldg(reinterpret_cast<const float4*>(a.p) +
                                              (int64_t)r * ld4 + c4)
                                      : make_float4(0.f, 0.f, 0.f, 0.f));
  }
  for (int i = tid; i < cells * LPR; i += threads) {
    const int c4 = a.col0 / 4 + i % LPR;
    int e = __ldg(P.cell + e0 + i / LPR);
    if (e < 0) e = ~e;
    for (int k = 0; k < D; ++k)
      sts4(qs + k * qk + i * 16,
           a.q && c4 < ld4 ? __ldg(reinterpret_cast<const float4*>(a.q) +
                                   ((int64_t)k * a.m + e) * ld4 + c4)
                           : make_float4(0.f, 0.f, 0.f, 0.f));
  }
  __syncthreads();

  // a lane keeps its column: the strides over items are whole warps
  const int c4 = a.col0 / 4 + tid % LPR;
  unsigned pl = ps + tid % LPR * 16, ql = qs + tid % LPR * 16, cell0 = smem_u32(cell_s),
           inc0 = smem_u32(inc_s), row0 = smem_u32(row_s);
  asm volatile("" : "+r"(pl), "+r"(ql), "+r"(cell0), "+r"(inc0), "+r"(row0));
  const int units = halo * 2 * LPR;
  // warps that copy the halo: all units in flight at once, an eighth at least
  const int copy = 32 * min(max(1, threads / 256), (units + 32 * kFetch - 1) / (32 * kFetch));
  const size_t xhalf = (size_t)P.n_x * (2 * LPR);
  for (int j = 0; j < a.steps; ++j) {
    const bool wait = j > 0 && units > 0;
    if (wait && tid >= threads - copy) {
      if (!fetch_halo<LPR>(a.xbuf + (size_t)(j & 1) * xhalf, smem_u32(halo_s), ps + own * SLOT,
                           units, (unsigned)j, tid - (threads - copy), copy, a.status, a.budget))
        failed = 1;
    } else {
      step_cells<D, LPR>(cell0, pl, ql, qk, 0, inner, tid, wait ? threads - copy : threads, a.dt);
    }
    __syncthreads();
    if (failed) return;
    step_cells<D, LPR>(cell0, pl, ql, qk, inner, cells, tid, threads, a.dt);
    __syncthreads();
    const int l = a.step0 + j;
    uint4* const xo = a.xbuf + (size_t)((j & 1) ^ 1) * xhalf + (size_t)x0 * (2 * LPR);
#pragma unroll 1
    for (int i = tid; i < own * LPR; i += threads) {
      const float4 rw = lds4(row0 + i / LPR * 16);
      const unsigned at = pl + i / LPR * SLOT;
      float4 pv = lds4(at);
      const int inc = __float_as_int(rw.z), r = __float_as_int(rw.w);
      float4 bt = make_float4(0.f, 0.f, 0.f, 0.f);
      unsigned s = inc0 + (inc & ((1 << kIncShift) - 1)) * 16;
      const unsigned end = s + (inc >> kIncShift) * 16;
#pragma unroll 2
      for (; s < end; s += 16) {
        const float4 w = lds4(s);
        const unsigned q = ql + __float_as_uint(w.x);
#pragma unroll
        for (int k = 0; k < D; ++k) bt = fma4f(k == 0 ? w.y : k == 1 ? w.z : w.w, lds4(q + k * qk), bt);
      }
      float4 rhs = make_float4(-bt.x, -bt.y, -bt.z, -bt.w);
      const int rr = r & ~kEventBit;
      if (r < 0) {
        const int s0 = __ldg(a.ev.src_ptr + rr), s1 = __ldg(a.ev.src_ptr + rr + 1);
        if (s0 != s1) add_source(a.ev, s0, s1, c4, __ldg(a.fl + l), rhs);
      }
      pv.x = fmaf(rw.x, fmaf(-rw.y, pv.x, rhs.x), pv.x);
      pv.y = fmaf(rw.x, fmaf(-rw.y, pv.y, rhs.y), pv.y);
      pv.z = fmaf(rw.x, fmaf(-rw.y, pv.z, rhs.z), pv.z);
      pv.w = fmaf(rw.x, fmaf(-rw.y, pv.w, rhs.w), pv.w);
      if (i < border * LPR) xstore(xo + (size_t)i * 2, pv, (unsigned)(j + 1));
      sts4(at, pv);
      if (r < 0 && a.traces)
        record(a.ev, __ldg(a.ev.rec_ptr + rr), __ldg(a.ev.rec_ptr + rr + 1), c4, a.traces, a.nt, l,
               pv);
      if (a.hist && c4 < ld4)
        reinterpret_cast<float4*>(a.hist + (size_t)j * a.state)[(int64_t)rr * ld4 + c4] = pv;
    }
    __syncthreads();
  }
  if (!a.out_p || c4 >= ld4) return;
  for (int i = tid; i < own * LPR; i += threads)
    reinterpret_cast<float4*>(a.out_p)[(int64_t)__ldg(P.row + r0 + i / LPR) * ld4 + c4] =
        lds4(ps + i * 16);
  for (int i = tid; i < cells * LPR; i += threads) {
    const int e = __ldg(P.cell + e0 + i / LPR);
    if (e < 0) continue;
    for (int k = 0; k < D; ++k)
      reinterpret_cast<float4*>(a.out_q)[((int64_t)k * a.m + e) * ld4 + c4] =
          lds4(qs + k * qk + i * 16);
  }
}

template <int D>
int launch_dim(const ResidentFluxArgs& a, const ResidentShape& s, cudaStream_t st) {
  switch (s.lpr) {
    case 1: return launch_resident(k_resident_flux<D, 1>, a, s, st);
    case 2: return launch_resident(k_resident_flux<D, 2>, a, s, st);
    case 4: return launch_resident(k_resident_flux<D, 4>, a, s, st);
    case 8: return launch_resident(k_resident_flux<D, 8>, a, s, st);
    case 16: return launch_resident(k_resident_flux<D, 16>, a, s, st);
    case 32: return launch_resident(k_resident_flux<D, 32>, a, s, st);
  }
  return MG_ERR_ARG;
}

}  // namespace

void resident_flux_shape(const DevFluxPatches& P, int d, int ld4, int smem_max,
                         ResidentShape& shape, double& us) {
  shape = ResidentShape();
  us = 0.0;
  const int rec = d == 2 ? kRecW<2> : kRecW<3>;
  for (int lpr = 1; lpr <= 32; lpr <<= 1) {
    if (lpr > 1 && lpr / 2 >= ld4) break;
    const int64_t smem = (int64_t)(P.max_slots + d * P.max_cells) * 16 * lpr +
                         16 * ((int64_t)P.max_cells * rec + P.max_inc + P.max_own) +
                         4 * P.max_halo;
    if (smem > smem_max) break;
    // from measurements on 3,997, 15,769 and 62,641 nodes of triangles and 4,199 of
    // tetrahedra, most within 15% of them: barriers and exchange, halo, the
    // states' and the constants' accesses to shared memory
    const double states = P.max_cells * (3.0 * d + 1.0) + (double)P.max_inc * d + 2.0 * P.max_own;
    const double constants = (double)P.max_cells * rec + P.max_inc + P.max_own;
    const double step = 1.2 + 4e-3 * P.max_halo + 0.775e-4 * lpr * states + 0.8e-4 * constants;
    const double all = (ld4 + lpr - 1) / lpr * step;
    if (shape.lpr && all >= us) continue;
    us = all;
    shape.lpr = lpr;
    shape.smem = (int)smem;
    shape.warps = std::min<int64_t>(
        kResidentThreads / 32,
        1 + ((int64_t)std::max(P.max_own, P.max_cells) * lpr + 31) / 32);
  }
}

int launch_resident_flux(const ResidentFluxArgs& a, int d, const ResidentShape& s,
                         cudaStream_t st) {
  return d == 2 ? launch_dim<2>(a, s, st) : launch_dim<3>(a, s, st);
}

}  // namespace mg
