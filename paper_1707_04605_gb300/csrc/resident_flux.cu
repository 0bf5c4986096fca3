// Resident kernel of the flux system's forward steps: one cooperative launch
// advances the patches (resident_flux.h) for 4 LPR shots.
//
// Bound by shared memory: a cell reads D + 1 pressures and reads and writes D
// fluxes, a row reads D fluxes per incident cell (42 accesses of 16 bytes per
// row and 4 columns in two dimensions), against two launches per step whose
// gathers go through L2.  Us per step, launches -> resident (lanes per row that
// fit): 62,641 nodes, 128 shots 91.6 -> 44 (4; 60 with 2), 4 shots 9.8 -> 2.8 (1);
// 15,769 nodes, 32 shots 8.1 -> 3.1 (8), 128 shots 17.1 -> 11.5 (16); 3,997
// nodes, 10 shots 5.9 -> 2.1 (4), 256 shots 11.2 -> 10.4 (32); 4,199 nodes of
// tetrahedra, 64 shots 29.8 -> 18.3 (4).
//
// A step: the last warps copy the halo pressures while the others advance the
// cells without halo rows; the cells with halo rows; the rows, border rows
// first, whose new pressures go out at once.  Three barriers, one state: a
// pressure is overwritten only after every cell has read it.
#include <algorithm>

#include "resident_flux.cuh"

namespace mg {
namespace {

template <int D, int LPR>
__global__ void __launch_bounds__(kResidentThreads, 1) k_resident_flux(ResidentFluxArgs a) {
  constexpr int SLOT = 16 * LPR;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int failed;
  const int tid = threadIdx.x, threads = blockDim.x;
  const DevFluxPatches& P = a.P;
  const unsigned ps = smem_u32(sm), qs = ps + P.max_slots * SLOT;
  const unsigned qk = P.max_cells * SLOT;
  const FluxPatch t = fill_flux<D, LPR>(P, a.ev, a.cell, a.keep, a.coef,
                                        sm + (size_t)(P.max_slots + D * P.max_cells) * SLOT, false);
  const int own = t.own;
  if (tid == 0) failed = 0;
  // a lane keeps its column: the strides over items are whole warps
  const int ld4 = a.ld / 4, c4 = a.col0 / 4 + tid % LPR;
  for (int i = tid; i < (own + t.halo) * LPR; i += threads) {
    const int s = i / LPR;
    const int r = s < own ? __ldg(P.row + t.r0 + s) : __ldg(P.halo + t.h0 + s - own);
    sts4(ps + i * 16, a.p && c4 < ld4 ? __ldg(reinterpret_cast<const float4*>(a.p) +
                                              (int64_t)r * ld4 + c4)
                                      : make_float4(0.f, 0.f, 0.f, 0.f));
  }
  load_fluxes<D, LPR>(P, t, a.q, a.m, ld4, c4, qs, qk);
  __syncthreads();

  unsigned pl = ps + tid % LPR * 16, ql = qs + tid % LPR * 16, cell0 = smem_u32(t.cell),
           inc0 = smem_u32(t.inc), row0 = smem_u32(t.row),
           slots0 = smem_u32(t.slots), w10 = smem_u32(t.w1);
  asm volatile("" : "+r"(pl), "+r"(ql), "+r"(cell0), "+r"(inc0), "+r"(row0),
               "+r"(slots0), "+r"(w10));
  const int units = t.halo * 2 * LPR;
  const int copy = copy_threads(units);
  const size_t xhalf = (size_t)P.n_x * (2 * LPR);
  for (int j = 0; j < a.steps; ++j) {
    const bool wait = j > 0 && units > 0;
    if (wait && tid >= threads - copy) {
      if (!fetch_halo<LPR>(a.xbuf + (size_t)(j & 1) * xhalf, smem_u32(t.halo_x), ps + own * SLOT,
                           units, (unsigned)j, tid - (threads - copy), copy, a.status, a.budget))
        failed = 1;
    } else {
      step_cells<D, LPR, 1>(cell0, slots0, P.max_cells, pl, ql, qk, 0, t.inner, tid, wait ? threads - copy : threads, a.dt);
    }
    __syncthreads();
    if (failed) return;
    step_cells<D, LPR, 1>(cell0, slots0, P.max_cells, pl, ql, qk, t.inner, t.cells, tid, threads, a.dt);
    __syncthreads();
    const int l = a.step0 + j;
    uint4* const xo = a.xbuf + (size_t)((j & 1) ^ 1) * xhalf + (size_t)t.x0 * (2 * LPR);
#pragma unroll 1
    for (int i = tid; i < own * LPR; i += threads) {
      const float4 rw = lds4(row0 + i / LPR * 16);
      const unsigned at = pl + i / LPR * SLOT;
      float4 pv = lds4(at);
      const int inc = __float_as_int(rw.z), r = __float_as_int(rw.w);
      const float4 bt = row_fluxes<D>(inc, inc0, w10, ql, qk);
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
      if (i < t.border * LPR) xstore(xo + (size_t)i * 2, pv, (unsigned)(j + 1));
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
    reinterpret_cast<float4*>(a.out_p)[(int64_t)__ldg(P.row + t.r0 + i / LPR) * ld4 + c4] =
        lds4(ps + i * 16);
  store_fluxes<D, LPR>(P, t, a.out_q, a.m, ld4, c4, qs, qk);
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

namespace {

// Shared memory and time per step of a launch of lpr lanes per row, with
// `more` float4 slots of state and bytes per own row: from measurements on
// 3,997, 15,769 and 62,641 nodes of triangles and 4,199 of tetrahedra, most
// within 15% of them (barriers and exchange, halo, the states' and the
// constants' accesses to shared memory).
int64_t flux_smem(const DevFluxPatches& P, int d, int lpr, int more, int bytes) {
  if (d == 2 && P.max_slots > 1 << kSlotBits) return INT64_MAX;
  const int64_t cell = d == 2 ? 16 * kRecW<2> + kCellMore<2> : 16 * kRecW<3>;
  const int64_t inc = d == 2 ? kIncBytes<2> + kIncMore<2> : kIncBytes<3>;
  return (int64_t)(P.max_slots + more * P.max_own + d * P.max_cells) * 16 * lpr +
         P.max_cells * cell + P.max_inc * inc + P.max_own * (16 + bytes) + 4 * P.max_halo;
}
double flux_us(const DevFluxPatches& P, int d, int lpr) {
  const int rec = d == 2 ? 3 : 5;
  const double states = P.max_cells * (3.0 * d + 1.0) + (double)P.max_inc * d + 2.0 * P.max_own;
  const double constants = (double)P.max_cells * rec + P.max_inc + P.max_own;
  return 1.2 + 4e-3 * P.max_halo + 0.775e-4 * lpr * states + 0.8e-4 * constants;
}
int flux_warps(const DevFluxPatches& P, int lpr) {
  return (int)std::min<int64_t>(kResidentThreads / 32,
                                1 + ((int64_t)std::max(P.max_own, P.max_cells) * lpr + 31) / 32);
}

}  // namespace

void resident_flux_shape(const DevFluxPatches& P, int d, int ld4, int smem_max,
                         ResidentShape& shape, double& us) {
  shape = ResidentShape();
  us = 0.0;
  for (int lpr = 1; lpr <= 32 && (lpr == 1 || lpr / 2 < ld4); lpr <<= 1) {
    const int64_t smem = flux_smem(P, d, lpr, 0, 0);
    if (smem > smem_max) break;
    const double all = (ld4 + lpr - 1) / lpr * flux_us(P, d, lpr);
    if (shape.lpr && all >= us) continue;
    us = all;
    shape.lpr = lpr;
    shape.smem = (int)smem;
    shape.warps = flux_warps(P, lpr);
  }
}

void resident_flux_adj_shape(const DevFluxPatches& P, int d, int ld4, int smem_max,
                             ResidentShape& shape, double& us) {
  shape = ResidentShape();
  const int lpr = std::min(32, ld4);
  const int64_t smem = flux_smem(P, d, lpr, 1, sizeof(double));
  us = (ld4 + lpr - 1) / lpr * (flux_us(P, d, lpr) + 0.5);
  if (smem > smem_max || ld4 % lpr || (lpr & (lpr - 1))) return;
  shape.lpr = lpr;
  shape.smem = (int)smem;
  shape.warps = flux_warps(P, lpr);
}

int launch_resident_flux(const ResidentFluxArgs& a, int d, const ResidentShape& s,
                         cudaStream_t st) {
  return d == 2 ? launch_dim<2>(a, s, st) : launch_dim<3>(a, s, st);
}

}  // namespace mg
