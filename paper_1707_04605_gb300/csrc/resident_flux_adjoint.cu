// Resident kernel of the flux system's reverse steps: the adjoint pressures of
// own rows, the scaled ones r of own and halo rows, the adjoint fluxes of the
// patch's cells and the rows' FP64 sums stay in shared memory for a whole
// segment; p_k and p_{k+1} come from the kept states.
//
// The lanes of a row are a whole group of the node adjoint's sum over the shots
// (32 float4, or all when there are fewer): the same tree, the same bits.
//
// A step: rows, border rows first, whose r goes out; the cells without halo
// rows, while the last warps copy the halo's r; the cells with halo rows.
// Bound as the forward kernel (resident_flux.cu), and by the latency of three
// barriers, one exchange and the kept states on small patches: 15,769 nodes, 32
// shots, the gradient of 300 steps 4.9 -> 3.5 ms, 4.5 us less per reverse step
// than two launches.
#include "resident_flux.cuh"

namespace mg {
namespace {

template <int D, int LPR>
__global__ void __launch_bounds__(kResidentThreads, 1)
    k_resident_flux_adj(ResidentFluxAdjArgs a) {
  constexpr int SLOT = 16 * LPR;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int failed;
  const int tid = threadIdx.x, threads = blockDim.x;
  const DevFluxPatches& P = a.P;
  // r of every slot, tp of the own ones, fluxes, constants, sums
  const unsigned rs = smem_u32(sm), ts = rs + P.max_slots * SLOT, qs = ts + P.max_own * SLOT;
  const unsigned qk = P.max_cells * SLOT;
  const FluxPatch t =
      fill_flux<D, LPR>(P, a.ev, a.cell, a.keep, a.coef,
                        sm + (size_t)(P.max_slots + P.max_own + D * P.max_cells) * SLOT, true);
  double* const hs = t.sums;
  const int own = t.own;
  const int ld4 = a.ld / 4, c4 = a.col0 / 4 + tid % LPR, seg = a.col0 / 128;
  const bool start = a.k == a.nt - 1;
  if (tid == 0) failed = 0;
  for (int i = tid; i < own * LPR; i += threads) {
    const int r = __ldg(P.row + t.r0 + i / LPR);
    sts4(ts + i * 16, start ? make_float4(0.f, 0.f, 0.f, 0.f)
                            : reinterpret_cast<const float4*>(a.tp)[(int64_t)r * ld4 + c4]);
  }
  for (int i = tid; i < own; i += threads)
    hs[i] = a.hacc[(int64_t)__ldg(P.row + t.r0 + i) * a.nseg + seg];
  load_fluxes<D, LPR>(P, t, a.Qt, a.m, ld4, c4, qs, qk);
  __syncthreads();

  unsigned rl = rs + tid % LPR * 16, tl = ts + tid % LPR * 16, ql = qs + tid % LPR * 16,
           cell0 = smem_u32(t.cell), inc0 = smem_u32(t.inc), row0 = smem_u32(t.row),
           slots0 = smem_u32(t.slots), w10 = smem_u32(t.w1);
  asm volatile("" : "+r"(rl), "+r"(tl), "+r"(ql), "+r"(cell0), "+r"(inc0), "+r"(row0),
               "+r"(slots0), "+r"(w10));
  const int units = t.halo * 2 * LPR, copy = copy_threads(units);
  const size_t xhalf = (size_t)P.n_x * (2 * LPR);
  const unsigned gmask = LPR == 32 ? 0xffffffffu
                                   : (((1u << (LPR & 31)) - 1u) << ((tid & 31) & ~(LPR - 1)));
  // the states of a thread's first row are read a step ahead
  const float4* pk = reinterpret_cast<const float4*>(a.p) + c4;
  const int64_t st4 = a.state / 4;
  const int64_t first =
      tid < own * LPR ? (int64_t)__ldg(P.row + t.r0 + tid / LPR) * ld4 : 0;
  float4 n1 = __ldg(pk + st4 + first), n0 = __ldg(pk + first);
  for (int j = 0; j < a.steps; ++j) {
    const int l = a.k - j;
    uint4* const xo = a.xbuf + (size_t)(j & 1) * xhalf + (size_t)t.x0 * (2 * LPR);
#pragma unroll 1
    for (int i = tid; i < own * LPR; i += threads) {
      const float4 rw = lds4(row0 + i / LPR * 16);
      const int r = __float_as_int(rw.w), rr = r & ~kEventBit;
      const int64_t at = (int64_t)rr * ld4;
      const float4 x1 = i == tid ? n1 : __ldg(pk + st4 + at), x0 = i == tid ? n0 : __ldg(pk + at);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (!start || j > 0)
        v = fma4f(a.dt, row_fluxes<D>(__float_as_int(rw.z), inc0, w10, ql, qk),
                  lds4(tl + i / LPR * SLOT));
      if (r < 0)
        for (int q = __ldg(a.ev.rec_ptr + rr); q < __ldg(a.ev.rec_ptr + rr + 1); ++q) {
          const int d = __ldg(a.ev.rec_shot + q) - 4 * c4;
          if (d < 0 || d > 3) continue;
          const float w = __ldg(a.w + (int64_t)__ldg(a.ev.rec_trace + q) * a.nt + l);
          if (d == 0) v.x += w;
          if (d == 1) v.y += w;
          if (d == 2) v.z += w;
          if (d == 3) v.w += w;
        }
      float h = v.x * (x1.x - x0.x);
      h = fmaf(v.y, x1.y - x0.y, h);
      h = fmaf(v.z, x1.z - x0.z, h);
      h = fmaf(v.w, x1.w - x0.w, h);
#pragma unroll
      for (int off = LPR / 2; off > 0; off >>= 1) h += __shfl_xor_sync(gmask, h, off);
      if (tid % LPR == 0) hs[i / LPR] += (double)h;
      const float4 o = make_float4(v.x * rw.x, v.y * rw.x, v.z * rw.x, v.w * rw.x);
      if (i < t.border * LPR) xstore(xo + (size_t)i * 2, o, (unsigned)(j + 1));
      sts4(rl + i / LPR * SLOT, o);
      sts4(tl + i / LPR * SLOT, make_float4(fmaf(-rw.y, o.x, v.x), fmaf(-rw.y, o.y, v.y),
                                            fmaf(-rw.y, o.z, v.z), fmaf(-rw.y, o.w, v.w)));
    }
    pk -= st4;
    if (j + 1 < a.steps) {
      n1 = n0;
      n0 = __ldg(pk + first);
    }
    __syncthreads();
    if (units > 0 && tid >= threads - copy) {
      if (!fetch_halo<LPR>(a.xbuf + (size_t)(j & 1) * xhalf, smem_u32(t.halo_x), rs + own * SLOT,
                           units, (unsigned)(j + 1), tid - (threads - copy), copy, a.status,
                           a.budget))
        failed = 1;
    } else {
      step_cells<D, LPR, -1>(cell0, slots0, P.max_cells, rl, ql, qk, 0, t.inner, tid,
                             units > 0 ? threads - copy : threads, 1.0f);
    }
    __syncthreads();
    if (failed) return;
    step_cells<D, LPR, -1>(cell0, slots0, P.max_cells, rl, ql, qk, t.inner, t.cells, tid, threads, 1.0f);
    __syncthreads();
  }
  for (int i = tid; i < own * LPR; i += threads)
    reinterpret_cast<float4*>(a.tp)[(int64_t)__ldg(P.row + t.r0 + i / LPR) * ld4 + c4] =
        lds4(ts + i * 16);
  for (int i = tid; i < own; i += threads)
    a.hacc[(int64_t)__ldg(P.row + t.r0 + i) * a.nseg + seg] = hs[i];
  store_fluxes<D, LPR>(P, t, a.Qt, a.m, ld4, c4, qs, qk);
}

template <int D>
int launch_dim(const ResidentFluxAdjArgs& a, const ResidentShape& s, cudaStream_t st) {
  switch (s.lpr) {
    case 1: return launch_resident(k_resident_flux_adj<D, 1>, a, s, st);
    case 2: return launch_resident(k_resident_flux_adj<D, 2>, a, s, st);
    case 4: return launch_resident(k_resident_flux_adj<D, 4>, a, s, st);
    case 8: return launch_resident(k_resident_flux_adj<D, 8>, a, s, st);
    case 16: return launch_resident(k_resident_flux_adj<D, 16>, a, s, st);
    case 32: return launch_resident(k_resident_flux_adj<D, 32>, a, s, st);
  }
  return MG_ERR_ARG;
}

}  // namespace

int launch_resident_flux_adj(const ResidentFluxAdjArgs& a, int d, const ResidentShape& s,
                             cudaStream_t st) {
  return d == 2 ? launch_dim<2>(a, s, st) : launch_dim<3>(a, s, st);
}

}  // namespace mg
