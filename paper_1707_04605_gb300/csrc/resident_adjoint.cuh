#pragma once

// Resident reverse steps: mu_{k-1} from mu_k and mu_{k+1} as the forward kernel
// advances p (resident_step.cuh), the sums over the shots of p_k with the
// differences of mu per row, and their Kahan sums over the steps in shared
// memory.  A row's lanes hold one whole source tile of the row kernel (up to
// 128 shots, one float4 per lane), so its shuffle tree adds in the same order:
// the same bits.  p_k is read from the history; each lane fetches the one of
// its next group, or of its first group of the next step, ahead of the product.
#include "resident_common.cuh"

namespace mg {
namespace {

template <int LPR, bool U>
__global__ void __launch_bounds__(kResidentThreads, 1) k_resident_adjoint(ResidentAdjArgs a) {
  constexpr int RPW = 32 / LPR, SLOT = 16 * LPR;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int failed[2];   // by step parity: no warp can be two steps ahead of another
  const int b = blockIdx.x, tid = threadIdx.x, threads = blockDim.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const DevPatches& D = a.P;
  const unsigned buf = (unsigned)D.max_slots * SLOT;
  float4* const sums = reinterpret_cast<float4*>(sm + 2 * (size_t)buf);   // {G, Gc, H, Hc} per row
  const Patch t =
      patch_tables<RPW>(D, reinterpret_cast<unsigned char*>(sums + D.max_groups * RPW), b);
  fill_patch<LPR>(D, a.ev, t, a.coef, b, tid, threads);
  if (tid < 2) failed[tid] = 0;
  const unsigned s0 = smem_u32(sm);
  const int own = t.ng * RPW;
  for (int i = tid; i < (own + t.halo) * LPR; i += threads) {
    const int s = i / LPR;   // mu_k of every slot, mu_{k+1} of the own ones
    const int r = s < own ? __ldg(D.row + t.g0 * RPW + s) : __ldg(D.halo + t.h0 + s - own);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u = v;
    if (r >= 0) {
      const size_t o = (size_t)r * a.ld + a.col0;
      v = __ldg(reinterpret_cast<const float4*>(a.mu + o) + i % LPR);
      if (s < own) u = __ldg(reinterpret_cast<const float4*>(a.mu1 + o) + i % LPR);
    }
    sts4(s0 + i * 16, v);
    sts4(s0 + buf + i * 16, u);
  }
  for (int i = tid; i < own; i += threads) {
    const int r = __ldg(D.row + t.g0 * RPW + i);
    sums[i] = r < 0 ? make_float4(0.f, 0.f, 0.f, 0.f)
                    : make_float4(a.G[r], a.Gc[r], a.H[r], a.Hc[r]);
  }
  __syncthreads();

  const int bw = border_warps_of(t.gb, t.ng, threads >> 5);
  const bool border = warp < bw;
  const int w = border ? warp : warp - bw, nw = border ? bw : (threads >> 5) - bw;
  const int g_first = (border ? 0 : t.gb) + w, g_end = border ? t.gb : t.ng;
  const size_t xhalf = (size_t)D.n_x * (2 * LPR);
  unsigned mine = s0 + lane * 16, st = s0 + lane % LPR * 16,
           pair0 = smem_u32(t.pair + lane / LPR), coef0 = smem_u32(t.coef + lane / LPR),
           row0 = smem_u32(t.row + lane / LPR), hdr0 = smem_u32(t.hdr),
           sum0 = smem_u32(sums + lane / LPR);
  int c0 = a.col0 + lane % LPR * 4;
  asm volatile("" : "+r"(mine), "+r"(st), "+r"(pair0), "+r"(coef0), "+r"(row0), "+r"(hdr0),
               "+r"(c0), "+r"(sum0));
  uint4* const xmine = a.xbuf + ((size_t)t.x0 * LPR + lane) * 2;   // border group g: + 64 g
  auto state_of = [&](int g, int j) -> float4 {   // p_k of the lane in group g, reverse step j
    const int r = lds1(row0 + g * (RPW * 4));
    return r < 0 ? make_float4(0.f, 0.f, 0.f, 0.f)
                 : __ldg(reinterpret_cast<const float4*>(a.pk - (ptrdiff_t)j * a.state +
                                                         (ptrdiff_t)r * a.ld + c0));
  };
  float4 next = make_float4(0.f, 0.f, 0.f, 0.f);
  if (g_first < g_end) next = state_of(g_first, 0);
  for (int j = 0; j < a.steps; ++j) {
    const unsigned in = (j & 1) * buf, out = ((j & 1) ^ 1) * buf;
    uint4* xo = xmine + (size_t)((j & 1) ^ 1) * xhalf;
    if (border && j > 0) {
      if (!fetch_halo<LPR>(a.xbuf + (size_t)(j & 1) * xhalf, smem_u32(t.halo_x),
                           s0 + in + own * SLOT, t.halo * 2 * LPR, (unsigned)j, tid, nw * 32,
                           a.status, a.budget))
        failed[j & 1] = 1;
      bar_sync(kBarBorder, nw * 32);
    }
#pragma unroll 1
    for (int g = g_first; g < g_end; g += nw) {
      const float4 pk = next;
      if (g + nw < g_end)
        next = state_of(g + nw, j);
      else if (j + 1 < a.steps)
        next = state_of(g_first, j + 1);
      const int h = lds1(hdr0 + g * 4);
      const float4 c = lds4(coef0 + g * (RPW * 16));
      const float4 self = lds4(mine + in + g * 512), old = lds4(mine + out + g * 512);
      const float4 acc =
          U ? row_product3<RPW>(st + in, pair0 + g * (3 * RPW * 16), c.w, self)
            : row_product<RPW>(st + in, pair0 + (h & ((1 << kPairShift) - 1)) * 16,
                               (h >> kPairShift) & kPairMask, c.w, self);
      float4 o = leap(c, self, old, acc);
      if (h < 0) {   // trace weights at the row's receivers
        const int r = lds1(row0 + g * (RPW * 4));
        if (r >= 0)
          for (int q = __ldg(a.ev.rec_ptr + r); q < __ldg(a.ev.rec_ptr + r + 1); ++q) {
            const int d = __ldg(a.ev.rec_shot + q) - c0;
            if (d >= 0 && d < 4)
              add_comp(o, d, __ldg(a.coef + r).w *
                                 __ldg(a.w + (size_t)__ldg(a.ev.rec_trace + q) * a.nt +
                                       (a.k - j - 1)));
          }
      }
      if (border) xstore(xo + g * 64, o, (unsigned)(j + 1));
      sts4(mine + out + g * 512, o);
      float t1 = 0.0f, t2 = 0.0f;
      adj_terms(pk, o, self, old, t1, t2);
#pragma unroll
      for (int off = LPR / 2; off > 0; off >>= 1) {
        t1 += __shfl_xor_sync(0xffffffffu, t1, off);
        t2 += __shfl_xor_sync(0xffffffffu, t2, off);
      }
      if (lane % LPR == 0) {
        float4 q = lds4(sum0 + g * (RPW * 16));
        kahan_add(&q.x, &q.y, t1);
        kahan_add(&q.z, &q.w, t2);
        sts4(sum0 + g * (RPW * 16), q);
      }
    }
    __syncthreads();
    if (failed[j & 1]) return;
  }
  const unsigned in = (a.steps & 1) * buf, out = ((a.steps & 1) ^ 1) * buf;
  for (int g = g_first; g < g_end; g += nw) {
    const int r = lds1(row0 + g * (RPW * 4));
    if (r < 0) continue;
    const size_t o = (size_t)r * a.ld + c0;
    *reinterpret_cast<float4*>(a.mu + o) = lds4(mine + in + g * 512);
    *reinterpret_cast<float4*>(a.mu1 + o) = lds4(mine + out + g * 512);
    if (lane % LPR == 0) {
      const float4 q = lds4(sum0 + g * (RPW * 16));
      a.G[r] = q.x;
      a.Gc[r] = q.y;
      a.H[r] = q.z;
      a.Hc[r] = q.w;
    }
  }
}

template <int LPR>
int launch_adj(const ResidentAdjArgs& a, const ResidentShape& s, cudaStream_t st) {
  return a.P.uniform == 3 ? launch_resident(k_resident_adjoint<LPR, true>, a, s, st)
                          : launch_resident(k_resident_adjoint<LPR, false>, a, s, st);
}

}  // namespace
}  // namespace mg
