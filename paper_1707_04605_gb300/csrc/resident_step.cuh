#pragma once

// Resident forward kernel and forward + tangent kernel: one cooperative launch
// advances a group of shots by many leapfrog steps with the states on chip
// (resident_common.cuh).
//
// TAN: p and dp of 2 LPR shots share the rows, the first half of a row's lanes
// holding p and the second dp: both are columns of the same product, and the
// lanes of dp take the correction of tangent_fix from their partner by
// shuffles (four values).
//
// Bound by shared memory bandwidth: a float4 of a row takes 41 reads and writes
// of 16 bytes per 4 columns (6 neighbours, self, p_{l-1}, result, entries,
// coefficients), 75% of the L1 data pipe's peak measured on 413-row patches.
// Against one launch per step: 62,641 nodes, 128 shots 28.1 -> 13.9 us per step
// (19.2 with the best row shape); 15,769 nodes, 37 shots 6.4 -> 2.7; 4,225
// nodes, 1 shot 3.8 -> 1.3; 30,525 nodes of tetrahedra, 24 shots 10.8 -> 5.3.
// Tried and slower: states in registers (unrolled over the groups: bound by
// instruction fetch), four rows per thread sharing their neighbours (15 reads
// for four rows instead of 28, but twice the FMAs and a longer chain for the
// border), flags and fences instead of tagged values (two more round trips).
//
// A warp is of one class for the whole launch.  Per step the inner warps
// advance the inner groups at once; the border warps first copy the halo rows
// of p_l from the exchange buffer, then advance the border groups and store
// their p_{l+1} there.  All warps meet once per step.
#include "resident_common.cuh"

namespace mg {
namespace {

// U: pairs of every row are 3 (straight code), else as the group headers say.
// HIST: every state p goes to the history.
template <int LPR, bool U, bool HIST, bool TAN>
__global__ void __launch_bounds__(kResidentThreads, 1) k_resident_step(ResidentArgs a) {
  constexpr int RPW = 32 / LPR, SLOT = 16 * LPR;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int failed[2];   // by step parity: no warp can be two steps ahead of another
  const int b = blockIdx.x, tid = threadIdx.x, threads = blockDim.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const DevPatches& D = a.P;
  const unsigned buf = (unsigned)D.max_slots * SLOT;
  float2* const tc = reinterpret_cast<float2*>(sm + 2 * (size_t)buf);   // TAN, per own slot
  const Patch t = patch_tables<RPW>(
      D, sm + 2 * (size_t)buf + (TAN ? (D.max_groups * RPW + 1) / 2 * 16 : 0), b);
  fill_patch<LPR>(D, a.ev, t, a.coef, b, tid, threads);
  if (tid < 2) failed[tid] = 0;
  if (TAN)
    for (int i = tid; i < t.ng * RPW; i += threads) {
      const int r = __ldg(D.row + t.g0 * RPW + i);
      tc[i] = r < 0 ? make_float2(0.f, 0.f) : __ldg(a.tcoef + r);
    }
  const unsigned s0 = smem_u32(sm);
  const int own = t.ng * RPW;
  for (int i = tid; i < (own + t.halo) * LPR; i += threads) {
    const int s = i / LPR;   // p_l of every slot, p_{l-1} of the own ones
    const int r = s < own ? __ldg(D.row + t.g0 * RPW + s) : __ldg(D.halo + t.h0 + s - own);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u = v;
    if (!TAN && a.p && r >= 0) {   // the tangent starts at rest
      const size_t o = (size_t)r * a.ld + a.col0;
      v = __ldg(reinterpret_cast<const float4*>(a.p + o) + i % LPR);
      if (s < own) u = __ldg(reinterpret_cast<const float4*>(a.pm + o) + i % LPR);
    }
    sts4(s0 + i * 16, v);
    sts4(s0 + buf + i * 16, u);
  }
  __syncthreads();

  const int bw = border_warps_of(t.gb, t.ng, threads >> 5);
  const bool border = warp < bw;
  const int w = border ? warp : warp - bw, nw = border ? bw : (threads >> 5) - bw;
  const int g_first = (border ? 0 : t.gb) + w, g_end = border ? t.gb : t.ng;
  const size_t xhalf = (size_t)D.n_x * (2 * LPR);
  // per-lane addresses, opaque: kept, not derived anew from the thread index at
  // every use
  unsigned mine = s0 + lane * 16, st = s0 + lane % LPR * 16,
           pair0 = smem_u32(t.pair + lane / LPR), coef0 = smem_u32(t.coef + lane / LPR),
           row0 = smem_u32(t.row + lane / LPR), hdr0 = smem_u32(t.hdr);
  constexpr int COLS = TAN ? LPR / 2 : LPR;   // lanes of a row with different shots
  const bool is_q = TAN && lane % LPR >= COLS;
  int c0 = a.col0 + lane % COLS * 4;
  unsigned tc0 = smem_u32(tc + lane / LPR);
  asm volatile("" : "+r"(mine), "+r"(st), "+r"(pair0), "+r"(coef0), "+r"(row0), "+r"(hdr0),
               "+r"(c0), "+r"(tc0));
  float* const traces = is_q ? a.dtraces : a.traces;
  uint4* const xmine = a.xbuf + ((size_t)t.x0 * LPR + lane) * 2;   // border group g: + 64 g
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
      const int h = lds1(hdr0 + g * 4);
      const float4 c = lds4(coef0 + g * (RPW * 16));
      const float4 self = lds4(mine + in + g * 512), old = lds4(mine + out + g * 512);
      const float4 acc =
          U ? row_product3<RPW>(st + in, pair0 + g * (3 * RPW * 16), c.w, self)
            : row_product<RPW>(st + in, pair0 + (h & ((1 << kPairShift) - 1)) * 16,
                               (h >> kPairShift) & kPairMask, c.w, self);
      float4 o = leap(c, self, old, acc);
      if (h < 0) resident_source(a, is_q ? -1 : lds1(row0 + g * (RPW * 4)), c0, a.step0 + j, c.z, o);
      if (TAN) {   // dp -= cm (p+ - 2 p + p-) + cd (p+ - p-)
        const int2 v = lds2(tc0 + g * (RPW * 8));
        const float4 f = tangent_term(o, self, old, make_float2(__int_as_float(v.x),
                                                                __int_as_float(v.y)));
        const float4 e = make_float4(__shfl_xor_sync(0xffffffffu, f.x, COLS),
                                     __shfl_xor_sync(0xffffffffu, f.y, COLS),
                                     __shfl_xor_sync(0xffffffffu, f.z, COLS),
                                     __shfl_xor_sync(0xffffffffu, f.w, COLS));
        if (is_q)
          o = make_float4(__fsub_rn(o.x, e.x), __fsub_rn(o.y, e.y), __fsub_rn(o.z, e.z),
                          __fsub_rn(o.w, e.w));
      }
      if (h < 0) resident_record(a, traces, lds1(row0 + g * (RPW * 4)), c0, a.step0 + j, o);
      if (border) xstore(xo + g * 64, o, (unsigned)(j + 1));
      sts4(mine + out + g * 512, o);
      if (HIST) {
        const int r = lds1(row0 + g * (RPW * 4));
        if (r >= 0 && !is_q)
          *reinterpret_cast<float4*>(a.hist + (size_t)j * a.state + (size_t)r * a.ld + c0) = o;
      }
    }
    __syncthreads();
    if (failed[j & 1]) return;
  }
  if (!TAN && a.out_p) {
    const unsigned in = (a.steps & 1) * buf, out = ((a.steps & 1) ^ 1) * buf;
    for (int g = g_first; g < g_end; g += nw) {
      const int r = lds1(row0 + g * (RPW * 4));
      if (r < 0) continue;
      const size_t o = (size_t)r * a.ld + c0;
      *reinterpret_cast<float4*>(a.out_p + o) = lds4(mine + in + g * 512);
      *reinterpret_cast<float4*>(a.out_pm + o) = lds4(mine + out + g * 512);
    }
  }
}

template <int LPR, bool U, bool HIST, bool TAN>
int launch_one(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st) {
  return launch_resident(k_resident_step<LPR, U, HIST, TAN>, a, s, st);
}

template <int LPR, bool TAN>
int launch_lpr(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st) {
  if (a.P.uniform == 3)
    return a.hist ? launch_one<LPR, true, true, TAN>(a, s, st)
                  : launch_one<LPR, true, false, TAN>(a, s, st);
  return a.hist ? launch_one<LPR, false, true, TAN>(a, s, st)
                : launch_one<LPR, false, false, TAN>(a, s, st);
}

}  // namespace
}  // namespace mg
