// Device parts shared by the resident kernels.  A CTA holds one patch of the
// mesh (resident.h) for 4 LPR columns (shots), for many leapfrog steps: two
// states of its own rows and the halo rows of the current one in shared memory
// (slot-major, LPR float4 per slot; a step writes p_{l+1} over p_{l-1}), the
// patch's stiffness and coefficients beside them.  Only the border rows travel:
// their new values go to a global exchange buffer, every value beside the
// number of its step, and the patches that need them poll the values themselves
// (no flag, no fence): the border warps, while the inner warps compute.
#pragma once

#include <cuda_runtime.h>

#include "../../include/mgwave.h"
#include "device_util.cuh"
#include "resident.h"

namespace mg {
namespace {

using namespace dev;

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ float4 lds4(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}
__device__ __forceinline__ int2 lds2(unsigned a) {
  int2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds1(unsigned a) {
  int v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(unsigned a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void sts2(unsigned a, unsigned x, unsigned y) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
constexpr int kBarBorder = 1;   // the border warps (barrier 0: all)

// Exchange of border rows: an element is 8 bytes {value, step}, written and
// read whole (64-bit relaxed accesses), so a reader that finds its step's
// number has its value.  Two halves by step parity: a patch writes step k's
// half only after it has read every neighbour's step k - 1, which each of
// them computed after reading step k - 2 from that half.
__device__ __forceinline__ unsigned long long xelem(float v, unsigned tag) {
  return (unsigned long long)tag << 32 | __float_as_uint(v);
}
__device__ __forceinline__ void xstore(uint4* p, float4 v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(xelem(v.x, tag)),
               "l"(xelem(v.y, tag))
               : "memory");
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p + 1),
               "l"(xelem(v.z, tag)), "l"(xelem(v.w, tag))
               : "memory");
}
__device__ __forceinline__ void xload(const uint4* p, unsigned long long& a,
                                      unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
}

// True while a wait may go on; past `budget` clock cycles or after another
// CTA's failure it sets *status.
__device__ __forceinline__ bool keep_waiting(long long& t0, int* status, long long budget) {
  const long long now = clock64();
  if (t0 == 0) t0 = now;
  if (now - t0 <= budget && *reinterpret_cast<volatile int*>(status) == 0) return true;
  atomicExch(status, 1);
  return false;
}

// Copies the `units` 16-byte exchange units (two elements each, 2 LPR per halo
// row) of step `tag` into the halo slots, thread t of n taking every n-th, up
// to kFetch of them in flight, and polls until they carry the tag; false when
// the wait ran out.
constexpr int kFetch = 4;
template <int LPR>
__device__ __forceinline__ bool fetch_halo(const uint4* x, unsigned halo_x, unsigned dst,
                                           int units, unsigned tag, int t, int n, int* status,
                                           long long budget) {
  long long t0 = 0;
  for (int u0 = t; u0 < units; u0 += kFetch * n) {
    int at[kFetch];
    unsigned long long a[kFetch], b[kFetch];
#pragma unroll
    for (int i = 0; i < kFetch; ++i) {   // past the end: the last unit again
      const int u = min(u0 + i * n, units - 1);
      at[i] = lds1(halo_x + u / (2 * LPR) * 4) * (2 * LPR) + u % (2 * LPR);
    }
    for (;;) {
      bool ok = true;
#pragma unroll
      for (int i = 0; i < kFetch; ++i) xload(x + at[i], a[i], b[i]);
#pragma unroll
      for (int i = 0; i < kFetch; ++i)
        ok = ok && (unsigned)(a[i] >> 32) == tag && (unsigned)(b[i] >> 32) == tag;
      if (ok) break;
      if (!keep_waiting(t0, status, budget)) return false;
    }
#pragma unroll
    for (int i = 0; i < kFetch; ++i)
      sts2(dst + min(u0 + i * n, units - 1) * 8, (unsigned)a[i], (unsigned)b[i]);
  }
  return true;
}

// The patch's tables in shared memory: entry pairs {offset, K, offset, K}
// (offsets in bytes within a state; the rows of a group side by side, so that
// one warp's load of a pair is one contiguous run), coefficients {alpha, beta,
// gamma, K_ii} and row per own slot, exchange rows of the halo, group headers.
struct Patch {
  float4* pair;
  float4* coef;
  int* row;
  int* halo_x;
  int* hdr;
  int gb, ng, halo;          // border groups, groups, halo rows
  int g0, h0, x0;            // first group, halo row and exchange row
};

template <int RPW>
__device__ __forceinline__ Patch patch_tables(const DevPatches& D, unsigned char* at, int b) {
  Patch t;
  t.pair = reinterpret_cast<float4*>(at);
  t.coef = t.pair + D.max_pairs;
  t.row = reinterpret_cast<int*>(t.coef + D.max_groups * RPW);
  t.halo_x = t.row + D.max_groups * RPW;
  t.hdr = t.halo_x + D.max_halo;
  t.g0 = __ldg(D.grp_off + b);
  t.ng = __ldg(D.grp_off + b + 1) - t.g0;
  t.gb = __ldg(D.border + b);
  t.h0 = __ldg(D.halo_off + b);
  t.halo = __ldg(D.halo_off + b + 1) - t.h0;
  t.x0 = __ldg(D.x_off + b);
  return t;
}

// Warps of a CTA's `warps` that take its gb border groups (of ng): one each
// when all groups get a warp; else their share of the warps, and 1.6 times it
// when the border is less than a third of the patch: the border's way (copy,
// compute, store, the neighbour's copy) is then the longer one.  Measured, us
// per step with 1, 1.3, 1.6, 2 times the share: 104 groups (20% border) 14.7,
// 14.6, 13.9, 14.3; 53 groups (40%) 2.67, 2.85, 2.92, 2.94; 50 groups of a
// tetrahedral patch (70%) 5.3, 7.4, 9.4, 9.4.  Around a third, forward and tangent
// of 64 shots with once and 1.6 times the share: 42% border 2.3, 4.2 and 2.2,
// 8.3; 37% 2.4, 4.8 and 2.6, 5.3; 34% 2.7, 5.7 and 2.7, 6.4; 31% 3.2, 7.2 and
// 2.9, 6.8; 22% (32 shots) 3.2, 7.2 and 2.9, 6.7.
__device__ __forceinline__ int border_warps_of(int gb, int ng, int warps) {
  if (ng <= warps) return max(gb, 1);
  const int share = gb * warps / ng;
  return min(min(gb, warps - 1), max(1, 3 * gb < ng ? share * 8 / 5 + 1 : share + 1));
}

template <int LPR>
__device__ __forceinline__ void fill_patch(const DevPatches& D, const DevEvents& ev,
                                           const Patch& t, const float4* __restrict__ coef, int b,
                                           int tid, int threads) {
  constexpr int RPW = 32 / LPR, SLOT = 16 * LPR;
  const int p0 = __ldg(D.pair_off + b), np = __ldg(D.pair_off + b + 1) - p0;
  const int s0 = t.g0 * RPW;
  for (int i = tid; i < np; i += threads) {
    const int4 q = __ldg(D.pair + p0 + i);   // {slot, slot, K, K}
    t.pair[i] = make_float4(__int_as_float(q.x * SLOT), __int_as_float(q.z),
                            __int_as_float(q.y * SLOT), __int_as_float(q.w));
  }
  for (int i = tid; i < t.halo; i += threads) t.halo_x[i] = __ldg(D.halo_x + t.h0 + i);
  for (int i = tid; i < t.ng * RPW; i += threads) {
    const int r = __ldg(D.row + s0 + i);
    t.row[i] = r;
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r >= 0) {
      c = __ldg(coef + r);
      c.w = __ldg(D.diag + s0 + i);
    }
    t.coef[i] = c;
  }
  for (int g = tid; g < t.ng; g += threads) {
    int h = __ldg(D.hdr + t.g0 + g);
    for (int i = 0; i < RPW; ++i) {
      const int r = __ldg(D.row + s0 + g * RPW + i);
      if (r >= 0 && (__ldg(ev.src_ptr + r) != __ldg(ev.src_ptr + r + 1) ||
                     __ldg(ev.rec_ptr + r) != __ldg(ev.rec_ptr + r + 1)))
        h |= kEventBit;
    }
    t.hdr[g] = h;
  }
}

// acc = K_ii self + the off-diagonal entries in the row's order (the FMAs of
// the row kernels); `st` is the lane's address of slot 0, q its row's first
// pair.
template <int RPW>
__device__ __forceinline__ float4 row_product3(unsigned st, unsigned q, float kd, float4 self) {
  const float4 e = lds4(q), f = lds4(q + RPW * 16), g = lds4(q + 2 * RPW * 16);
  const float4 x0 = lds4(st + __float_as_uint(e.x)), x1 = lds4(st + __float_as_uint(e.z));
  const float4 x2 = lds4(st + __float_as_uint(f.x)), x3 = lds4(st + __float_as_uint(f.z));
  const float4 x4 = lds4(st + __float_as_uint(g.x)), x5 = lds4(st + __float_as_uint(g.z));
  float4 acc = scale4(kd, self);
  acc = fma4(e.y, x0, acc);
  acc = fma4(e.w, x1, acc);
  acc = fma4(f.y, x2, acc);
  acc = fma4(f.w, x3, acc);
  acc = fma4(g.y, x4, acc);
  return fma4(g.w, x5, acc);
}
template <int RPW>
__device__ __forceinline__ float4 row_product(unsigned st, unsigned q, int pairs, float kd,
                                              float4 self) {
  float4 acc = scale4(kd, self);
#pragma unroll 2
  for (int k = 0; k < pairs; ++k) {
    const float4 e = lds4(q + k * RPW * 16);
    const float4 x = lds4(st + __float_as_uint(e.x));
    const float4 y = lds4(st + __float_as_uint(e.z));
    acc = fma4(e.y, x, acc);
    acc = fma4(e.w, y, acc);
  }
  return acc;
}

// Sources of row r (-1: none) at step l; c0: the lane's first shot column.
__device__ __forceinline__ void resident_source(const ResidentArgs& a, int r, int c0, int l,
                                                float gamma, float4& o) {
  if (r < 0) return;
  const int q0 = __ldg(a.ev.src_ptr + r), q1 = __ldg(a.ev.src_ptr + r + 1);
  if (q0 == q1) return;
  const float sv = gamma * __ldg(a.wavelet + l);
  for (int q = q0; q < q1; ++q) {
    const int d = __ldg(a.ev.src_shot + q) - c0;
    if (d >= 0 && d < 4) add_comp(o, d, sv);
  }
}
// Receivers of row r: sample l of their traces.
__device__ __forceinline__ void resident_record(const ResidentArgs& a, float* traces, int r,
                                                int c0, int l, const float4& o) {
  if (r < 0 || !traces) return;
  for (int q = __ldg(a.ev.rec_ptr + r); q < __ldg(a.ev.rec_ptr + r + 1); ++q) {
    const int d = __ldg(a.ev.rec_shot + q) - c0;
    if (d >= 0 && d < 4) traces[(size_t)__ldg(a.ev.rec_trace + q) * a.nt + l] = get_comp(o, d);
  }
}
// What tangent_fix subtracts.
__device__ __forceinline__ float4 tangent_term(float4 pn, float4 ps, float4 pold, float2 tc) {
  return make_float4(
      __fmaf_rn(tc.x, d2t(pn.x, ps.x, pold.x), __fmul_rn(tc.y, d1t(pn.x, pold.x))),
      __fmaf_rn(tc.x, d2t(pn.y, ps.y, pold.y), __fmul_rn(tc.y, d1t(pn.y, pold.y))),
      __fmaf_rn(tc.x, d2t(pn.z, ps.z, pold.z), __fmul_rn(tc.y, d1t(pn.z, pold.z))),
      __fmaf_rn(tc.x, d2t(pn.w, ps.w, pold.w), __fmul_rn(tc.y, d1t(pn.w, pold.w))));
}

// Cooperative launch (patches wait for one another: all resident), the
// exchange buffer's step numbers cleared first.  MG_ERR_UNSUPPORTED when the
// device cannot hold it.
template <class A>
int launch_resident(void (*kern)(A), const A& a, const ResidentShape& s, cudaStream_t st) {
  const int rc = resident_smem_limit(reinterpret_cast<const void*>(kern), s.smem);
  if (rc != MG_OK) return rc;
  if (a.P.n_x && cudaMemsetAsync(a.xbuf, 0, (size_t)2 * a.P.n_x * s.lpr * 2 * sizeof(uint4),
                                 st) != cudaSuccess)
    return MG_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.P.B);
  cfg.blockDim = dim3(32 * s.warps);
  cfg.dynamicSmemBytes = s.smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a);
  if (e == cudaSuccess) return MG_OK;
  cudaGetLastError();
  return e == cudaErrorCooperativeLaunchTooLarge ? MG_ERR_UNSUPPORTED : MG_ERR_CUDA;
}

}  // namespace
}  // namespace mg
