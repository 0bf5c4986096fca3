// The paper's first-order leapfrog with element flux variables and the
// split-field perfectly matched layer (App. A, Eqs. (system1), (system2),
// (leap-frog1), (leap-frog2)).
//
//   q^(k)_{l+1/2} = (1 - dt zeta^(k)) q^(k)_{l-1/2} + dt sum_a dphi_a/dx_k p_l[a]   (per cell)
//   p_{l+1}       = p_l + dt/C (f_l - (R + S) p_l - sum_k B^(k)T q^(k)_{l+1/2})      (per node)
//
// A_ii = |T_i|, B^(k)_{ij} = |T_i| dphi_j/dx_k, C the lumped eps-mass, R the
// lumped sigma-mass (the handle's conductivity), S the lumped xi-mass, and
// f_l = dt sum_{m <= l} s_m (the source is the time integral of the
// wavelet).  Natural outer boundary: the layer absorbs.  State: p [n][ld],
// q [d][m][ld] FP32 (ld = padded shot count); a thread advances one float4
// of shots of one node or one cell.  Sample l of a trace is p_{l+1}.
//
// Jacobians with respect to the cell permittivity (only C depends on it):
//  * tangent, in lockstep with the forward: the fluxes of dp follow the
//    same update; dp_{l+1} = dp_l + dt/C (-(R+S) dp_l - sum_k B^(k)T dq^(k))
//    - (dC/C)(p_{l+1} - p_l), dC the lumped mass of the direction;
//  * adjoint, backwards over checkpointed segments (p and q stored every
//    ckpt_every steps, each segment's p states recomputed into a buffer):
//    with a the adjoint of p_{l+1} (traces' weights at the receivers plus
//    what step l+1 sends back) and r = a dt / C, the scaled flux adjoint
//    Qt^(k) = Q^(k)/|e| becomes (1 - dt zeta_k) Qt^(k) - sum_a dphi_a/dx_k r[v_a],
//    p_l receives a - (R+S) r + dt sum_k B^(k)T Qt^(k), and the C-sensitivity
//    gathers -sum_l a (p_{l+1} - p_l) / C; the cell gradient is
//    |e|/(d+1) times its sum over the cell's vertices, restricted to a level.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/mgwave.h"
#include "flux_common.cuh"
#include "kernels.cuh"
#include "mesh_view.h"
#include "mg_internal.h"

namespace mg {
namespace {

constexpr int kMaxDim = 3;

// Step kernels run as programmatic dependents of the previous kernel on
// the stream: each waits for it to complete (and its stores to be visible)
// before touching any state, then lets the next launch be scheduled.
__device__ __forceinline__ void pdl_sync() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Step index of a launch: l, plus the device int *base when the launch is
// a node of a CUDA graph replayed once per chunk of steps (the graph moves
// the base at its end).  Read after pdl_sync.
struct StepRef {
  int l;
  const int* base;
};
__device__ __forceinline__ int step_of(const StepRef& s) { return s.base ? s.l + *s.base : s.l; }

// p states kept in slots of one buffer: p_l in slot l mod K (stride ns4
// float4), so that a launch finds its states from its step index alone;
// seg == nullptr: the launch's own state pointers.
struct Slots {
  float4* seg;
  int64_t ns4;
  int K;
};
__device__ __forceinline__ float4* slot_of(const Slots& s, int l) {
  return s.seg + (int64_t)(l % s.K) * s.ns4;
}

// per node: {dt / C_i, R_i + S_i}
__global__ void k_flux_coefs(CoefArgs c, const double* __restrict__ xi, double dt,
                             float2* __restrict__ out) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= c.n) return;
  double C = 0.0, RS = 0.0;
  for (int64_t q = c.nc_ptr[r]; q < c.nc_ptr[r + 1]; ++q) {
    const int e = c.nc_cell[q];
    C += c.eps[e] * c.nc_w[q];
    if (c.sigma) RS += c.sigma[e] * c.nc_w[q];
    if (xi) RS += xi[e] * c.nc_w[q];
  }
  out[r] = make_float2((float)(dt / C), (float)RS);
}

// Damping factors 1 - dt zeta of the cells; *bad is set when a value is
// negative or not finite.
__global__ void k_flux_keep(int64_t count, const double* __restrict__ zeta, float dt,
                            float* __restrict__ keep, int* bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const double z = zeta ? zeta[i] : 0.0;
  if (!(z >= 0.0) || !isfinite(z)) *bad = 1;
  keep[i] = 1.0f - dt * (float)z;
}

// An incidence: {cell, |e| dphi_i/dx_k}, one 16-byte load.
template <int D>
struct Cell {
  int v[D + 1];
  float g[D + 1][D];
};
template <int D>
__device__ __forceinline__ Cell<D> load_cell(const float4* __restrict__ cell, int64_t e) {
  float w[4 * kCellW<D>];
#pragma unroll
  for (int i = 0; i < kCellW<D>; ++i) {
    const float4 x = __ldg(cell + e * kCellW<D> + i);
    w[4 * i] = x.x;
    w[4 * i + 1] = x.y;
    w[4 * i + 2] = x.z;
    w[4 * i + 3] = x.w;
  }
  Cell<D> c;
#pragma unroll
  for (int a = 0; a <= D; ++a) {
    c.v[a] = __float_as_int(w[a]);
#pragma unroll
    for (int k = 0; k < D; ++k) c.g[a][k] = w[D + 1 + a * D + k];
  }
  return c;
}

// One thread per float4 of shots (threadIdx.x) of one cell or node
// (threadIdx.y): see item_block.
struct Item {
  int64_t i;
  int c4;
  bool ok;
};
__device__ __forceinline__ Item item_of(int64_t count, int ld4) {
  Item t;
  t.i = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
  t.c4 = blockIdx.y * blockDim.x + threadIdx.x;
  t.ok = t.i < count && t.c4 < ld4;
  return t;
}

// q^(k) <- keep_k q^(k) + dt sum_a grad[a][k] p[v_a]; SIGN < 0, dt = 1: the
// adjoint's Qt^(k) <- keep_k Qt^(k) - sum_a grad[a][k] r[v_a].
//
// Bound by the states' traffic through L2: a step gathers and writes 900 MB at
// 62,641 nodes, 124,416 cells and 128 shots in its two kernels.  Against one
// load per constant and 64-bit divisions, us per step: tangent 183 -> 169,
// reverse 133 -> 131; tetrahedra (30,525 nodes, 32 shots) forward 51 -> 44,
// tangent 132 -> 116, with reverse 117 -> 102; 249,697 nodes, 64 shots forward
// 186 -> 184, tangent 375 -> 342.  Advancing 32 shots at a time gains 10% on the
// forward, 16 at a time loses 40%: left out.
template <int D, int SIGN>
__global__ void __launch_bounds__(256) k_flux_q(int64_t m, int ld4,
                                                const float4* __restrict__ cell,
                                                const float* __restrict__ keep,
                                                const float4* __restrict__ p,
                                                float4* __restrict__ q, float dt, StepRef sr,
                                                Slots sl) {
  const Item t = item_of(m, ld4);
  if (!t.ok) return;
  const Cell<D> c = load_cell<D>(cell, t.i);
  float kp[D];
#pragma unroll
  for (int k = 0; k < D; ++k) kp[k] = __ldg(keep + t.i * D + k);
  // the constants are complete before the call's first step
  pdl_sync();
  if (sl.seg) p = slot_of(sl, step_of(sr));
  float4 pv[D + 1], o[D];
#pragma unroll
  for (int k = 0; k < D; ++k) o[k] = q[((int64_t)k * m + t.i) * ld4 + t.c4];
#pragma unroll
  for (int a = 0; a <= D; ++a) pv[a] = __ldg(p + (int64_t)c.v[a] * ld4 + t.c4);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a <= D; ++a) acc = fma4f(c.g[a][k], pv[a], acc);
    float4* qp = q + ((int64_t)k * m + t.i) * ld4 + t.c4;
    *qp = SIGN > 0 ? make_float4(fmaf(kp[k], o[k].x, dt * acc.x), fmaf(kp[k], o[k].y, dt * acc.y),
                                 fmaf(kp[k], o[k].z, dt * acc.z), fmaf(kp[k], o[k].w, dt * acc.w))
                   : make_float4(fmaf(kp[k], o[k].x, -acc.x), fmaf(kp[k], o[k].y, -acc.y),
                                 fmaf(kp[k], o[k].z, -acc.z), fmaf(kp[k], o[k].w, -acc.w));
  }
}

// bt_n += sum_{e ni i} sum_k w[e,i,k] q_n^(k)_e for NQ flux fields, in the order
// of the incidences.  One incidence at a time, and the row's own values are
// loaded after it: what is in flight across the loop costs more warps than it
// gains (62,641 nodes, 128 shots, 256 forward steps with one, two, three and
// four incidences in flight 25.0, 28.6, 29.1, 32.8 ms; with the row's values
// loaded ahead the tangent 200 us per step instead of 169, tetrahedra forward 59
// instead of 44).
template <int D, int NQ>
__device__ __forceinline__ void gather_flux(int s0, int s1, const int4* __restrict__ inc,
                                            int64_t m, int ld4, int c4,
                                            const float4* const (&q)[NQ], float4 (&bt)[NQ]) {
#pragma unroll 1
  for (int s = s0; s < s1; ++s) {
    const int4 w = __ldg(inc + s);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const float wk = __int_as_float(k == 0 ? w.y : k == 1 ? w.z : w.w);
#pragma unroll
      for (int n = 0; n < NQ; ++n)
        bt[n] = fma4f(wk, __ldg(q[n] + ((int64_t)k * m + w.x) * ld4 + c4), bt[n]);
    }
  }
}

// pout <- p + dt/C (f delta_src - (R+S) p - sum_{e ni i} sum_k w[e,i,k] q^(k)_e)
// (pout may be p); sources and traces of the row's shots
template <int D>
__global__ void __launch_bounds__(256) k_flux_p(
    int64_t n, int64_t m, int ld4, const int32_t* __restrict__ inc_ptr,
    const int4* __restrict__ inc, const float2* __restrict__ coef, const float4* __restrict__ q,
    const float4* p, float4* pout, DevEvents ev, const float* __restrict__ fl,
    float* __restrict__ traces, int nt, StepRef sr, Slots sl) {
  pdl_sync();
  const int l = step_of(sr);
  if (sl.seg) {   // p_l in slot l, p_{l+1} into the next slot
    pout = slot_of(sl, l);
    p = pout;
    pout += sl.ns4;
  }
  const Item it = item_of(n, ld4);
  if (!it.ok) return;
  const int64_t i = it.i, t = i * ld4 + it.c4;
  const int c4 = it.c4;
  float4 bt[1] = {make_float4(0.f, 0.f, 0.f, 0.f)};
  const float4* const qs[1] = {q};
  gather_flux<D, 1>(__ldg(inc_ptr + i), __ldg(inc_ptr + i + 1), inc, m, ld4, c4, qs, bt);
  float4 pv = p[t];
  const float2 c = __ldg(coef + i);
  const int s0 = __ldg(ev.src_ptr + i), s1 = __ldg(ev.src_ptr + i + 1);
  const int r0 = __ldg(ev.rec_ptr + i), r1 = __ldg(ev.rec_ptr + i + 1);
  float4 rhs = make_float4(-bt[0].x, -bt[0].y, -bt[0].z, -bt[0].w);
  if (s0 != s1) add_source(ev, s0, s1, c4, __ldg(fl + l), rhs);
  pv.x = fmaf(c.x, fmaf(-c.y, pv.x, rhs.x), pv.x);
  pv.y = fmaf(c.x, fmaf(-c.y, pv.y, rhs.y), pv.y);
  pv.z = fmaf(c.x, fmaf(-c.y, pv.z, rhs.z), pv.z);
  pv.w = fmaf(c.x, fmaf(-c.y, pv.w, rhs.w), pv.w);
  pout[t] = pv;
  if (r0 != r1) record(ev, r0, r1, c4, traces, nt, l, pv);
}

// C_i = sum_{e ni i} x[e] |e| / (d+1) in FP64 (x = eps, or a direction)
__global__ void k_flux_mass(CoefArgs c, const double* __restrict__ x, double* __restrict__ out) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= c.n) return;
  double s = 0.0;
  for (int64_t q = c.nc_ptr[r]; q < c.nc_ptr[r + 1]; ++q) s += x[c.nc_cell[q]] * c.nc_w[q];
  out[r] = s;
}

__global__ void k_flux_ratio(int64_t n, const double* __restrict__ dC, const double* __restrict__ C,
                             float* __restrict__ ratio) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) ratio[r] = (float)(dC[r] / C[r]);
}

// Tangent node update: p as in k_flux_p, and
// dp <- dp + dt/C (-(R+S) dp - sum B^T dq) - ratio (p_new - p_old); traces of dp.
template <int D>
__global__ void __launch_bounds__(256) k_flux_p_tan(
    int64_t n, int64_t m, int ld4, const int32_t* __restrict__ inc_ptr,
    const int4* __restrict__ inc, const float2* __restrict__ coef,
    const float* __restrict__ ratio, const float4* __restrict__ q,
    const float4* __restrict__ dq, float4* __restrict__ p, float4* __restrict__ dp, DevEvents ev,
    const float* __restrict__ fl, float* __restrict__ traces, int nt, StepRef sr) {
  pdl_sync();
  const int l = step_of(sr);
  const Item it = item_of(n, ld4);
  if (!it.ok) return;
  const int64_t i = it.i, t = i * ld4 + it.c4;
  const int c4 = it.c4;
  float4 b2[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  const float4* const qs[2] = {q, dq};
  gather_flux<D, 2>(__ldg(inc_ptr + i), __ldg(inc_ptr + i + 1), inc, m, ld4, c4, qs, b2);
  float4 pv = p[t], dv = dp[t];
  const float2 c = __ldg(coef + i);
  const float rt = __ldg(ratio + i);
  const int s0 = __ldg(ev.src_ptr + i), s1 = __ldg(ev.src_ptr + i + 1);
  const int r0 = __ldg(ev.rec_ptr + i), r1 = __ldg(ev.rec_ptr + i + 1);
  const float4 dbt = b2[1];
  float4 rhs = make_float4(-b2[0].x, -b2[0].y, -b2[0].z, -b2[0].w);
  if (s0 != s1) add_source(ev, s0, s1, c4, __ldg(fl + l), rhs);
  const float4 inc4 = make_float4(fmaf(-c.y, pv.x, rhs.x), fmaf(-c.y, pv.y, rhs.y),
                                  fmaf(-c.y, pv.z, rhs.z), fmaf(-c.y, pv.w, rhs.w));
  dv.x = fmaf(-rt, c.x * inc4.x, fmaf(c.x, fmaf(-c.y, dv.x, -dbt.x), dv.x));
  dv.y = fmaf(-rt, c.x * inc4.y, fmaf(c.x, fmaf(-c.y, dv.y, -dbt.y), dv.y));
  dv.z = fmaf(-rt, c.x * inc4.z, fmaf(c.x, fmaf(-c.y, dv.z, -dbt.z), dv.z));
  dv.w = fmaf(-rt, c.x * inc4.w, fmaf(c.x, fmaf(-c.y, dv.w, -dbt.w), dv.w));
  pv.x = fmaf(c.x, inc4.x, pv.x);
  pv.y = fmaf(c.x, inc4.y, pv.y);
  pv.z = fmaf(c.x, inc4.z, pv.z);
  pv.w = fmaf(c.x, inc4.w, pv.w);
  p[t] = pv;
  dp[t] = dv;
  if (r0 != r1) record(ev, r0, r1, c4, traces, nt, l, dv);
}

// Adjoint node kernel of reverse step l (p_l in slot l mod K of sl, p_{l+1}
// in the next slot).  a = adjoint of p_{l+1}: what step
// l+1 sent back (tp + dt sum_k B^(k)T Qt^(k); zero when l = nt-1) plus the
// weights of the row's receivers at sample l.  Sums a (p_{l+1} - p_l) over
// the node's shots in FP32 (the threads of a node are consecutive lanes:
// the float4s of a node within a warp are summed by a fixed shuffle tree)
// and adds one partial per warp segment of 32 float4 to the FP64 time
// accumulator hacc[i][segment] (GB300's FP64 rate is a small fraction of
// its FP32 rate: one FP64 add per node and step), then stores r = a dt/C
// and tp = a - (R+S) r.
template <int D>
__global__ void __launch_bounds__(256) k_flux_adj_p(
    int64_t n, int64_t m, int ld4, const int32_t* __restrict__ inc_ptr,
    const int4* __restrict__ inc, const float2* __restrict__ coef,
    const float4* __restrict__ Qt, float4* __restrict__ tp, float4* __restrict__ rr, Slots sl,
    double* __restrict__ hacc, DevEvents ev, const float* __restrict__ W, int nt, StepRef sr,
    float dt) {
  pdl_sync();
  const int l = step_of(sr);
  const bool first = l == nt - 1;
  const float4* __restrict__ p0 = slot_of(sl, l);   // p_l; p_{l+1} in the next slot
  const float4* __restrict__ p1 = p0 + sl.ns4;
  const Item it = item_of(n, ld4);
  if (!it.ok) return;
  const int64_t i = it.i, t = i * ld4 + it.c4;
  const int c4 = it.c4;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!first) {
    float4 bt[1] = {a};
    const float4* const qs[1] = {Qt};
    gather_flux<D, 1>(__ldg(inc_ptr + i), __ldg(inc_ptr + i + 1), inc, m, ld4, c4, qs, bt);
    a = fma4f(dt, bt[0], tp[t]);
  }
  const int r0 = __ldg(ev.rec_ptr + i), r1 = __ldg(ev.rec_ptr + i + 1);
  for (int r = r0; r < r1; ++r) {
    const int d = __ldg(ev.rec_shot + r) - 4 * c4;
    if (d < 0 || d > 3) continue;
    const float v = __ldg(W + (int64_t)__ldg(ev.rec_trace + r) * nt + l);
    if (d == 0) a.x += v;
    if (d == 1) a.y += v;
    if (d == 2) a.z += v;
    if (d == 3) a.w += v;
  }
  const float4 x1 = __ldg(p1 + t), x0 = __ldg(p0 + t);
  float h = a.x * (x1.x - x0.x);
  h = fmaf(a.y, x1.y - x0.y, h);
  h = fmaf(a.z, x1.z - x0.z, h);
  h = fmaf(a.w, x1.w - x0.w, h);
  // ld4 is a power of two or a multiple of 32 and blockDim.x is ld4 or a multiple of 32:
  // the gw lanes of a node's segment are consecutive and active together
  const int gw = ld4 < 32 ? ld4 : 32;
  const int lane = (threadIdx.y * blockDim.x + threadIdx.x) & 31;
  const unsigned gmask = gw == 32 ? 0xffffffffu : (((1u << gw) - 1u) << (lane & ~(gw - 1)));
  for (int off = gw / 2; off > 0; off >>= 1) h += __shfl_xor_sync(gmask, h, off);
  if ((c4 & (gw - 1)) == 0) {
    const int nseg = ld4 < 32 ? 1 : ld4 / 32;
    hacc[i * nseg + c4 / 32] += (double)h;
  }
  const float2 c = __ldg(coef + i);
  const float4 r = make_float4(a.x * c.x, a.y * c.x, a.z * c.x, a.w * c.x);
  rr[t] = r;
  tp[t] = make_float4(fmaf(-c.y, r.x, a.x), fmaf(-c.y, r.y, a.y), fmaf(-c.y, r.z, a.z),
                      fmaf(-c.y, r.w, a.w));
}

// gC_i = -sum_seg hacc[i][seg] / C_i (fixed order over the shot segments)
__global__ void k_flux_hsum(int64_t n, int nseg, const double* __restrict__ hacc,
                            const double* __restrict__ C, double* __restrict__ gC) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int j = 0; j < nseg; ++j) s += hacc[i * nseg + j];
  gC[i] = -s / C[i];
}

// g_e = |e| / (d+1) sum_a gC[v_a]
__global__ void k_flux_cell_grad(int64_t m, int k1, const int32_t* __restrict__ cells,
                                 const double* __restrict__ vol, const double* __restrict__ gC,
                                 double* __restrict__ g) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  double s = 0.0;
  for (int a = 0; a < k1; ++a) s += gC[cells[e * k1 + a]];
  g[e] = vol[e] / k1 * s;
}

// Work buffers of a call, left on the handle for the next one (in the order of
// use, so the same call finds its sizes again).  A call takes them away from
// the handle while it runs: a second thread's call finds none and allocates
// its own.  More than kKeepBytes, or a second set, is freed at the end.
// Allocated and freed in the order of the call's stream: cudaMalloc and cudaFree
// wait for the whole device, other streams and handles included.  The calls end
// with a synchronisation of their stream, on errors in the destructor: the next
// call may use another one.
constexpr size_t kKeepBytes = (size_t)2 << 30;
struct Scratch {
  mg_mesh* M;
  cudaStream_t st;
  size_t next = 0;
  std::vector<FluxBuffer> own;
  Scratch(mg_mesh* m, cudaStream_t s) : M(m), st(s) { mesh_take_scratch(M, own); }
  ~Scratch() {
    cudaStreamSynchronize(st);
    size_t total = 0;
    for (const FluxBuffer& b : own) total += b.bytes;
    if (total > kKeepBytes || !mesh_keep_scratch(M, own))
      for (const FluxBuffer& b : own)
        if (b.p) cudaFreeAsync(b.p, st);
  }
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
  template <class T>
  T* get(size_t count) {
    const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
    if (next == own.size()) own.push_back({nullptr, 0});
    FluxBuffer& b = own[next++];
    if (b.bytes < bytes) {
      if (b.p) cudaFreeAsync(b.p, st);
      b = {nullptr, 0};
      if (cudaMallocAsync(&b.p, bytes, st) != cudaSuccess) {
        cudaGetLastError();
        b.p = nullptr;
        return nullptr;
      }
      b.bytes = bytes;
    }
    return static_cast<T*>(b.p);
  }
  template <class T>
  T* put(const T* src, size_t count) {   // host array
    T* x = get<T>(count);
    if (x && count &&
        cudaMemcpyAsync(x, src, count * sizeof(T), cudaMemcpyHostToDevice, st) != cudaSuccess)
      return nullptr;
    return x;
  }
  template <class T>
  T* put(const std::vector<T>& v) { return put(v.data(), v.size()); }
};

// Block and grid of a kernel over `count` cells or nodes of ld4 float4 each
// (item_of): rows of up to 256 float4, no division in the kernel.
struct ItemGrid {
  dim3 block, grid;
};
ItemGrid item_grid(int64_t count, int ld4) {
  const int ny = (ld4 + 255) / 256;
  const int bx = ny == 1 ? ld4 : ((ld4 + ny - 1) / ny + 31) / 32 * 32, by = 256 / bx;
  return {dim3(bx, by), dim3((unsigned)((count + by - 1) / by), ny)};
}

// Launch of a step kernel as a programmatic dependent (see pdl_sync).
template <class... KArgs, class... Args>
void launch_pdl(void (*kern)(KArgs...), const ItemGrid& g, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = g.grid;
  cfg.blockDim = g.block;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Everything the three entry points share: geometry, layer damping, event
// lists, source amplitudes, per-node coefficients, device inputs.
struct Flux {
  int d = 0, k1 = 0, S = 0, ld = 0, ld4 = 0, nt = 0;
  int64_t n = 0, m = 0, R = 0;
  double dt = 0.0;
  bool host = false;
  cudaStream_t st = nullptr;
  MeshView V;
  CoefArgs c;
  const double* eps_d = nullptr;
  FluxGeometry geo;
  float* keep = nullptr;    // 1 - dt zeta
  DevEvents ev{};
  float* fl = nullptr;      // f_l (FP32) per step, device
  float2* coef = nullptr;
  ResidentShape shape;      // lpr = 0: launches per step
  ResidentFluxArgs ra{};
  ResidentShape rshape;     // reverse steps

  // Steps [l, l + steps) with the resident kernel, from (p, q) (null: rest);
  // the last states into (out_p, out_q), every new p into hist, `state` floats
  // apart (each may be null).  MG_ERR_UNSUPPORTED before anything has run: the
  // launches per step are the path then.
  int advance(int l, int steps, const float* p, const float* q, float* out_p, float* out_q,
              float* hist, float* traces) {
    ResidentFluxArgs a = ra;
    a.step0 = l;
    a.steps = steps;
    a.p = p;
    a.q = q;
    a.out_p = out_p;
    a.out_q = out_q;
    a.hist = hist;
    a.traces = traces;
    for (a.col0 = 0; a.col0 < ld; a.col0 += 4 * shape.lpr) {
      const int rc = launch_resident_flux(a, d, shape, st);
      if (rc == MG_ERR_UNSUPPORTED && l == 0 && a.col0 == 0) shape.lpr = 0;
      if (rc != MG_OK) return rc;
    }
    return MG_OK;
  }
  // After the last launch: synchronises, and tells of a wait that ran out.
  int finish() {
    int word = 0;
    if (ra.status && cudaMemcpyAsync(&word, ra.status, sizeof(int), cudaMemcpyDeviceToHost, st) !=
                         cudaSuccess)
      return MG_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return MG_ERR_CUDA;
    return word ? MG_ERR_TIMEOUT : MG_OK;
  }

  // flux update from p (or, with sl.seg, from the slot of step sr)
  void step_q(float* p, float* q, cudaStream_t s, StepRef sr = {0, nullptr},
              Slots sl = {nullptr, 0, 1}) const {
    launch_pdl(d == 2 ? k_flux_q<2, 1> : k_flux_q<3, 1>, item_grid(m, ld4), s, m, ld4, geo.cell,
               keep, reinterpret_cast<const float4*>(p), reinterpret_cast<float4*>(q), (float)dt,
               sr, sl);
  }
  // node update of step sr: p_{l+1} into pout (nullptr: in place over p),
  // or with sl.seg from the step's slot into the next one
  void step_p(const float* q, float* p, float* traces, StepRef sr, cudaStream_t s,
              float* pout = nullptr, Slots sl = {nullptr, 0, 1}) const {
    launch_pdl(d == 2 ? k_flux_p<2> : k_flux_p<3>, item_grid(n, ld4), s, n, m, ld4, geo.inc_ptr,
               geo.inc, coef, reinterpret_cast<const float4*>(q),
               reinterpret_cast<const float4*>(p), reinterpret_cast<float4*>(pout ? pout : p), ev,
               fl, traces, nt, sr, sl);
  }
};

// One captured chunk of steps, replayed with cudaGraphLaunch on the
// caller's stream.  Recorded on a private stream (the caller's may be the
// legacy default stream, which cannot be captured); destroyed with the
// call, after the stream it ran on has drained.
struct Chunk {
  cudaGraphExec_t exec = nullptr;
  cudaStream_t used = nullptr;
  Chunk() = default;
  Chunk(const Chunk&) = delete;
  Chunk& operator=(const Chunk&) = delete;
  ~Chunk() {
    if (!exec) return;
    if (used) cudaStreamSynchronize(used);
    cudaGraphExecDestroy(exec);
  }
  template <class Body>
  int record(Body&& body) {
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return MG_ERR_CUDA;
    int rc = MG_OK;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      rc = MG_ERR_CUDA;
    } else {
      rc = body(cs);
      if (cudaStreamEndCapture(cs, &g) != cudaSuccess && rc == MG_OK) rc = MG_ERR_CUDA;
    }
    if (rc == MG_OK && cudaGraphInstantiate(&exec, g, 0) != cudaSuccess) {
      exec = nullptr;
      rc = MG_ERR_CUDA;
    }
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (rc != MG_OK) cudaGetLastError();
    return rc;
  }
  int launch(cudaStream_t st) {
    used = st;
    return cudaGraphLaunch(exec, st) == cudaSuccess ? MG_OK : MG_ERR_CUDA;
  }
};

#define MG_FX(x)                  \
  do {                            \
    const int rc_ = (x);          \
    if (rc_ != MG_OK) return rc_; \
  } while (0)

// The packed geometry of the handle's mesh, built on first use and kept with
// it: gradients of the barycentric functions and incidence weights |e|
// dphi_i/dx_k (FP64 -> FP32).
int flux_geometry(mg_mesh* M, const HostMesh& hm, FluxGeometry& out) {
  std::lock_guard<std::mutex> lock(mesh_flux_mutex(M));
  if (mesh_flux_geometry(M, &out)) return MG_OK;
  const int d = hm.dim, k1 = d + 1, cw = (k1 * k1 + 3) / 4;
  const int64_t n = hm.n, m = hm.m;
  std::vector<float> grad((size_t)m * k1 * d), cell((size_t)m * cw * 4, 0.0f);
  int bad = 0;
#pragma omp parallel for schedule(static) reduction(+ : bad)
  for (int64_t e = 0; e < m; ++e) {
    const int32_t* v = hm.cells.data() + (size_t)e * k1;
    double E[kMaxDim][kMaxDim], inv[kMaxDim][kMaxDim];
    for (int a = 0; a < d; ++a)
      for (int b = 0; b < d; ++b)
        E[a][b] = hm.coords[(size_t)v[b + 1] * d + a] - hm.coords[(size_t)v[0] * d + a];
    // inverse of E (columns x_b - x_0); rows of inv are grad phi_1..phi_d
    double det;
    if (d == 2) {
      det = E[0][0] * E[1][1] - E[0][1] * E[1][0];
      inv[0][0] = E[1][1] / det; inv[0][1] = -E[0][1] / det;
      inv[1][0] = -E[1][0] / det; inv[1][1] = E[0][0] / det;
    } else {
      det = E[0][0] * (E[1][1] * E[2][2] - E[1][2] * E[2][1]) -
            E[0][1] * (E[1][0] * E[2][2] - E[1][2] * E[2][0]) +
            E[0][2] * (E[1][0] * E[2][1] - E[1][1] * E[2][0]);
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
          const int a1 = (b + 1) % 3, a2 = (b + 2) % 3, b1 = (a + 1) % 3, b2 = (a + 2) % 3;
          inv[a][b] = (E[a1][b1] * E[a2][b2] - E[a1][b2] * E[a2][b1]) / det;
        }
    }
    if (!(det != 0.0) || !std::isfinite(det)) {
      ++bad;
      continue;
    }
    for (int k = 0; k < d; ++k) {
      double g0 = 0.0;
      for (int a = 1; a <= d; ++a) {
        const double g = inv[a - 1][k];
        grad[((size_t)e * k1 + a) * d + k] = (float)g;
        g0 -= g;
      }
      grad[((size_t)e * k1) * d + k] = (float)g0;
    }
    float* c = cell.data() + (size_t)e * cw * 4;
    for (int a = 0; a < k1; ++a) {
      std::memcpy(c + a, v + a, sizeof(float));
      for (int k = 0; k < d; ++k) c[k1 + a * d + k] = grad[((size_t)e * k1 + a) * d + k];
    }
  }
  std::vector<int32_t> ptr(n + 1);
  std::vector<int4> inc(hm.nc_cell.size());
  if (hm.nc_cell.size() > 0x7fffffff) return MG_ERR_UNSUPPORTED;
#pragma omp parallel for schedule(static) reduction(+ : bad)
  for (int64_t i = 0; i < n; ++i) {
    ptr[i] = (int32_t)hm.nc_ptr[i];
    for (int64_t s = hm.nc_ptr[i]; s < hm.nc_ptr[i + 1]; ++s) {
      const int32_t e = hm.nc_cell[s];
      int a = 0;
      while (a < k1 && hm.cells[(size_t)e * k1 + a] != i) ++a;
      if (a == k1) {
        ++bad;
        continue;
      }
      float w[3] = {0.0f, 0.0f, 0.0f};
      for (int k = 0; k < d; ++k)
        w[k] = (float)(hm.cell_vol[e] * grad[((size_t)e * k1 + a) * d + k]);
      int4 q = make_int4(e, 0, 0, 0);
      std::memcpy(&q.y, w, 3 * sizeof(float));
      inc[s] = q;
    }
  }
  ptr[n] = (int32_t)hm.nc_ptr[n];
  if (bad) return MG_ERR_ARG;
  // patches for the resident kernels, where one column of them can fit
  int n_sm = 0, smem = 0;
  if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, mesh_device(M)) ||
      cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, mesh_device(M)))
    return MG_ERR_CUDA;
  const int B = (int)std::min<int64_t>(n_sm, std::max<int64_t>(1, n / 32));
  HostFluxPatches H;
  if (((n + m * d) * 16 + m * 36 + (int64_t)inc.size() * 12) / B < smem) {
    int rc;
    try {
      rc = build_flux_patches(hm, B, inc, H);
    } catch (const std::bad_alloc&) {
      rc = MG_ERR_OOM;
    }
    if (rc == MG_ERR_UNSUPPORTED || rc == MG_ERR_OOM) H = HostFluxPatches();   // no patches
    else if (rc != MG_OK) return rc;
  }
  return mesh_set_flux_geometry(M, cell, ptr, inc, H, &out);
}

// whole_groups: pad the shots so that the float4s of a node (ld4) are a power
// of two up to 32 or a multiple of 32.  The node adjoint sums them with warp
// shuffles over such groups; any other count would put lanes of two nodes
// into one group and lanes outside the shuffle's mask (ld4 = 3 for 10 shots).
int flux_setup(mg_mesh* M, const double* eps, const mg_shots* shots, const double* wavelet,
               double dt, int nt, const double* xi, const double* zeta, int flags,
               cudaStream_t st, Scratch& X, Flux& F, bool whole_groups = false) {
  if (!M || !eps || !shots || !wavelet || nt < 1 || !(dt > 0.0)) return MG_ERR_ARG;
  const HostMesh* hm = host_mesh(M);
  const int d = hm->dim, k1 = d + 1;
  if (d < 2 || d > kMaxDim) return MG_ERR_UNSUPPORTED;
  const int S = shots->n_shots;
  if (S < 1 || !shots->src || !shots->rec_ptr || (shots->rec_ptr[S] > 0 && !shots->rec) ||
      shots->rec_ptr[0] != 0)
    return MG_ERR_ARG;
  const int64_t n = hm->n, m = hm->m, R = shots->rec_ptr[S];
  for (int s = 0; s < S; ++s) {
    if (shots->src[s] < 0 || shots->src[s] >= n || shots->rec_ptr[s + 1] < shots->rec_ptr[s])
      return MG_ERR_ARG;
  }
  for (int64_t r = 0; r < R; ++r)
    if (shots->rec[r] < 0 || shots->rec[r] >= n) return MG_ERR_ARG;
  const bool host = flags & MG_HOST_PTRS;
  F.d = d;
  F.k1 = k1;
  F.S = S;
  F.n = n;
  F.m = m;
  F.R = R;
  F.nt = nt;
  F.dt = dt;
  F.host = host;
  F.st = st;

  MG_FX(flux_geometry(M, *hm, F.geo));
  F.ld = S <= 4 ? 4 : ((S + 3) / 4) * 4;
  F.ld4 = F.ld / 4;
  if (whole_groups) {
    int g = 1;
    while (g < F.ld4 && g < 32) g <<= 1;
    F.ld4 = (F.ld4 + g - 1) / g * g;
    F.ld = 4 * F.ld4;
  }
  std::vector<int32_t> sp(n + 1, 0), ss(S), rp(n + 1, 0), rs(R), rt(R);
  const std::vector<int32_t>& perm = hm->perm;
  for (int s = 0; s < S; ++s) sp[perm[shots->src[s]] + 1]++;
  for (int64_t r = 0; r < R; ++r) rp[perm[shots->rec[r]] + 1]++;
  for (int64_t i = 0; i < n; ++i) {
    sp[i + 1] += sp[i];
    rp[i + 1] += rp[i];
  }
  {
    std::vector<int32_t> fs(sp.begin(), sp.end() - 1), fr(rp.begin(), rp.end() - 1);
    for (int s = 0; s < S; ++s) ss[fs[perm[shots->src[s]]]++] = s;
    for (int s = 0; s < S; ++s)
      for (int64_t r = shots->rec_ptr[s]; r < shots->rec_ptr[s + 1]; ++r) {
        const int32_t row = perm[shots->rec[r]];
        rs[fr[row]] = s;
        rt[fr[row]++] = (int32_t)r;
      }
  }
  // source amplitudes f_l = dt sum_{m <= l} s_m (FP64 sum, FP32 value)
  std::vector<double> wav_h(nt);
  if (host) std::copy(wavelet, wavelet + nt, wav_h.begin());
  else if (cudaMemcpy(wav_h.data(), wavelet, nt * sizeof(double), cudaMemcpyDeviceToHost) !=
           cudaSuccess)
    return MG_ERR_CUDA;
  std::vector<float> fl_h(nt);
  double acc = 0.0;
  for (int l = 0; l < nt; ++l) {
    acc += dt * wav_h[l];
    fl_h[l] = (float)acc;
  }

  if (mesh_view(M, &F.V) != MG_OK) return MG_ERR_ARG;
  F.eps_d = eps;
  const double* xi_d = xi;
  if (host) {
    F.eps_d = X.put(eps, (size_t)m);
    if (xi) xi_d = X.put(xi, (size_t)m);
    if (!F.eps_d || (xi && !xi_d)) return MG_ERR_OOM;
  }
  const double* zeta_d = zeta;
  if (host && zeta) {
    zeta_d = X.put(zeta, (size_t)m * d);
    if (!zeta_d) return MG_ERR_OOM;
  }
  F.keep = X.get<float>((size_t)m * d);
  int* bad = X.get<int>(1);
  if (!F.keep || !bad) return MG_ERR_OOM;
  if (cudaMemsetAsync(bad, 0, sizeof(int), st) != cudaSuccess) return MG_ERR_CUDA;
  k_flux_keep<<<(unsigned)((m * d + 255) / 256), 256, 0, st>>>(m * d, zeta_d, (float)dt, F.keep,
                                                               bad);
  int bad_h = 0;
  if (cudaMemcpyAsync(&bad_h, bad, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return MG_ERR_CUDA;
  if (bad_h) return MG_ERR_ARG;
  if (!(flags & MG_ALLOW_CFL)) {
    double dtc = 0.0;
    const int rc = mg_cfl_dt(M, F.eps_d, 0, st, &dtc);
    if (rc) return rc;
    if (dt > dtc * (1.0 + 1e-12)) return MG_ERR_CFL;
  }
  F.ev = {X.put(sp), X.put(ss), X.put(rp), X.put(rs), X.put(rt)};
  F.fl = X.put(fl_h);
  F.coef = X.get<float2>(n);
  if (!F.ev.src_ptr || !F.ev.src_shot || !F.ev.rec_ptr || !F.ev.rec_shot || !F.ev.rec_trace ||
      !F.fl || !F.coef)
    return MG_ERR_OOM;
  F.c = F.V.coef_base;
  F.c.eps = F.eps_d;
  k_flux_coefs<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(F.c, xi_d, dt, F.coef);
  return cudaGetLastError() == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}

// Chooses the path of a call's forward steps, `steps` of them at a time:
// the resident kernel when its estimate is below that of two launches per step
// (latency, then the gathers and states through L2).
int flux_path(mg_mesh* M, int steps, Scratch& X, Flux& F, bool reverse = false) {
  if (!F.geo.patches.B || steps < 16) return MG_OK;
  int smem = 0;
  if (cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, mesh_device(M)))
    return MG_ERR_CUDA;
  double us = 0.0;
  resident_flux_shape(F.geo.patches, F.d, F.ld4, smem - 1024, F.shape, us);
  // 16-byte accesses of a float4 column, at the measured rates: triangles 14 to
  // 18 TB/s with states in L2 and 10 beyond it, tetrahedra 5 to 10
  const double moved = ((double)F.m * (F.k1 * F.d + 3 * F.d + 1) + 2.0 * F.n) * F.ld4 * 16.0;
  const double held = ((double)F.m * F.d + F.n) * F.ld4 * 16.0;
  const double rows = 5.0 + moved / (F.d == 2 && held < 100e6 ? 17e6 : 10e6);
  if (us > rows) F.shape.lpr = 0;
  if (reverse && F.shape.lpr) {   // after resident forward steps only
    resident_flux_adj_shape(F.geo.patches, F.d, F.ld4, smem - 1024, F.rshape, us);
    if (us > rows) F.rshape.lpr = 0;
  }
  if (!F.shape.lpr) return MG_OK;
  ResidentFluxArgs& a = F.ra;
  a.P = F.geo.patches;
  a.ev = F.ev;
  a.coef = F.coef;
  a.cell = F.geo.cell;
  a.keep = F.keep;
  a.fl = F.fl;
  a.nt = F.nt;
  a.ld = F.ld;
  a.m = F.m;
  a.dt = (float)F.dt;
  a.state = F.n * F.ld;
  a.budget = mesh_wait_budget(M);
  a.xbuf = X.get<uint4>((size_t)2 * a.P.n_x * std::max(F.shape.lpr, F.rshape.lpr) * 2);
  a.status = X.get<int>(1);
  if (!a.xbuf || !a.status) {   // no memory: launches per step
    F.shape.lpr = F.rshape.lpr = 0;
    a.status = nullptr;
    return MG_OK;
  }
  return cudaMemsetAsync(a.status, 0, sizeof(int), F.st) == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}

struct DeviceScope {
  int prev = 0;
  bool ok = false;
  explicit DeviceScope(int dev) {
    ok = cudaGetDevice(&prev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess;
  }
  ~DeviceScope() { cudaSetDevice(prev); }
};


// Steps per CUDA-graph chunk for a call (0: plain launches): the handle's
// chunk length, unless MG_NO_GRAPH.
int chunk_len(const mg_mesh* M, int flags) {
  const int c = mesh_graph_chunk(M);
  return (flags & MG_NO_GRAPH) || c < 2 ? 0 : c;
}

}  // namespace
}  // namespace mg

extern "C" int mg_forward_pml(mg_mesh* M, const double* eps, const mg_shots* shots,
                              const double* wavelet, double dt, int nt, const double* xi,
                              const double* zeta, float* traces, void* stream, int flags) {
  using namespace mg;
  if (!M || !eps || !shots || !wavelet || !traces || nt < 1 || !(dt > 0.0)) return MG_ERR_ARG;
  if (flags & ~(MG_HOST_PTRS | MG_ALLOW_CFL | MG_NO_GRAPH)) return MG_ERR_UNSUPPORTED;
  DeviceScope scope(mesh_device(M));
  if (!scope.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Scratch X(M, st);
  Flux F;
  MG_FX(flux_setup(M, eps, shots, wavelet, dt, nt, xi, zeta, flags, st, X, F));
  const int64_t n = F.n, m = F.m, R = F.R;
  float* tr = F.host ? X.get<float>((size_t)R * nt) : traces;
  if (!tr) return MG_ERR_OOM;
  MG_FX(flux_path(M, nt, X, F));
  int l = 0;   // steps done
  if (F.shape.lpr) {
    const int rc = F.advance(0, nt, nullptr, nullptr, nullptr, nullptr, nullptr, tr);
    if (rc == MG_OK) l = nt;
    else if (rc != MG_ERR_UNSUPPORTED) return rc;
  }
  float *p = nullptr, *q = nullptr;
  int* base = nullptr;
  if (l < nt) {
    p = X.get<float>((size_t)n * F.ld);
    q = X.get<float>((size_t)F.d * m * F.ld);
    base = X.get<int>(1);
    if (!p || !q || !base) return MG_ERR_OOM;
    if (cudaMemsetAsync(p, 0, (size_t)n * F.ld * sizeof(float), st) ||
        cudaMemsetAsync(q, 0, (size_t)F.d * m * F.ld * sizeof(float), st))
      return MG_ERR_CUDA;
  }
  add_launches(M, 2 + (l ? (F.ld4 + F.shape.lpr - 1) / F.shape.lpr : 2 * (int64_t)nt));
  const int C = chunk_len(M, flags);
  Chunk ch;
  if (C && nt - l >= C) {   // whole chunks: one graph launch each
    MG_FX(launch_set_int(base, 0, st));
    MG_FX(ch.record([&](cudaStream_t cs) {
      for (int j = 0; j < C; ++j) {
        F.step_q(p, q, cs);
        F.step_p(q, p, tr, {j, base}, cs);
      }
      return launch_add_int(base, C, cs);
    }));
    for (; l + C <= nt; l += C) MG_FX(ch.launch(st));
  }
  for (; l < nt; ++l) {
    F.step_q(p, q, st);
    F.step_p(q, p, tr, {l, nullptr}, st);
  }
  if (cudaGetLastError() != cudaSuccess) return MG_ERR_CUDA;
  if (F.host && cudaMemcpyAsync(traces, tr, (size_t)R * nt * sizeof(float),
                                cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return MG_ERR_CUDA;
  return F.finish();
}

extern "C" int mg_jacobian_apply_pml(mg_mesh* M, int level, const double* eps,
                                     const mg_shots* shots, const double* wavelet, double dt,
                                     int nt, const double* xi, const double* zeta,
                                     const double* v, float* jv, void* stream, int flags) {
  using namespace mg;
  if (!M || !eps || !shots || !wavelet || !v || !jv || nt < 1 || !(dt > 0.0)) return MG_ERR_ARG;
  if (flags & ~(MG_HOST_PTRS | MG_ALLOW_CFL | MG_NO_GRAPH)) return MG_ERR_UNSUPPORTED;
  const HostMesh* hm = host_mesh(M);
  if (level < 0 || level >= hm->n_levels) return MG_ERR_ARG;
  DeviceScope scope(mesh_device(M));
  if (!scope.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Scratch X(M, st);
  Flux F;
  MG_FX(flux_setup(M, eps, shots, wavelet, dt, nt, xi, zeta, flags, st, X, F));
  const int64_t n = F.n, m = F.m, R = F.R, nc = hm->n_cells_level[level];
  const double* v_d = F.host ? X.put(v, (size_t)nc) : v;
  const int32_t* anc = X.put(hm->ancestors[level]);
  double* dv = X.get<double>(m);
  double* C = X.get<double>(n);
  double* dC = X.get<double>(n);
  float* ratio = X.get<float>(n);
  const size_t ns = (size_t)n * F.ld, qs = (size_t)F.d * m * F.ld;
  float* p = X.get<float>(ns);
  float* dp = X.get<float>(ns);
  float* q = X.get<float>(qs);
  float* dq = X.get<float>(qs);
  float* tr = F.host ? X.get<float>((size_t)R * nt) : jv;
  int* base = X.get<int>(1);
  if (!v_d || !anc || !dv || !C || !dC || !ratio || !p || !dp || !q || !dq || !tr || !base)
    return MG_ERR_OOM;
  MG_FX(launch_prolong(m, anc, v_d, nullptr, dv, st));
  const unsigned gn = (unsigned)((n + 255) / 256);
  k_flux_mass<<<gn, 256, 0, st>>>(F.c, F.eps_d, C);
  k_flux_mass<<<gn, 256, 0, st>>>(F.c, dv, dC);
  k_flux_ratio<<<gn, 256, 0, st>>>(n, dC, C, ratio);
  if (cudaMemsetAsync(p, 0, ns * sizeof(float), st) ||
      cudaMemsetAsync(dp, 0, ns * sizeof(float), st) ||
      cudaMemsetAsync(q, 0, qs * sizeof(float), st) ||
      cudaMemsetAsync(dq, 0, qs * sizeof(float), st))
    return MG_ERR_CUDA;
  const ItemGrid gp = item_grid(n, F.ld4);
  auto step = [&](StepRef sr, cudaStream_t s) {
    F.step_q(p, q, s);
    F.step_q(dp, dq, s);
    launch_pdl(F.d == 2 ? k_flux_p_tan<2> : k_flux_p_tan<3>, gp, s, n, m, F.ld4, F.geo.inc_ptr,
               F.geo.inc, F.coef, ratio, reinterpret_cast<const float4*>(q),
               reinterpret_cast<const float4*>(dq), reinterpret_cast<float4*>(p),
               reinterpret_cast<float4*>(dp), F.ev, F.fl, tr, nt, sr);
  };
  const int CL = chunk_len(M, flags);
  int l = 0;
  Chunk ch;
  if (CL && nt >= CL) {   // whole chunks: one graph launch each
    MG_FX(launch_set_int(base, 0, st));
    MG_FX(ch.record([&](cudaStream_t cs) {
      for (int j = 0; j < CL; ++j) step({j, base}, cs);
      return launch_add_int(base, CL, cs);
    }));
    for (; l + CL <= nt; l += CL) MG_FX(ch.launch(st));
  }
  for (; l < nt; ++l) step({l, nullptr}, st);
  if (cudaGetLastError() != cudaSuccess) return MG_ERR_CUDA;
  add_launches(M, 5 + 3 * (int64_t)nt);
  if (F.host && cudaMemcpyAsync(jv, tr, (size_t)R * nt * sizeof(float), cudaMemcpyDeviceToHost,
                                st) != cudaSuccess)
    return MG_ERR_CUDA;
  return cudaStreamSynchronize(st) == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}

extern "C" int mg_jacobian_T_apply_pml(mg_mesh* M, int level, const double* eps,
                                       const mg_shots* shots, const double* wavelet, double dt,
                                       int nt, const double* xi, const double* zeta,
                                       const float* w, double* g, int ckpt_every, void* stream,
                                       int flags) {
  using namespace mg;
  if (!M || !eps || !shots || !wavelet || !w || !g || nt < 1 || !(dt > 0.0) || ckpt_every < 1)
    return MG_ERR_ARG;
  if (flags & ~(MG_HOST_PTRS | MG_ALLOW_CFL | MG_NO_GRAPH)) return MG_ERR_UNSUPPORTED;
  const HostMesh* hm = host_mesh(M);
  if (level < 0 || level >= hm->n_levels) return MG_ERR_ARG;
  DeviceScope scope(mesh_device(M));
  if (!scope.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Scratch X(M, st);
  Flux F;
  MG_FX(flux_setup(M, eps, shots, wavelet, dt, nt, xi, zeta, flags, st, X, F, true));
  const int64_t n = F.n, m = F.m, R = F.R, nc = hm->n_cells_level[level];
  const int K = std::min(ckpt_every, nt);
  const int nck = (nt + K - 1) / K;
  // one segment (ckpt_every >= nt): the forward keeps every state, and the
  // reverse steps run with no recompute
  const bool keep = nck == 1;
  const size_t ns = (size_t)n * F.ld, qs = (size_t)F.d * m * F.ld;
  const int nseg = F.ld4 < 32 ? 1 : F.ld4 / 32;
  const float* W = F.host ? X.put(w, (size_t)R * nt) : w;
  float* ck_p = X.get<float>(ns * nck);
  float* ck_q = X.get<float>(qs * nck);
  float* seg = X.get<float>(ns * (K + 1));
  float* p = keep ? seg : X.get<float>(ns);   // the forward's state (keep: unused)
  float* q = X.get<float>(qs);
  float* trd = X.get<float>((size_t)R * nt);
  float* tp = X.get<float>(ns);
  float* rr = X.get<float>(ns);
  float* Qt = X.get<float>(qs);
  double* hacc = X.get<double>((size_t)n * nseg);
  double* C = X.get<double>(n);
  double* gC = X.get<double>(n);
  double* vol = X.put(hm->cell_vol);
  double* gf = X.get<double>(m);
  std::vector<int64_t> lp;
  std::vector<int32_t> li;
  level_children(*hm, level, lp, li);
  int64_t* lp_d = X.put(lp);
  int32_t* li_d = X.put(li);
  double* go = F.host ? X.get<double>(nc) : g;
  int* base = X.get<int>(1);
  if (!W || !ck_p || !ck_q || !p || !q || !seg || !trd || !tp || !rr || !Qt || !hacc || !C ||
      !gC || !vol || !gf || !lp_d || !li_d || !go || !base)
    return MG_ERR_OOM;
  if (cudaMemsetAsync(p, 0, ns * sizeof(float), st) ||
      cudaMemsetAsync(q, 0, qs * sizeof(float), st) ||
      cudaMemsetAsync(Qt, 0, qs * sizeof(float), st) ||
      cudaMemsetAsync(hacc, 0, (size_t)n * nseg * sizeof(double), st))
    return MG_ERR_CUDA;
  int64_t launches = 0;
  const int CL = chunk_len(M, flags);
  // p_l in slot l of seg (keep: the whole run, slots 0..nt) or in slot
  // l - l0 of the segment [l0, l0 + K) being reversed
  const Slots sl{reinterpret_cast<float4*>(seg), (int64_t)ns / 4, keep ? nt + 1 : K};
  // forward, keeping (p_l, q_{l-1/2}) at l = 0, K, 2K, ... (or every p_l)
  if (keep && cudaMemsetAsync(seg, 0, ns * sizeof(float), st)) return MG_ERR_CUDA;
  // resident: the forward steps in intervals of K; the last one's only as the
  // first segment's recompute
  MG_FX(flux_path(M, K, X, F, true));
  if (F.shape.lpr) {
    int rc = MG_OK;
    if (!keep && (cudaMemsetAsync(ck_p, 0, ns * sizeof(float), st) ||
                  cudaMemsetAsync(ck_q, 0, qs * sizeof(float), st)))
      return MG_ERR_CUDA;
    for (int c = 0; c < (keep ? 1 : nck - 1) && rc == MG_OK; ++c) {
      rc = keep ? F.advance(0, nt, nullptr, nullptr, nullptr, nullptr, seg + ns, nullptr)
                : F.advance(c * K, K, c ? ck_p + ns * c : nullptr, c ? ck_q + qs * c : nullptr,
                            ck_p + ns * (c + 1), ck_q + qs * (c + 1), nullptr, nullptr);
      launches += (F.ld4 + std::max(F.shape.lpr, 1) - 1) / std::max(F.shape.lpr, 1);
    }
    if (rc != MG_OK && rc != MG_ERR_UNSUPPORTED) return rc;
  }
  const bool res = F.shape.lpr > 0;
  auto fwd_slots = [&](StepRef sr, cudaStream_t s) {   // p_l in its slot, p_{l+1} the next
    F.step_q(seg, q, s, sr, sl);
    F.step_p(q, seg, trd, sr, s, nullptr, sl);
  };
  auto fwd = [&](StepRef sr, cudaStream_t s) {
    if (keep) {
      fwd_slots(sr, s);
    } else {
      F.step_q(p, q, s);
      F.step_p(q, p, trd, sr, s);
    }
  };
  // graph chunks: keep, CL steps; else one checkpoint interval of K steps
  const int LF = keep ? CL : (CL ? K : 0);
  int l = res ? nt : 0;
  Chunk chf;
  if (LF >= 2 && nt - l >= LF) {
    MG_FX(launch_set_int(base, 0, st));
    MG_FX(chf.record([&](cudaStream_t cs) {
      for (int j = 0; j < LF; ++j) fwd({j, base}, cs);
      return launch_add_int(base, LF, cs);
    }));
    for (; l + LF <= nt; l += LF) {
      if (!keep &&
          (cudaMemcpyAsync(ck_p + ns * (l / K), p, ns * sizeof(float), cudaMemcpyDeviceToDevice,
                           st) ||
           cudaMemcpyAsync(ck_q + qs * (l / K), q, qs * sizeof(float), cudaMemcpyDeviceToDevice,
                           st)))
        return MG_ERR_CUDA;
      MG_FX(chf.launch(st));
      launches += 2 * LF;
    }
  }
  for (; l < nt; ++l) {
    if (!keep && l % K == 0 &&
        (cudaMemcpyAsync(ck_p + ns * (l / K), p, ns * sizeof(float), cudaMemcpyDeviceToDevice,
                         st) ||
         cudaMemcpyAsync(ck_q + qs * (l / K), q, qs * sizeof(float), cudaMemcpyDeviceToDevice,
                         st)))
      return MG_ERR_CUDA;
    fwd({l, nullptr}, st);
    launches += 2;
  }
  // reverse step l: p_l, p_{l+1} from their slots
  const ItemGrid gp = item_grid(n, F.ld4), gq = item_grid(m, F.ld4);
  const float fdt = (float)dt;
  auto rev = [&](StepRef sr, cudaStream_t s) {
    launch_pdl(F.d == 2 ? k_flux_adj_p<2> : k_flux_adj_p<3>, gp, s, n, m, F.ld4, F.geo.inc_ptr,
               F.geo.inc, F.coef, reinterpret_cast<const float4*>(Qt),
               reinterpret_cast<float4*>(tp), reinterpret_cast<float4*>(rr), sl, hacc, F.ev, W, nt,
               sr, fdt);
    launch_pdl(F.d == 2 ? k_flux_q<2, -1> : k_flux_q<3, -1>, gq, s, m, F.ld4, F.geo.cell, F.keep,
               reinterpret_cast<const float4*>(rr), reinterpret_cast<float4*>(Qt), 1.0f,
               StepRef{0, nullptr}, Slots{nullptr, 0, 1});
  };
  // segment [l0, l0 + len) with p_{l0} in slot 0 and q_{l0-1/2} in q: its
  // forward steps into slots 1..len (q in place), then the reverse steps
  // l0 + len - 1 .. l0; s0 is step l0
  auto segment = [&](int len, StepRef s0, cudaStream_t s) {
    for (int j = 0; j < len && !res; ++j) fwd_slots({s0.l + j, s0.base}, s);
    for (int j = len - 1; j >= 0; --j) rev({s0.l + j, s0.base}, s);
  };
  // reverse steps l0 + len - 1 .. l0 with the resident kernel, p_{l0} in slot 0
  auto reverse = [&](int l0, int len) {
    ResidentFluxAdjArgs a{};
    a.P = F.geo.patches;
    a.ev = F.ev;
    a.coef = F.coef;
    a.cell = F.geo.cell;
    a.keep = F.keep;
    a.w = W;
    a.nt = nt;
    a.k = l0 + len - 1;
    a.steps = len;
    a.ld = F.ld;
    a.nseg = nseg;
    a.m = m;
    a.dt = fdt;
    a.p = seg + ns * (len - 1);
    a.state = (int64_t)ns;
    a.tp = tp;
    a.Qt = Qt;
    a.hacc = hacc;
    a.xbuf = F.ra.xbuf;
    a.status = F.ra.status;
    a.budget = F.ra.budget;
    int rc = MG_OK;
    for (; a.col0 < F.ld && rc == MG_OK; a.col0 += 4 * F.rshape.lpr) {
      rc = launch_resident_flux_adj(a, F.d, F.rshape, st);
      launches += 1;
    }
    if (rc == MG_ERR_UNSUPPORTED && l0 + len == nt) F.rshape.lpr = 0;   // nothing has run
    return rc;
  };
  Chunk chr;
  if (keep) {   // reverse steps nt-1 .. 0 in chunks of CL (base: the chunk's first step)
    int k = nt;   // steps below k remain
    if (res && F.rshape.lpr) {
      const int rc = reverse(0, nt);
      if (rc == MG_OK) k = 0;
      else if (rc != MG_ERR_UNSUPPORTED) return rc;
    }
    if (CL >= 2 && k >= CL) {
      MG_FX(launch_set_int(base, nt - 1, st));
      MG_FX(chr.record([&](cudaStream_t cs) {
        for (int j = 0; j < CL; ++j) rev({-j, base}, cs);
        return launch_add_int(base, -CL, cs);
      }));
      for (; k >= CL; k -= CL) {
        MG_FX(chr.launch(st));
        launches += 2 * CL;
      }
    }
    for (int r = k - 1; r >= 0; --r) {
      rev({r, nullptr}, st);
      launches += 2;
    }
  } else {
    const int nfull = nt / K;
    auto load = [&](int c) {   // checkpoint c into slot 0 and q (resident: its segment)
      const int len = std::min(K, nt - c * K);
      if (res) {
        launches += (F.ld4 + F.shape.lpr - 1) / F.shape.lpr;
        return cudaMemcpyAsync(seg, ck_p + ns * c, ns * sizeof(float), cudaMemcpyDeviceToDevice,
                               st) == cudaSuccess &&
               F.advance(c * K, len, ck_p + ns * c, ck_q + qs * c, nullptr, nullptr, seg + ns,
                         nullptr) == MG_OK;
      }
      return cudaMemcpyAsync(seg, ck_p + ns * c, ns * sizeof(float), cudaMemcpyDeviceToDevice,
                             st) == cudaSuccess &&
             cudaMemcpyAsync(q, ck_q + qs * c, qs * sizeof(float), cudaMemcpyDeviceToDevice,
                             st) == cudaSuccess;
    };
    int c0 = nck;   // segments below c0 remain
    while (res && F.rshape.lpr && c0 > 0) {
      const int c = c0 - 1, len = std::min(K, nt - c * K);
      if (!load(c)) return MG_ERR_CUDA;
      const int rc = reverse(c * K, len);
      if (rc == MG_OK) c0 = c;
      else if (rc != MG_ERR_UNSUPPORTED) return rc;
    }
    if (c0 > 0 && nt % K) {   // the last, shorter segment: plain launches
      if (!load(nfull)) return MG_ERR_CUDA;
      segment(nt - nfull * K, {nfull * K, nullptr}, st);
      launches += (res ? 2 : 4) * (int64_t)(nt - nfull * K);
    }
    if (CL && K >= 2 && nfull >= 1 && c0 > 0) {   // full segments: one graph launch each
      MG_FX(launch_set_int(base, (nfull - 1) * K, st));
      MG_FX(chr.record([&](cudaStream_t cs) {
        segment(K, {0, base}, cs);
        return launch_add_int(base, -K, cs);
      }));
      for (int c = nfull - 1; c >= 0; --c) {
        if (!load(c)) return MG_ERR_CUDA;
        MG_FX(chr.launch(st));
        launches += (res ? 2 : 4) * (int64_t)K;
      }
    } else {
      for (int c = std::min(c0, nfull) - 1; c >= 0; --c) {
        if (!load(c)) return MG_ERR_CUDA;
        segment(K, {c * K, nullptr}, st);
        launches += (res ? 2 : 4) * (int64_t)K;
      }
    }
  }
  // gradient: C-sensitivity per node, per finest cell, restricted to the level
  const unsigned gn = (unsigned)((n + 255) / 256), gm = (unsigned)((m + 255) / 256);
  k_flux_mass<<<gn, 256, 0, st>>>(F.c, F.eps_d, C);
  k_flux_hsum<<<gn, 256, 0, st>>>(n, nseg, hacc, C, gC);
  k_flux_cell_grad<<<gm, 256, 0, st>>>(m, F.k1, F.geo.cells, vol, gC, gf);
  if (cudaGetLastError() != cudaSuccess) return MG_ERR_CUDA;
  MG_FX(launch_restrict(nc, lp_d, li_d, gf, go, st));
  add_launches(M, launches + 5);
  if (F.host && cudaMemcpyAsync(g, go, nc * sizeof(double), cudaMemcpyDeviceToHost, st) !=
                    cudaSuccess)
    return MG_ERR_CUDA;
  return F.finish();
}
