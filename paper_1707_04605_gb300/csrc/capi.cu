// C ABI of the leapfrog wave library: mesh handle, device residency,
// scratch management and the forward / tangent / adjoint drivers.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <initializer_list>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/mgwave.h"
#include "kernels.cuh"
#include "mg_internal.h"
#include "mesh_view.h"
#include "resident.h"

namespace {

struct Buf {
  void* p = nullptr;
  size_t bytes = 0;
};

int ensure(Buf& b, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (b.bytes >= bytes) return MG_OK;
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.bytes = 0;
  if (cudaMalloc(&b.p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return MG_ERR_OOM;
  }
  b.bytes = bytes;
  return MG_OK;
}

template <class T>
int upload(Buf& b, const std::vector<T>& v) {
  int rc = ensure(b, v.size() * sizeof(T));
  if (rc) return rc;
  if (!v.empty() && cudaMemcpy(b.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess)
    return MG_ERR_CUDA;
  return MG_OK;
}

template <class T>
T* P(Buf& b) { return static_cast<T*>(b.p); }
template <class T>
T* P_(const Buf& b) { return static_cast<T*>(b.p); }

int round_pad(int S) {
  if (S <= 4) return 4;
  if (S <= 128) {
    int p = 4;
    while (p < S) p <<= 1;
    return p;
  }
  return (S + 127) / 128 * 128;
}

// RAII: make the handle's device current for the duration of a call.
struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; cudaGetLastError(); return; }
    if (prev != dev && cudaSetDevice(dev) != cudaSuccess) { ok = false; cudaGetLastError(); }
  }
  ~DeviceGuard() {
    int cur;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

}  // namespace

struct mg_mesh {
  int device = 0;
  mg::HostMesh hm;
  // resident mesh arrays
  Buf ell, slice_off, slice_w, nc_ptr, nc_cell, nc_w, nf_ptr, nf_cell, nf_w,
      is_bnd, row_abs, cells, vol, cf_ptr, cf_facet, bnd, bnd_meas;
  std::vector<Buf> anc, lvl_ptr, lvl_idx;  // per level, uploaded on first use
  // scratch
  Buf eps_h, wav_h, wavf, coef, tcoef, mass, scal, stA, stB, stC, stD, out_h,
      w_h, v_h, g_h, ev, G, ckpt, seg, gfine, step_base;
  // event cache
  std::vector<int32_t> ev_src, ev_rec;
  std::vector<int64_t> ev_ptr;
  int ev_S_pad = 0;
  int64_t ev_n_src = 0, ev_n_rec = 0;
  bool ev_valid = false;
  int64_t ev_gen = 0;                     // bumped whenever the event lists change
  // checkpoints of the last mg_forward with MG_KEEP_CHECKPOINTS
  bool ck_valid = false;
  bool seg_full = false;                  // seg holds p_{-1}..p_nt of that forward (MG_KEEP_STATES)
  int ck_every = 0, ck_nt = 0, ck_S_pad = 0, ck_nshots = 0;
  double ck_dt = 0.0;
  int64_t ck_ev_gen = -1;
  int64_t ck_gen = 0;                     // bumped whenever checkpoints or kept states change
  int64_t launches = 0;
  // CUDA graphs of step chunks, keyed by kind, buffers and sizes
  int chunk = 128;                        // steps per graph (even), 0 = off
  // per kernel kind (0 forward/recompute, 1 tangent, 2 adjoint): row-kernel
  // float4 vectors per lane, shared-memory tile rows (0 = row kernel), shots
  // per staged pass, shot groups advanced one after another inside a graph
  // chunk or checkpoint segment
  struct Tuning {
    int batch = 1;
    int tile_rows = 0;
    int src_tile = 32;
    int groups = 1;
    int min_blocks = 0;   // forward row kernel: 0, or 5 resident CTAs per SM
    int bulk = 0;         // forward: neighbour rows staged by bulk async copies
    int ring = 0;         // row kernels: gather ring of 4 or 8 slots per lane, 0 = plain loads
    int sweep = 0;        // forward row kernel: consecutive row blocks per CTA (0, 1: one)
    int tma = 0;          // forward: rows per tile of the bulk-copy tiled kernel (0 = off)
    int stream = 0;       // row kernels: once-read loads bypass L1 allocation
    int prefetch = 0;     // capped row kernels: prefetch of late-loaded rows (1 L1, 2 L2)
    int wide = 1;         // capped forward: 8 consecutive shots per lane (256-bit loads)
    int path = MG_PATH_AUTO;   // what runs (mg_mesh_set_kernel_path)
  } tune[3];
  int dep_launch = 1;                     // row kernels launched as programmatic dependents
  Buf ellu;                               // ELL with every slice padded to wu columns
  Buf ellc;                               // chunk-major ELL for cchunk lanes per row
  int cchunk = 0;                         // its chunk (0: none)
  int64_t cstride = 0;                    // entries per slice in it
  bool chunked_ell = false;
  std::map<int, Buf> auto_ellc;           // the same for the default launch shapes, by chunk
  int auto_w = 0;                         // and the widest slice, once one of them is built
  int wu = 0;
  bool uniform_ell = false;
  int cache_hints = 1;                    // kept history: L2 evict-first on last reads
  Buf errbuf;                             // device status word of bounded waits, then the
                                          // persistent forward's barrier counter
  int persist_steps = 128;                // MG_PERSISTENT: steps per cooperative launch
  long long persist_budget = 1LL << 31;   // SM clock cycles one barrier wait may take
  int persist_extra = 0;                  // barrier arrivals awaited beyond the grid (tests)
  struct TileTables {
    Buf ell_off, ell_idx, ell_val, sinfo, halo_off, halo_cnt, halo;
    int n_tiles = 0, max_ell = 0, max_halo = 0;
    double ratio = 0.0;
  };
  std::map<int, TileTables> tiles;        // by rows per tile
  int smem_optin = 0;
  int n_sm = 0;
  // partitions of the resident kernels by patch count, their row groups by rows
  // per warp
  struct PatchTables {
    mg::HostPatches host;                 // B = 0: the mesh cannot be cut so
    struct Groups {
      std::array<Buf, 11> buf;
      mg::DevPatches dev{};               // sizes; the pointers once on_device
      bool on_device = false;
      std::unique_ptr<mg::HostGroups> host;   // until uploaded, where the choice took them
    };
    std::map<int, Groups> groups;
  };
  std::map<int, PatchTables> patches;
  Buf xbuf;                               // resident kernels: exchange of border rows
  bool status_clear = false;              // the running call cleared the status word for them
  // autotuned choices by (n_shots padded), so repeated calls skip the search
  std::map<int, std::array<Tuning, 3>> tuned;
  cudaStream_t cap = nullptr;             // private capture stream
  std::map<std::string, cudaGraphExec_t> graphs;
  Buf sigma;                              // conductivity per finest cell (FP64)
  bool has_sigma = false;
  Buf tr;                                 // internal trace buffer [R][nt]
  Buf trf;                                // forward traces of the fused forward + tangent
  Buf tune_scratch;                       // autotuner inputs/outputs
  std::vector<mg::FluxBuffer> flux_scratch;   // work buffers of the flux path's calls
  mutable std::mutex flux_mu;             // guards them and the packed geometry
  Buf flux_cell, flux_ptr, flux_inc, flux_pinc;      // its packed geometry
  std::array<Buf, 13> flux_tab;           // and patch tables
  mg::DevFluxPatches flux_patches{};
};

namespace {

const char* kErr[] = {"ok", "invalid argument", "invalid nesting", "out of device memory",
                      "CUDA error", "dt above the CFL bound", "device wait timed out",
                      "unsupported combination"};

mg::DevEll dev_ell(mg_mesh* M) {
  mg::DevEll K{P<const int2>(M->ell), P<const int64_t>(M->slice_off),
               P<const int32_t>(M->slice_w), (int32_t)M->hm.n};
  if (M->uniform_ell && M->ellu.p) {
    K.ellu = P<const int2>(M->ellu);
    K.wu = M->wu;
  }
  if (M->chunked_ell && M->ellc.p) {
    K.ellc = P<const int2>(M->ellc);
    K.cchunk = M->cchunk;
    K.cstride = M->cstride;
  }
  return K;
}

mg::CoefArgs coef_args(mg_mesh* M, const double* eps, double dt) {
  mg::CoefArgs c;
  c.n = (int32_t)M->hm.n;
  c.nc_ptr = P<int64_t>(M->nc_ptr); c.nc_cell = P<int32_t>(M->nc_cell); c.nc_w = P<double>(M->nc_w);
  c.nf_ptr = P<int64_t>(M->nf_ptr); c.nf_cell = P<int32_t>(M->nf_cell); c.nf_w = P<double>(M->nf_w);
  c.is_bnd = P<int32_t>(M->is_bnd);
  c.eps = eps;
  c.dt = dt;
  c.bc = M->hm.bc;
  c.coef = P<float4>(M->coef);
  c.mass = nullptr;
  c.sigma = M->has_sigma ? P<double>(M->sigma) : nullptr;
  return c;
}

int validate_shots(mg_mesh* M, const mg_shots* sh) {
  if (!sh || sh->n_shots < 1 || !sh->src || !sh->rec_ptr) return MG_ERR_ARG;
  if (sh->rec_ptr[0] != 0) return MG_ERR_ARG;
  for (int k = 0; k < sh->n_shots; ++k) {
    if (sh->src[k] < 0 || sh->src[k] >= M->hm.n) return MG_ERR_ARG;
    if (sh->rec_ptr[k + 1] < sh->rec_ptr[k]) return MG_ERR_ARG;
  }
  const int64_t R = sh->rec_ptr[sh->n_shots];
  if (R > 0 && !sh->rec) return MG_ERR_ARG;
  if (R > 0x7fffffffLL) return MG_ERR_ARG;
  for (int64_t r = 0; r < R; ++r)
    if (sh->rec[r] < 0 || sh->rec[r] >= M->hm.n) return MG_ERR_ARG;
  return MG_OK;
}

// Per-row source / receiver lists of a shot batch, uploaded once per batch.
int build_events(mg_mesh* M, const mg_shots* sh, mg::DevEvents& ev) {
  const int64_t n = M->hm.n;
  const int S = sh->n_shots;
  const int64_t R = sh->rec_ptr[S];
  std::vector<int32_t> src(sh->src, sh->src + S), rec(sh->rec, sh->rec + R);
  std::vector<int64_t> ptr(sh->rec_ptr, sh->rec_ptr + S + 1);
  const bool same = M->ev_valid && src == M->ev_src && rec == M->ev_rec && ptr == M->ev_ptr;
  const size_t total = 2 * (size_t)(n + 1) + S + 2 * (size_t)R;
  if (!same) {
    std::vector<int32_t> h(total, 0);
    int32_t* src_ptr = h.data();
    int32_t* src_shot = src_ptr + (n + 1);
    int32_t* rec_ptr = src_shot + S;
    int32_t* rec_shot = rec_ptr + (n + 1);
    int32_t* rec_trace = rec_shot + R;
    for (int k = 0; k < S; ++k) src_ptr[M->hm.perm[src[k]] + 1]++;
    for (int64_t r = 0; r < n; ++r) src_ptr[r + 1] += src_ptr[r];
    {
      std::vector<int32_t> fill(src_ptr, src_ptr + n);
      for (int k = 0; k < S; ++k) src_shot[fill[M->hm.perm[src[k]]]++] = k;
    }
    for (int64_t r = 0; r < R; ++r) rec_ptr[M->hm.perm[rec[r]] + 1]++;
    for (int64_t r = 0; r < n; ++r) rec_ptr[r + 1] += rec_ptr[r];
    {
      std::vector<int32_t> fill(rec_ptr, rec_ptr + n);
      for (int k = 0; k < S; ++k)
        for (int64_t r = ptr[k]; r < ptr[k + 1]; ++r) {
          const int32_t pos = fill[M->hm.perm[rec[r]]]++;
          rec_shot[pos] = k;
          rec_trace[pos] = (int32_t)r;
        }
    }
    int rc = upload(M->ev, h);
    if (rc) return rc;
    M->ev_src = src;
    M->ev_rec = rec;
    M->ev_ptr = ptr;
    M->ev_valid = true;
    M->ev_gen++;
  }
  int32_t* base = P<int32_t>(M->ev);
  ev.src_ptr = base;
  ev.src_shot = base + (n + 1);
  ev.rec_ptr = ev.src_shot + S;
  ev.rec_shot = ev.rec_ptr + (n + 1);
  ev.rec_trace = ev.rec_shot + R;
  return MG_OK;
}

int ensure_level(mg_mesh* M, int level) {
  if (M->anc[level].p) return MG_OK;
  int rc = upload(M->anc[level], M->hm.ancestors[level]);
  if (rc) return rc;
  std::vector<int64_t> ptr;
  std::vector<int32_t> idx;
  mg::level_children(M->hm, level, ptr, idx);
  rc = upload(M->lvl_ptr[level], ptr);
  if (rc) return rc;
  return upload(M->lvl_idx[level], idx);
}

// Inputs: device pointers, staged from the host when MG_HOST_PTRS is set.
int stage_in(Buf& b, const void* src, size_t bytes, int flags, cudaStream_t st,
             const void** dev) {
  if (!(flags & MG_HOST_PTRS)) { *dev = src; return MG_OK; }
  int rc = ensure(b, bytes);
  if (rc) return rc;
  if (cudaMemcpyAsync(b.p, src, bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return MG_ERR_CUDA;
  *dev = b.p;
  return MG_OK;
}

// Results leave the handle's buffer for the caller's: device to device on
// the stream, or device to host followed by a stream synchronisation.
int deliver(Buf& b, void* dst, size_t bytes, int flags, cudaStream_t st) {
  if (bytes == 0) return MG_OK;
  const bool host = flags & MG_HOST_PTRS;
  if (cudaMemcpyAsync(dst, b.p, bytes, host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice,
                      st) != cudaSuccess)
    return MG_ERR_CUDA;
  if (!host) return MG_OK;
  return cudaStreamSynchronize(st) == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}

// Flags every propagation call accepts; each adds its own.
constexpr int kCommonFlags = MG_HOST_PTRS | MG_NO_GRAPH | MG_ALLOW_CFL;

#define MG_TRY(x) do { int _rc = (x); if (_rc != MG_OK) return _rc; } while (0)
#define MG_CU(x) do { if ((x) != cudaSuccess) { cudaGetLastError(); return MG_ERR_CUDA; } } while (0)

int cfl_lambda(mg_mesh* M, const double* eps_d, cudaStream_t st, double* lam) {
  MG_TRY(ensure(M->mass, M->hm.n * sizeof(double)));
  MG_TRY(ensure(M->coef, M->hm.n * sizeof(float4)));
  MG_TRY(ensure(M->scal, 8 * sizeof(double)));
  mg::CoefArgs c = coef_args(M, eps_d, 1.0);
  c.mass = P<double>(M->mass);
  MG_TRY(mg::launch_coefs(c, st));
  MG_TRY(mg::launch_cfl_reduce((int32_t)M->hm.n, P<double>(M->row_abs), P<double>(M->mass),
                               P<double>(M->scal), st));
  M->launches += 2;
  MG_CU(cudaMemcpyAsync(lam, M->scal.p, sizeof(double), cudaMemcpyDeviceToHost, st));
  MG_CU(cudaStreamSynchronize(st));
  return MG_OK;
}

int ensure_tiles(mg_mesh* M);
mg_mesh::Tuning in_force(const mg_mesh* M, int kind);

// Common preparation of a propagation call: inputs on the device, per-row
// coefficients, wavelet in FP32, event lists, dt check.
struct Prep {
  const double* eps = nullptr;
  const double* wav = nullptr;
  mg::DevEvents ev{};
  int S = 0, S_pad = 0, tiles = 1;
  int64_t R = 0;
};

int* err_word(mg_mesh* M);

int prepare(mg_mesh* M, const double* eps, const mg_shots* shots, const double* wavelet,
            double dt, int nt, int flags, cudaStream_t st, Prep& pp) {
  if (!eps || !wavelet || nt < 1 || !(dt > 0.0) || !std::isfinite(dt)) return MG_ERR_ARG;
  M->status_clear = false;
  MG_TRY(validate_shots(M, shots));
  pp.S = shots->n_shots;
  pp.S_pad = round_pad(pp.S);
  pp.tiles = pp.S_pad >= 128 ? pp.S_pad / 128 : 1;
  pp.R = shots->rec_ptr[pp.S];
  const void* d;
  MG_TRY(stage_in(M->eps_h, eps, M->hm.m * sizeof(double), flags, st, &d));
  pp.eps = static_cast<const double*>(d);
  MG_TRY(stage_in(M->wav_h, wavelet, nt * sizeof(double), flags, st, &d));
  pp.wav = static_cast<const double*>(d);
  if (!(flags & MG_ALLOW_CFL)) {
    double lam = 0.0;
    MG_TRY(cfl_lambda(M, pp.eps, st, &lam));
    if (!(lam > 0.0) || dt > 2.0 / std::sqrt(lam) * (1.0 + 1e-12)) return MG_ERR_CFL;
  }
  MG_TRY(ensure(M->coef, M->hm.n * sizeof(float4)));
  MG_TRY(mg::launch_coefs(coef_args(M, pp.eps, dt), st));
  MG_TRY(ensure(M->wavf, nt * sizeof(float)));
  MG_TRY(mg::launch_d2f(pp.wav, P<float>(M->wavf), nt, st));
  M->launches += 2;
  MG_TRY(build_events(M, shots, pp.ev));
  MG_TRY(ensure_tiles(M));
  // the status word of bounded device waits exists before any graph capture
  const mg_mesh::Tuning t = in_force(M, 0);
  if ((t.bulk || t.tma) && !err_word(M)) return MG_ERR_OOM;
  return MG_OK;
}

// Tile tables for every tile size the kernel kinds use, built on the host
// and uploaded on first use.
int ensure_tiles(mg_mesh* M) {
  for (int k = 0; k < 4; ++k) {
    const int P = k < 3 ? in_force(M, k).tile_rows : in_force(M, 0).tma;
    if (P <= 0 || M->tiles.count(P)) continue;
    mg::HostTiles T;
    MG_TRY(mg::build_tiles(M->hm, P, T));
    mg_mesh::TileTables& D = M->tiles[P];
    MG_TRY(upload(D.ell_off, T.ell_off));
    MG_TRY(upload(D.ell_idx, T.ell_idx));
    MG_TRY(upload(D.ell_val, T.ell_val));
    MG_TRY(upload(D.sinfo, T.slice_info));
    MG_TRY(upload(D.halo_off, T.halo_off));
    MG_TRY(upload(D.halo_cnt, T.halo_cnt));
    MG_TRY(upload(D.halo, T.halo));
    D.n_tiles = (int)T.n_tiles;
    D.max_ell = T.max_ell;
    D.max_halo = T.max_halo;
    D.ratio = T.halo_ratio;
  }
  if (!M->smem_optin)
    MG_CU(cudaDeviceGetAttribute(&M->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin,
                                 M->device));
  return MG_OK;
}

// Launch shape in force for a kind: the one on the handle where its path says
// so, else the defaults (row_shape picks the library's own).
mg_mesh::Tuning in_force(const mg_mesh* M, int kind) {
  const mg_mesh::Tuning& t = M->tune[kind];
  if (t.path == MG_PATH_SHAPE || t.path == MG_PATH_RESIDENT) return t;
  mg_mesh::Tuning d;
  d.stream = t.stream;
  d.prefetch = t.prefetch;
  d.wide = t.wide;
  d.path = t.path;
  return d;
}

// Shot columns per group of a kernel kind: S_pad / groups when that is a
// valid launch width (a power of two >= 4 up to 128, or a multiple of 128),
// else S_pad (one group).
int group_cols(const mg_mesh* M, int kind, int S_pad) {
  const int G = in_force(M, kind).groups;
  if (G <= 1 || S_pad % G) return S_pad;
  const int W = S_pad / G;
  const bool ok = W >= 4 && (W % 128 == 0 || (W <= 128 && (W & (W - 1)) == 0));
  return ok ? W : S_pad;
}

// Tiled launch description for `cols` shot columns per launch and a kernel
// kind (0 forward, 1 tangent, 2 adjoint), or n_tiles = 0 when that kind runs
// the row kernel (no tiles, or the tiled footprint exceeds shared memory).
// The tangent stages two states per pass, so it passes half as many shots
// to stay within the one-state footprint.
// Device tables of the P-row tiling (built by ensure_tiles), or n_tiles = 0.
mg::DevTiles tile_tables(mg_mesh* M, int P) {
  mg::DevTiles T{};
  auto it = M->tiles.find(P);
  if (P <= 0 || it == M->tiles.end()) return T;
  const mg_mesh::TileTables& D = it->second;
  T.P = P;
  T.n_tiles = D.n_tiles;
  T.ell_off = P_<const int64_t>(D.ell_off);
  T.ell_idx = P_<const uint16_t>(D.ell_idx);
  T.ell_val = P_<const float>(D.ell_val);
  T.slice_info = P_<const int32_t>(D.sinfo);
  T.halo_off = P_<const int64_t>(D.halo_off);
  T.halo_cnt = P_<const int32_t>(D.halo_cnt);
  T.halo = P_<const int32_t>(D.halo);
  T.max_ell = D.max_ell;
  T.max_halo = D.max_halo;
  return T;
}

mg::DevTiles dev_tiles(mg_mesh* M, int cols, int kind) {
  mg::DevTiles T{};
  const mg_mesh::Tuning t = in_force(M, kind);
  const int P = t.tile_rows;
  auto it = M->tiles.find(P);
  if (P <= 0 || it == M->tiles.end()) return T;
  const mg_mesh::TileTables& D = it->second;
  T.P = P;
  T.n_tiles = D.n_tiles;
  T.ell_off = P_<const int64_t>(D.ell_off);
  T.ell_idx = P_<const uint16_t>(D.ell_idx);
  T.ell_val = P_<const float>(D.ell_val);
  T.slice_info = P_<const int32_t>(D.sinfo);
  T.halo_off = P_<const int64_t>(D.halo_off);
  T.halo_cnt = P_<const int32_t>(D.halo_cnt);
  T.halo = P_<const int32_t>(D.halo);
  T.max_ell = D.max_ell;
  T.max_halo = D.max_halo;
  T.st_w = std::min(t.src_tile, cols);
  if (kind == 1) T.st_w = std::max(4, T.st_w / 2);
  if (mg::tiled_smem_bytes(T, kind) > (size_t)M->smem_optin) T.n_tiles = 0;
  return T;
}

// Device words of bounded waits: status (mg_mesh_device_status), arrivals of the
// persistent kernels' barrier, whether the kept states come from a launch whose
// wait ran out, and how many outputs were set to NaN so far.
enum { kWordStatus, kWordArrivals, kWordKept, kWordPoisoned };
int* err_word(mg_mesh* M) {
  if (!M->errbuf.p) {
    if (ensure(M->errbuf, 16) != MG_OK) return nullptr;
    if (cudaMemset(M->errbuf.p, 0, 16) != cudaSuccess) return nullptr;
  }
  return P<int>(M->errbuf);
}

// Launch shape of a kind on `cols` columns: the one that was asked for, or by
// default (from 16 columns on) two float4 per lane under the register cap with
// chunk-major entries, for the tangent one float4 per lane under the cap (it
// gathers two states).  Measured against one float4 without the cap and by
// column, us per step: forward, 232,505 nodes of tetrahedra, 128 shots 190.9 ->
// 114.8, 32 shots 60.2 -> 38.4, 8 shots 18.9 -> 18.5; reverse steps, 62,641
// nodes, 128 shots 39.0 -> 26.4, 256 shots 85.2 -> 59.6; tangent, 62,641 nodes,
// 128 shots 55.3 -> 49.2, 30,525 nodes of tetrahedra, 256 shots 71.7 -> 65.1.
// The source tiles of the adjoint stay 128 columns wide: the same sums.
struct RowShape {
  int batch, min_blocks, most_cols;
  bool chunked;   // from M->auto_ellc
};
RowShape row_shape(const mg_mesh* M, int kind, int cols) {
  const mg_mesh::Tuning t = in_force(M, kind);
  if (t.path == MG_PATH_SHAPE || t.path == MG_PATH_RESIDENT || cols < 16)
    return {t.batch, t.min_blocks, 512, false};
  return {kind == 1 ? 1 : 2, 5, 128, !M->chunked_ell};
}

// Chunk-major entries for the default shape of a kind, built on the device on
// first use (before any graph capture) where there is memory for them.
int ensure_auto_entries(mg_mesh* M, int kind, int cols, cudaStream_t st) {
  const RowShape r = row_shape(M, kind, cols);
  const int chunk = mg::rows_lanes(cols, r.batch, kind == 2 ? r.most_cols : 512);
  if (!r.chunked || chunk < 2 || chunk > 16) return MG_OK;
  Buf& b = M->auto_ellc[chunk];
  if (b.p) return MG_OK;
  int w = 0;
  for (int32_t x : M->hm.slice_w) w = std::max(w, (int)x);
  const int64_t stride = (int64_t)(w + chunk - 1) / chunk * mg::kSliceH * chunk;
  M->auto_w = w;
  if (ensure(b, (size_t)M->hm.n_slices * stride * sizeof(int2)) != MG_OK)
    return MG_OK;   // no memory: the entries as they are
  M->launches += 1;
  return mg::launch_chunk_entries(dev_ell(M), chunk, stride, P<int2>(b), st);
}

void use_auto_entries(mg_mesh* M, const RowShape& r, int kind, int cols, mg::DevEll& K) {
  if (!r.chunked) return;
  const int chunk = mg::rows_lanes(cols, r.batch, kind == 2 ? r.most_cols : 512);
  auto it = M->auto_ellc.find(chunk);
  if (it == M->auto_ellc.end() || !it->second.p) return;
  K.ellc = P<const int2>(it->second);
  K.cchunk = chunk;
  K.cstride = (int64_t)(M->auto_w + chunk - 1) / chunk * mg::kSliceH * chunk;
}

int do_step(mg_mesh* M, const mg::StepArgs& a, int S_pad, cudaStream_t st) {
  const int cols = a.cols ? a.cols : S_pad;
  const mg::DevTiles T = dev_tiles(M, cols, 0);
  if (T.n_tiles) return mg::launch_step_tiled(a, T, st);
  mg::StepArgs b = a;
  const RowShape rs = row_shape(M, 0, cols);
  b.batch = rs.batch;
  b.min_blocks = rs.min_blocks;
  use_auto_entries(M, rs, 0, cols, b.K);
  const mg_mesh::Tuning t = in_force(M, 0);
  b.ring = t.ring;
  b.sweep = t.sweep;
  b.stream = t.stream;
  b.prefetch = t.prefetch;
  b.wide = t.wide;
  b.pdl = M->dep_launch;
  if (t.tma) {
    const mg::DevTiles TT = tile_tables(M, t.tma);
    int* err = err_word(M);
    if (!err) return MG_ERR_OOM;
    if (!TT.n_tiles) return MG_ERR_ARG;
    return mg::launch_step_tma(b, TT, S_pad, err, st);
  }
  if (t.bulk) {
    int* err = err_word(M);
    if (!err) return MG_ERR_OOM;
    return mg::launch_step_bulk(b, S_pad, err, st);
  }
  return mg::launch_step(b, S_pad, st);
}

void row_tangent_args(mg_mesh* M, int cols, mg::TangentArgs& b) {
  const RowShape rs = row_shape(M, 1, cols);
  b.f.batch = rs.batch;
  b.f.min_blocks = rs.min_blocks;
  use_auto_entries(M, rs, 1, cols, b.f.K);
  const mg_mesh::Tuning t = in_force(M, 1);
  b.f.ring = t.ring;
  b.f.stream = t.stream;
  b.f.prefetch = t.prefetch;
  b.f.pdl = M->dep_launch;
}

int do_tangent(mg_mesh* M, const mg::TangentArgs& a, int S_pad, cudaStream_t st) {
  const mg::DevTiles T = dev_tiles(M, a.f.cols ? a.f.cols : S_pad, 1);
  if (T.n_tiles) return mg::launch_tangent_tiled(a, T, st);
  mg::TangentArgs b = a;
  row_tangent_args(M, a.f.cols ? a.f.cols : S_pad, b);
  return mg::launch_tangent(b, S_pad, st);
}

int do_adjoint(mg_mesh* M, const mg::AdjointArgs& a, int S_pad, cudaStream_t st) {
  const mg::DevTiles T = dev_tiles(M, a.cols ? a.cols : S_pad, 2);
  if (T.n_tiles) return mg::launch_adjoint_tiled(a, T, st);
  mg::AdjointArgs b = a;
  const int cols = a.cols ? a.cols : S_pad;
  const RowShape rs = row_shape(M, 2, cols);
  b.batch = rs.batch;
  b.min_blocks = rs.min_blocks;
  b.most_cols = rs.most_cols;
  use_auto_entries(M, rs, 2, cols, b.K);
  const mg_mesh::Tuning t = in_force(M, 2);
  b.ring = t.ring;
  b.stream = t.stream;
  b.prefetch = t.prefetch;
  b.pdl = M->dep_launch;
  return mg::launch_adjoint(b, S_pad, st);
}

// Accumulator sets of the adjoint when every launch covers `cols` columns:
// one for the tiled kernel (a CTA sums all shots of its rows, launches run
// one after another), else one per source tile of the whole shot range.
int adjoint_sets(mg_mesh* M, int S_pad, int cols) {
  if (dev_tiles(M, cols, 2).n_tiles) return 1;
  const RowShape rs = row_shape(M, 2, cols);
  return (S_pad / cols) * mg::rows_tiles(cols, rs.batch, rs.most_cols);
}

mg::StepArgs step_args(mg_mesh* M, const Prep& pp, int ld, int nt) {
  mg::StepArgs a{};
  a.K = dev_ell(M);
  a.ev = pp.ev;
  a.coef = P<const float4>(M->coef);
  a.ld = ld;
  a.wavelet = P<const float>(M->wavf);
  a.nt = nt;
  a.step_base = nullptr;
  a.batch = in_force(M, 0).batch;
  return a;
}

// Replays a captured sequence of launches on `st`.  The sequence is recorded
// once per key on the handle's private capture stream (the caller's stream
// may be the legacy default stream, which cannot be captured); step indices
// inside it are relative to the device int `step_base`.
template <class F>
int run_graph(mg_mesh* M, const std::string& key, int nodes, cudaStream_t st, F&& record) {
  auto it = M->graphs.find(key);
  cudaGraphExec_t exec = nullptr;
  if (it == M->graphs.end()) {
    if (!M->cap) MG_CU(cudaStreamCreateWithFlags(&M->cap, cudaStreamNonBlocking));
    MG_CU(cudaStreamBeginCapture(M->cap, cudaStreamCaptureModeThreadLocal));
    const int rc = record(M->cap);
    cudaGraph_t g = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(M->cap, &g);
    if (rc != MG_OK || ec != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return rc != MG_OK ? rc : MG_ERR_CUDA;
    }
    const cudaError_t ei = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (ei != cudaSuccess) { cudaGetLastError(); return MG_ERR_CUDA; }
    M->graphs[key] = exec;
  } else {
    exec = it->second;
  }
  MG_CU(cudaGraphLaunch(exec, st));
  M->launches += nodes;
  return MG_OK;
}

std::string key_of(const char* kind, std::initializer_list<const void*> ptrs,
                   std::initializer_list<long long> ints) {
  std::string k(kind);
  char buf[32];
  for (const void* p : ptrs) { snprintf(buf, sizeof buf, "|%p", p); k += buf; }
  for (long long v : ints) { snprintf(buf, sizeof buf, "|%lld", v); k += buf; }
  return k;
}

bool graphs_on(mg_mesh* M, int flags) { return M->chunk >= 2 && !(flags & MG_NO_GRAPH); }

// Barrier arguments of the handle's persistent launches (status word and
// counter, cleared on the stream first).
int persist_args(mg_mesh* M, cudaStream_t st, float* seg, size_t state, mg::PersistArgs& pa) {
  int* status = err_word(M);
  if (!status) return MG_ERR_OOM;
  MG_CU(cudaMemsetAsync(status, 0, sizeof(int), st));
  pa.count = reinterpret_cast<unsigned*>(status + kWordArrivals);
  pa.status = status;
  pa.budget = M->persist_budget;
  pa.extra = M->persist_extra;
  pa.seg = seg;
  pa.state = (int64_t)state;
  return MG_OK;
}

// After persistent launches: wait for them, then MG_ERR_TIMEOUT (status
// word cleared) if a barrier wait ran out.
int persist_status(mg_mesh* M, cudaStream_t st) {
  int word = 0;
  MG_CU(cudaMemcpyAsync(&word, M->errbuf.p, sizeof(int), cudaMemcpyDeviceToHost, st));
  MG_CU(cudaStreamSynchronize(st));
  if (word == 0) return MG_OK;
  MG_CU(cudaMemset(M->errbuf.p, 0, sizeof(int)));
  return MG_ERR_TIMEOUT;
}

// Row groups of the partition into B patches with rpw rows per warp, built on
// the host on first use: their sizes (kept) and, when asked for, their tables on
// the host or the device.  MG_ERR_UNSUPPORTED (remembered) when the mesh cannot
// be cut so, MG_ERR_OOM when the host's memory runs out.
using PatchGroups = mg_mesh::PatchTables::Groups;
int patch_groups(mg_mesh* M, int B, int rpw, bool tables, PatchGroups*& out) {
  try {
    auto it = M->patches.find(B);
    if (it == M->patches.end()) {
      mg::HostPatches H;
      const int rc = mg::build_patches(M->hm, B, H);
      if (rc == MG_ERR_OOM) return rc;
      if (rc != MG_OK) H = mg::HostPatches();
      it = M->patches.emplace(B, mg_mesh::PatchTables()).first;
      it->second.host = std::move(H);
    }
    mg_mesh::PatchTables& T = it->second;
    if (!T.host.B) return MG_ERR_UNSUPPORTED;
    auto ig = T.groups.find(rpw);
    if (ig == T.groups.end() || (tables && !ig->second.on_device && !ig->second.host)) {
      std::unique_ptr<mg::HostGroups> G(new mg::HostGroups());
      mg::group_rows(M->hm, T.host, rpw, *G);
      PatchGroups& R = T.groups[rpw];
      mg::DevPatches& d = R.dev;
      d.B = B;
      d.n_x = G->x_off[B];
      d.max_pairs = G->max_pairs;
      d.max_groups = G->max_groups;
      d.uniform = G->uniform;
      d.max_halo = G->max_halo;
      d.max_slots = G->max_slots;
      R.host = std::move(G);
      ig = T.groups.find(rpw);
    }
    out = &ig->second;
    return MG_OK;
  } catch (const std::bad_alloc&) {
    return MG_ERR_OOM;
  }
}

// The groups' tables on the device, all of them or none.
int upload_groups(PatchGroups& R) {
  if (R.on_device) return MG_OK;
  const mg::HostGroups& G = *R.host;
  std::array<Buf, 11> b;
  int k = 0, rc = MG_OK;
  auto put = [&](const auto& v) {
    Buf& x = b[k++];
    if (rc == MG_OK) rc = upload(x, v);
    return x.p;
  };
  mg::DevPatches d = R.dev;
  d.grp_off = static_cast<const int32_t*>(put(G.grp_off));
  d.border = static_cast<const int32_t*>(put(G.border));
  d.pair_off = static_cast<const int32_t*>(put(G.pair_off));
  d.halo_off = static_cast<const int32_t*>(put(G.halo_off));
  d.x_off = static_cast<const int32_t*>(put(G.x_off));
  d.hdr = static_cast<const int32_t*>(put(G.hdr));
  d.row = static_cast<const int32_t*>(put(G.row));
  d.halo = static_cast<const int32_t*>(put(G.halo));
  d.halo_x = static_cast<const int32_t*>(put(G.halo_x));
  d.diag = static_cast<const float*>(put(G.diag));
  d.pair = static_cast<const int4*>(put(G.pair));
  // a copy from pageable memory may still be under way when it returns: the
  // caller's stream need not wait for the one that it ran on
  if (rc == MG_OK && cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) rc = MG_ERR_CUDA;
  if (rc != MG_OK) {
    cudaGetLastError();
    for (Buf& x : b)
      if (x.p) cudaFree(x.p);
    return rc;
  }
  R.dev = d;
  R.buf = b;
  R.host.reset();
  R.on_device = true;
  return MG_OK;
}

// Estimates of a step's time on the two paths, in us, from measurements at 2 to
// 256 columns on triangles (3,997 to 249,697 nodes) and tetrahedra (30,525), most
// within 15% of them.  Resident: a launch per column group, each the exchange of
// border rows, the patch's shared memory accesses (a row read by fewer than 8
// lanes conflicts with others, less so on triangles, whose neighbours lie side by
// side) and its halo's; where many narrow launches follow one another (large
// patches) also their table fills, over the steps of a launch.  Row kernels:
// launch and tail, then the gathers (fewer than 16 columns run one float4 per
// lane without the register cap), or the states' traffic when they exceed L2.
//
// hist: a step's states also go to a history, `mb` MB of them.  The row kernels
// write them in whole rows.  A resident launch writes the columns of its group,
// and its other columns of the same sectors come launches later, when these have
// left L2: less than 128 bytes a row cost their sectors again, 16 bytes (one
// lane) a sector each, more so the more launches there are.  Measured, us per
// step without and with history: 249,697 nodes x 256 shots (one lane, 64
// launches) 185 and 494 to 625, with row kernels 163 and 181; 197,377 x 256
// (two lanes) 111 and 168, row kernels 130 and 144; 151,201 x 256 (four) 76 and
// 99, 100 and 111; 62,641 x 256 (eight) 28.5 and 33, 43 and 48.  The row kernels'
// rows of 64 and 128 bytes cost more than wider ones: 120,601 x 16 8.1 and 10.0,
// x 32 10.8 and 12.9.
double history_us(int lanes, int launches, double mb) {
  const double per_mb = launches == 1 ? 0.1 : lanes >= 8 ? 0.07 : lanes == 4 ? 0.15
                        : lanes == 2 ? std::min(0.28, 0.08 * launches)
                                     : std::min(1.7, 0.08 * launches);
  return per_mb * mb;
}
double resident_us(const mg::DevPatches& D, const mg::ResidentShape& s, int kind, int S_pad,
                   int steps, double mb) {
  const bool tri = D.uniform == 3;
  const double conflicts = s.lpr >= 8   ? 1.0
                           : s.lpr == 4 ? (tri ? 1.15 : 1.5)
                           : s.lpr == 2 ? (tri ? 1.15 : 2.4)
                                        : 1.6;
  const double pairs = (double)D.max_pairs / (D.max_groups * (32 / s.lpr));
  const double group = 14.0 + pairs * (1.0 + 8.0 * conflicts) + (kind == 1 ? 6.0 : kind == 2 ? 12.0 : 0.0);
  const int launches = S_pad / (kind == 1 ? 2 * s.lpr : 4 * s.lpr);
  const double fill = s.lpr <= 2 ? 12.0 / steps : 0.0;
  return launches * (0.9 + 0.65e-3 * group * D.max_groups + 0.3e-3 * D.max_halo * 2 * s.lpr + fill) +
         history_us(kind == 1 ? s.lpr / 2 : s.lpr, launches, mb);
}
double rows_us(const mg_mesh* M, int kind, int S_pad, double mb) {
  const double work = (double)M->hm.rowptr.back() * S_pad, cols = (double)M->hm.n * S_pad;
  const bool tri = M->hm.rowptr.back() < 8 * M->hm.n;
  const double gathers = kind == 0   ? 4.0 + (S_pad < 16 ? 0.4e-6 : 0.27e-6) * work
                         : kind == 2 ? 4.0 + 0.38e-6 * work
                         : tri       ? 4.5 + 0.54e-6 * work
                                     : 4.0 + 0.5e-6 * work;
  const double held = (kind == 1 ? 16.0 : 8.0) * cols;   // bytes of the states of a step
  const double moved = (kind == 0 ? 12.0 : kind == 1 ? 24.0 : 16.0) * cols;
  const double hist = (kind == 1 ? 0.02 : S_pad == 16 ? 0.2 : S_pad == 32 ? 0.14 : 0.07) * mb;
  if (held < (kind == 1 ? 65e6 : 100e6)) return gathers + hist;
  const double rate = kind == 1 ? (held < 200e6 ? 3.8e6 : 4.2e6) : held < 150e6 ? 4.1e6 : 4.5e6;
  return std::max(gathers, moved / rate) + hist;
}

// Resident launch shape of a call that advances S_pad columns for `steps`
// steps (launch, tables and exchange buffer cost about 10 us: at least 16 of
// them).  Forward: the widest column group whose patches fit; tangent: the
// same with p and dp as columns (2 lpr shots per launch); adjoint: whole source
// tiles of the row kernel only, for the same sums over the shots.
// shape.lpr = 0: the row kernels are the path (nothing fits, they are estimated
// to be faster, the kind's path asks for them, or there is no memory for the
// tables, which they need none of; MG_PATH_RESIDENT leaves the estimate out,
// but for calls that write a history).
int resident_shape(mg_mesh* M, int kind, int S_pad, int steps, mg::DevPatches& D,
                   mg::ResidentShape& shape, bool hist = false) {
  shape = mg::ResidentShape();
  const int path = M->tune[kind].path;
  if (path == MG_PATH_SHAPE || path == MG_PATH_ROWS || steps < 16 || M->hm.max_row_nnz > 256)
    return MG_OK;
  if (!M->n_sm)
    MG_CU(cudaDeviceGetAttribute(&M->n_sm, cudaDevAttrMultiProcessorCount, M->device));
  const int B = (int)std::min<int64_t>(M->n_sm, std::max<int64_t>(1, M->hm.n / 32));
  const int widest = kind == 1 ? std::min(32, S_pad / 2) : std::min(S_pad, 128) / 4;
  const int row_bytes = kind == 1 ? 8 : kind == 2 ? 16 : 0;
  PatchGroups* R = nullptr;
  for (int lpr = widest; lpr >= (kind == 1 ? 2 : 1); lpr >>= 1) {
    // where rows and entries alone are too large no tables are needed to see it
    const int64_t rows = M->hm.n / B, entries = (M->hm.rowptr.back() - M->hm.n) / B;
    if (rows * (32 * lpr + 20 + row_bytes) + entries * 8 <= M->smem_optin) {
      if (patch_groups(M, B, 32 / lpr, false, R) != MG_OK) return MG_OK;
      if (mg::resident_fit(R->dev, lpr, row_bytes, M->smem_optin - 1024, shape) == MG_OK) break;
      shape = mg::ResidentShape();
      R->host.reset();
    }
    if (kind == 2) break;
  }
  if (!shape.lpr) return MG_OK;
  const double mb = hist ? 4e-6 * (double)M->hm.n * S_pad : 0.0;
  if ((path == MG_PATH_AUTO || hist) &&
      resident_us(R->dev, shape, kind, S_pad, steps, mb) > rows_us(M, kind, S_pad, mb)) {
    shape.lpr = 0;
    R->host.reset();
    return MG_OK;
  }
  int rc = patch_groups(M, B, 32 / shape.lpr, true, R);
  if (rc == MG_OK) rc = upload_groups(*R);
  if (rc == MG_OK) D = R->dev;
  else shape.lpr = 0;
  return rc == MG_ERR_OOM ? MG_OK : rc;
}

// Exchange buffer and status word (cleared once per call) of resident launches;
// MG_ERR_UNSUPPORTED (the row kernels are the path) when there is no memory.
template <class A>
int resident_buffers(mg_mesh* M, const mg::DevPatches& D, int lpr, cudaStream_t st, A& r) {
  r.status = err_word(M);
  if (!r.status || ensure(M->xbuf, (size_t)2 * D.n_x * lpr * 2 * sizeof(uint4)) != MG_OK)
    return MG_ERR_UNSUPPORTED;
  if (!M->status_clear) MG_CU(cudaMemsetAsync(r.status, 0, sizeof(int), st));
  M->status_clear = true;
  r.xbuf = P<uint4>(M->xbuf);
  r.budget = M->persist_budget;
  return MG_OK;
}

// Outputs of a call become NaN where one of its resident launches ran out of a
// wait, or (reused) those that kept the states it has read.
int poison(mg_mesh* M, float* x, int64_t n, bool reused, cudaStream_t st) {
  if (!M->errbuf.p || !(M->status_clear || reused)) return MG_OK;
  int* w = P<int>(M->errbuf);
  M->launches += 1;
  return mg::launch_poison(x, n, M->status_clear ? w + kWordStatus : nullptr,
                           reused ? w + kWordKept : nullptr, w + kWordStatus, w + kWordPoisoned,
                           st);
}

// After the launches of a call that keeps states: whether they can be trusted.
int note_kept(mg_mesh* M, cudaStream_t st) {
  if (!M->errbuf.p) return MG_OK;
  int* w = P<int>(M->errbuf);
  M->launches += 1;
  return mg::launch_note_kept(M->status_clear ? w + kWordStatus : nullptr, w + kWordKept, st);
}

mg::ResidentArgs resident_args(mg_mesh* M, const Prep& pp, int nt, const mg::DevPatches& D) {
  mg::ResidentArgs r{};
  r.P = D;
  r.ev = pp.ev;
  r.coef = P<const float4>(M->coef);
  r.wavelet = P<const float>(M->wavf);
  r.nt = nt;
  r.steps = nt;
  r.ld = pp.S_pad;
  r.state = (int64_t)M->hm.n * pp.S_pad;
  return r;
}

// p_{l+1} .. p_{l+steps} of the states p_l, p_{l-1} into hist (state floats
// apart), every column group.
int run_recompute_resident(mg_mesh* M, const Prep& pp, int nt, int l, int steps, const float* p,
                           const float* pm, float* hist, const mg::DevPatches& D,
                           const mg::ResidentShape& shape, cudaStream_t st) {
  mg::ResidentArgs r = resident_args(M, pp, nt, D);
  MG_TRY(resident_buffers(M, D, shape.lpr, st, r));
  r.step0 = l;
  r.steps = steps;
  r.p = p;
  r.pm = pm;
  r.hist = hist;
  for (r.col0 = 0; r.col0 < pp.S_pad; r.col0 += 4 * shape.lpr) {
    MG_TRY(mg::launch_resident_step(r, shape, st));
    M->launches += 1;
  }
  return MG_OK;
}

// The tangent (and with traces or hist the forward it rides on) from rest.
int run_tangent_resident(mg_mesh* M, const Prep& pp, int nt, float* traces, float* dtraces,
                         float* hist, const mg::DevPatches& D, const mg::ResidentShape& shape,
                         cudaStream_t st) {
  mg::ResidentArgs r = resident_args(M, pp, nt, D);
  MG_TRY(resident_buffers(M, D, shape.lpr, st, r));
  r.tcoef = P<const float2>(M->tcoef);
  r.traces = traces;
  r.dtraces = dtraces;
  r.hist = hist;
  for (r.col0 = 0; r.col0 < pp.S_pad; r.col0 += 2 * shape.lpr) {
    MG_TRY(mg::launch_resident_tangent(r, shape, st));
    M->launches += 1;
  }
  for (float* x : {traces, dtraces})
    if (x) MG_TRY(poison(M, x, pp.R * nt, false, st));
  return MG_OK;
}

// Steps [0, nt) with the resident kernel, one launch per column group and
// checkpoint interval.  Checkpoints as run_forward's; hist: slot j of it
// receives p_{j-1} (slots 0 and 1 zero).  MG_ERR_UNSUPPORTED before anything
// has run when the device cannot hold the launch.
int run_forward_resident(mg_mesh* M, const Prep& pp, int nt, float* traces, int ckpt_every,
                         float* ckpt, float* hist, const mg::DevPatches& D,
                         const mg::ResidentShape& shape, cudaStream_t st) {
  const size_t state = (size_t)M->hm.n * pp.S_pad;
  mg::ResidentArgs r = resident_args(M, pp, nt, D);
  r.traces = traces;
  MG_TRY(resident_buffers(M, D, shape.lpr, st, r));
  if (hist) MG_CU(cudaMemsetAsync(hist, 0, 2 * state * sizeof(float), st));
  if (ckpt) MG_CU(cudaMemsetAsync(ckpt, 0, 2 * state * sizeof(float), st));
  const int len = ckpt ? ckpt_every : nt;
  for (int l = 0; l < nt; l += len) {
    r.step0 = l;
    r.steps = std::min(len, nt - l);
    float* slot = ckpt && l ? ckpt + (size_t)(l / len) * 2 * state : nullptr;
    float* next = ckpt && l + len < nt ? ckpt + (size_t)(l / len + 1) * 2 * state : nullptr;
    r.p = slot;
    r.pm = slot ? slot + state : nullptr;
    r.out_p = next;
    r.out_pm = next ? next + state : nullptr;
    r.hist = hist ? hist + (size_t)(l + 2) * state : nullptr;
    for (r.col0 = 0; r.col0 < pp.S_pad; r.col0 += 4 * shape.lpr) {
      MG_TRY(mg::launch_resident_step(r, shape, st));
      M->launches += 1;
    }
  }
  return traces ? poison(M, traces, pp.R * nt, false, st) : MG_OK;
}

// Batched forward loop over steps [0, nt); optional traces and checkpoints.
// Whole chunks of M->chunk steps run as one graph launch each.
int run_forward(mg_mesh* M, const Prep& pp, int nt, float* traces, int ckpt_every,
                float* ckpt, cudaStream_t st, int flags) {
  const int64_t n = M->hm.n;
  const size_t state = (size_t)n * pp.S_pad;
  if (!(flags & MG_PERSISTENT)) {
    mg::DevPatches D;
    mg::ResidentShape shape;
    MG_TRY(resident_shape(M, 0, pp.S_pad, ckpt ? std::min(ckpt_every, nt) : nt, D, shape));
    if (shape.lpr) {
      const int rc =
          run_forward_resident(M, pp, nt, traces, ckpt_every, ckpt, nullptr, D, shape, st);
      if (rc != MG_ERR_UNSUPPORTED) return rc;
    }
    MG_TRY(ensure_auto_entries(M, 0, group_cols(M, 0, pp.S_pad), st));
  }
  MG_TRY(ensure(M->stA, state * sizeof(float)));
  MG_TRY(ensure(M->stB, state * sizeof(float)));
  float* p = P<float>(M->stA);
  float* pm = P<float>(M->stB);
  MG_CU(cudaMemsetAsync(p, 0, state * sizeof(float), st));
  MG_CU(cudaMemsetAsync(pm, 0, state * sizeof(float), st));
  mg::StepArgs a = step_args(M, pp, pp.S_pad, nt);
  a.traces = traces;
  int l = 0;
  if (flags & MG_PERSISTENT) {
    // several steps per cooperative launch, ending at every checkpoint; the
    // status word is cleared first (a stale time-out would stop the barrier)
    mg::PersistArgs pa{};
    MG_TRY(persist_args(M, st, nullptr, 0, pa));
    while (l < nt) {
      if (ckpt && l % ckpt_every == 0) {
        float* slot = ckpt + (size_t)(l / ckpt_every) * 2 * state;
        MG_TRY(mg::launch_copy_f4(p, slot, (int64_t)state, st));
        MG_TRY(mg::launch_copy_f4(pm, slot + state, (int64_t)state, st));
        M->launches += 2;
      }
      int end = std::min(nt, l + M->persist_steps);
      if (ckpt) end = std::min(end, (l / ckpt_every + 1) * ckpt_every);
      a.p = p;
      a.pm = pm;
      a.pout = pm;
      a.step = l;
      pa.steps = end - l;
      MG_TRY(mg::launch_step_persist(a, pp.S_pad, pa, st));
      M->launches += 1;
      if ((end - l) % 2) std::swap(p, pm);
      l = end;
    }
    return MG_OK;
  }
  const int C = M->chunk;
  if (graphs_on(M, flags) && nt >= C && (!ckpt || ckpt_every % C == 0)) {
    MG_TRY(ensure(M->step_base, 16));
    int32_t* base = P<int32_t>(M->step_base);
    MG_TRY(mg::launch_set_int(base, 0, st));
    M->launches += 1;
    const int W = group_cols(M, 0, pp.S_pad), NG = pp.S_pad / W;
    const std::string key = key_of("fwd", {p, pm, traces, a.wavelet, a.coef, a.ev.src_ptr, base},
                                   {pp.S_pad, pp.S, pp.R, nt, C, n, W});
    for (; l + C <= nt; l += C) {
      if (ckpt && l % ckpt_every == 0) {
        float* slot = ckpt + (size_t)(l / ckpt_every) * 2 * state;
        MG_TRY(mg::launch_copy_f4(p, slot, (int64_t)state, st));
        MG_TRY(mg::launch_copy_f4(pm, slot + state, (int64_t)state, st));
        M->launches += 2;
      }
      MG_TRY(run_graph(M, key, NG * C + 1, st, [&](cudaStream_t cs) {
        mg::StepArgs b = a;
        b.step_base = base;
        b.cols = W;
        for (int g = 0; g < NG; ++g) {   // each shot group runs the whole chunk
          b.col0 = g * W;
          float* x = p;
          float* y = pm;
          for (int j = 0; j < C; ++j) {
            b.p = x;
            b.pm = y;
            b.pout = y;
            b.step = j;
            MG_TRY(do_step(M, b, pp.S_pad, cs));
            std::swap(x, y);
          }
        }
        return mg::launch_add_int(base, C, cs);
      }));
    }
  }
  for (; l < nt; ++l) {
    if (ckpt && l % ckpt_every == 0) {
      float* slot = ckpt + (size_t)(l / ckpt_every) * 2 * state;
      MG_TRY(mg::launch_copy_f4(p, slot, (int64_t)state, st));
      MG_TRY(mg::launch_copy_f4(pm, slot + state, (int64_t)state, st));
      M->launches += 2;
    }
    a.p = p;
    a.pm = pm;
    a.pout = pm;
    a.step = l;
    MG_TRY(do_step(M, a, pp.S_pad, st));
    M->launches += 1;
    std::swap(p, pm);
  }
  return MG_OK;
}

// Forward that keeps every state: slot j of `seg` holds p_{j-1}
// (j = 0..nt+1), the layout of one adjoint segment covering the whole run.
int run_forward_states(mg_mesh* M, const Prep& pp, int nt, float* traces, float* seg,
                       cudaStream_t st, int flags) {
  const size_t state = (size_t)M->hm.n * pp.S_pad;
  mg::DevPatches D;
  mg::ResidentShape shape;
  MG_TRY(resident_shape(M, 0, pp.S_pad, nt, D, shape, true));
  if (shape.lpr) {
    const int rc = run_forward_resident(M, pp, nt, traces, 0, nullptr, seg, D, shape, st);
    if (rc != MG_ERR_UNSUPPORTED) return rc;
  }
  MG_CU(cudaMemsetAsync(seg, 0, 2 * state * sizeof(float), st));
  mg::StepArgs a = step_args(M, pp, pp.S_pad, nt);
  a.traces = traces;
  a.hint = M->cache_hints;
  const int W = group_cols(M, 0, pp.S_pad), NG = pp.S_pad / W;
  MG_TRY(ensure_auto_entries(M, 0, W, st));
  if (graphs_on(M, flags) && nt % 2 == 0) {
    MG_TRY(ensure(M->step_base, 16));
    int32_t* base = P<int32_t>(M->step_base);
    MG_TRY(mg::launch_set_int(base, 0, st));
    M->launches += 1;
    const std::string key = key_of("fwdst", {seg, traces, a.wavelet, a.coef, a.ev.src_ptr, base},
                                   {pp.S_pad, pp.S, pp.R, nt, (int64_t)M->hm.n, W});
    return run_graph(M, key, NG * nt, st, [&](cudaStream_t cs) {
      mg::StepArgs b = a;
      b.step_base = base;
      b.cols = W;
      for (int g = 0; g < NG; ++g) {   // each shot group runs the whole history
        b.col0 = g * W;
        for (int l = 0; l < nt; ++l) {
          b.p = seg + (size_t)(l + 1) * state;
          b.pm = seg + (size_t)l * state;
          b.pout = seg + (size_t)(l + 2) * state;
          b.step = l;
          MG_TRY(do_step(M, b, pp.S_pad, cs));
        }
      }
      return MG_OK;
    });
  }
  for (int l = 0; l < nt; ++l) {
    a.p = seg + (size_t)(l + 1) * state;
    a.pm = seg + (size_t)l * state;
    a.pout = seg + (size_t)(l + 2) * state;
    a.step = l;
    MG_TRY(do_step(M, a, pp.S_pad, st));
    M->launches += 1;
  }
  return MG_OK;
}

int run_forward_single(mg_mesh* M, const Prep& pp, int nt, float* traces, cudaStream_t st) {
  const int64_t n = M->hm.n;
  MG_TRY(ensure(M->stA, n * sizeof(float)));
  MG_TRY(ensure(M->stB, n * sizeof(float)));
  mg::StepArgs a = step_args(M, pp, 1, nt);
  a.traces = traces;
  for (int s = 0; s < pp.S; ++s) {
    float* p = P<float>(M->stA);
    float* pm = P<float>(M->stB);
    MG_CU(cudaMemsetAsync(p, 0, n * sizeof(float), st));
    MG_CU(cudaMemsetAsync(pm, 0, n * sizeof(float), st));
    for (int l = 0; l < nt; ++l) {
      a.p = p;
      a.pm = pm;
      a.pout = pm;
      a.step = l;
      MG_TRY(mg::launch_step_single(a, s, st));
      M->launches += 1;
      std::swap(p, pm);
    }
  }
  return MG_OK;
}

}  // namespace

extern "C" {

const char* mg_strerror(int code) {
  if (code > 0 || code < -7) return "unknown error";
  return kErr[-code];
}

int mg_version(void) { return 100; }

int mg_mesh_create(int dim, int n_levels, const double* coords, int64_t n_nodes,
                   const int32_t* cells, int64_t n_cells,
                   const int32_t* const* cell_parent,
                   const int64_t* n_cells_per_level, const int32_t* bnd,
                   int64_t n_bnd, int bc_mode, int order, mg_mesh** out) {
  if (!out) return MG_ERR_ARG;
  *out = nullptr;
  mg_mesh* M = new mg_mesh();
  std::string msg;
  int rc = mg::build_host_mesh(dim, n_levels, coords, n_nodes, cells, n_cells, cell_parent,
                               n_cells_per_level, bnd, n_bnd, bc_mode, order, M->hm, msg);
  if (rc != MG_OK) {
    delete M;
    return rc;
  }
  if (cudaGetDevice(&M->device) != cudaSuccess) {
    cudaGetLastError();
    delete M;
    return MG_ERR_CUDA;
  }
  mg::HostMesh& h = M->hm;
  // cell -> owned boundary facets
  std::vector<int64_t> cf_ptr(h.m + 1, 0);
  for (int64_t f = 0; f < h.nb; ++f) cf_ptr[h.bnd_owner[f] + 1]++;
  for (int64_t c = 0; c < h.m; ++c) cf_ptr[c + 1] += cf_ptr[c];
  std::vector<int32_t> cf_facet(h.nb);
  {
    std::vector<int64_t> fill(cf_ptr.begin(), cf_ptr.end() - 1);
    for (int64_t f = 0; f < h.nb; ++f) cf_facet[fill[h.bnd_owner[f]]++] = (int32_t)f;
  }
  std::vector<int32_t> ell_raw(2 * h.ell.size());
  std::memcpy(ell_raw.data(), h.ell.data(), h.ell.size() * sizeof(mg::EllEntry));
  rc = MG_OK;
  if (!rc) rc = upload(M->ell, ell_raw);
  if (!rc) rc = upload(M->slice_off, h.slice_off);
  if (!rc) rc = upload(M->slice_w, h.slice_w);
  if (!rc) rc = upload(M->nc_ptr, h.nc_ptr);
  if (!rc) rc = upload(M->nc_cell, h.nc_cell);
  if (!rc) rc = upload(M->nc_w, h.nc_w);
  if (!rc) rc = upload(M->nf_ptr, h.nf_ptr);
  if (!rc) rc = upload(M->nf_cell, h.nf_cell);
  if (!rc) rc = upload(M->nf_w, h.nf_w);
  if (!rc) rc = upload(M->is_bnd, h.is_bnd_row);
  if (!rc) rc = upload(M->row_abs, h.row_abs);
  if (!rc) rc = upload(M->cells, h.cells);
  if (!rc) rc = upload(M->vol, h.cell_vol);
  if (!rc) rc = upload(M->cf_ptr, cf_ptr);
  if (!rc) rc = upload(M->cf_facet, cf_facet);
  if (!rc) rc = upload(M->bnd, h.bnd);
  if (!rc) rc = upload(M->bnd_meas, h.bnd_meas);
  M->anc.resize(h.n_levels);
  M->lvl_ptr.resize(h.n_levels);
  M->lvl_idx.resize(h.n_levels);
  // the fixed array of mg_forward_noalloc: its module is loaded and its
  // address looked up here (an allocating call anyway), so that the
  // no-allocation entry point itself reserves nothing on this device
  if (!rc) rc = mg::noalloc_prepare(M->device);
  if (rc != MG_OK) {
    mg_mesh_destroy(M);
    return rc;
  }
  // the global ELL image is on the device now; (col, val) stay on the host
  // for building row tiles on demand
  std::vector<mg::EllEntry>().swap(h.ell);
  *out = M;
  return MG_OK;
}

void mg_mesh_destroy(mg_mesh* M) {
  if (!M) return;
  DeviceGuard g(M->device);
  Buf* all[] = {&M->ell, &M->slice_off, &M->slice_w, &M->nc_ptr, &M->nc_cell, &M->nc_w,
                &M->nf_ptr, &M->nf_cell, &M->nf_w, &M->is_bnd, &M->row_abs, &M->cells,
                &M->vol, &M->cf_ptr, &M->cf_facet, &M->bnd, &M->bnd_meas, &M->ellu,
                &M->ellc, &M->flux_cell, &M->flux_ptr, &M->flux_inc, &M->flux_pinc};
  for (Buf* b : all)
    if (b->p) cudaFree(b->p);
  for (auto* v : {&M->anc, &M->lvl_ptr, &M->lvl_idx})
    for (Buf& b : *v)
      if (b.p) cudaFree(b.p);
  for (auto& kv : M->auto_ellc)
    if (kv.second.p) cudaFree(kv.second.p);
  for (Buf& b : M->flux_tab)
    if (b.p) cudaFree(b.p);
  for (auto& kv : M->tiles) {
    mg_mesh::TileTables& D = kv.second;
    for (Buf* b : {&D.ell_off, &D.ell_idx, &D.ell_val, &D.sinfo, &D.halo_off, &D.halo_cnt, &D.halo})
      if (b->p) cudaFree(b->p);
  }
  for (auto& kv : M->patches) {
    for (auto& g : kv.second.groups)
      for (Buf& b : g.second.buf)
        if (b.p) cudaFree(b.p);
  }
  mg_mesh_trim(M);
  if (M->cap) cudaStreamDestroy(M->cap);
  delete M;
}

int mg_mesh_trim(mg_mesh* M) {
  if (!M) return MG_ERR_ARG;
  DeviceGuard g(M->device);
  // graphs hold the scratch pointers: drop them with the scratch
  for (auto& kv : M->graphs) cudaGraphExecDestroy(kv.second);
  M->graphs.clear();
  Buf* all[] = {&M->eps_h, &M->wav_h, &M->wavf, &M->coef, &M->tcoef, &M->mass, &M->scal,
                &M->stA, &M->stB, &M->stC, &M->stD, &M->out_h, &M->w_h, &M->v_h, &M->g_h,
                &M->ev, &M->G, &M->ckpt, &M->seg, &M->gfine, &M->step_base, &M->tr,
                &M->trf, &M->tune_scratch, &M->xbuf};
  for (Buf* b : all) {
    if (b->p) cudaFree(b->p);
    b->p = nullptr;
    b->bytes = 0;
  }
  std::vector<mg::FluxBuffer> flux;   // a flux call of another thread may be taking or leaving them
  mg::mesh_take_scratch(M, flux);
  for (mg::FluxBuffer& b : flux) cudaFree(b.p);
  M->ev_valid = false;
  M->ck_valid = false;  M->ck_gen++;
  M->seg_full = false;
  return MG_OK;
}

int mg_mesh_set_conductivity(mg_mesh* M, const double* sigma, void* stream, int flags) {
  if (!M) return MG_ERR_ARG;
  if (flags & ~MG_HOST_PTRS) return MG_ERR_UNSUPPORTED;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  M->ck_valid = false;  M->ck_gen++;  // checkpoints of an earlier forward no longer apply
  M->seg_full = false;
  if (!sigma) {
    M->has_sigma = false;
    return MG_OK;
  }
  const size_t bytes = (size_t)M->hm.m * sizeof(double);
  if (flags & MG_HOST_PTRS)
    for (int64_t e = 0; e < M->hm.m; ++e)
      if (!(sigma[e] >= 0.0) || !std::isfinite(sigma[e])) return MG_ERR_ARG;
  MG_TRY(ensure(M->sigma, bytes));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  MG_CU(cudaMemcpyAsync(M->sigma.p, sigma, bytes,
                        (flags & MG_HOST_PTRS) ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                        st));
  if (flags & MG_HOST_PTRS) MG_CU(cudaStreamSynchronize(st));
  M->has_sigma = true;
  return MG_OK;
}

int mg_prolong(mg_mesh* M, int level, const double* v, const double* base, double* out,
               void* stream, int flags) {
  if (!M || !v || !out || level < 0 || level >= M->hm.n_levels) return MG_ERR_ARG;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  MG_TRY(ensure_level(M, level));
  const int64_t m = M->hm.m;
  const void* dv;
  MG_TRY(stage_in(M->v_h, v, M->hm.n_cells_level[level] * sizeof(double), flags, st, &dv));
  const void* db = nullptr;
  if (base) MG_TRY(stage_in(M->eps_h, base, m * sizeof(double), flags, st, &db));
  double* o = out;
  if (flags & MG_HOST_PTRS) {
    MG_TRY(ensure(M->g_h, m * sizeof(double)));
    o = P<double>(M->g_h);
  }
  MG_TRY(mg::launch_prolong(m, P<int32_t>(M->anc[level]), static_cast<const double*>(dv),
                            static_cast<const double*>(db), o, st));
  M->launches += 1;
  return (flags & MG_HOST_PTRS) ? deliver(M->g_h, out, m * sizeof(double), flags, st) : MG_OK;
}

static bool tuning_ok(int batch, int tile_rows, int src_tile) {
  if (batch != -1 && batch != 1 && batch != 2 && batch != 4) return false;
  if (tile_rows != -1 && (tile_rows < 0 || tile_rows % mg::kSliceH != 0 || tile_rows > 8192))
    return false;
  if (src_tile != -1 && src_tile != 4 && src_tile != 8 && src_tile != 16 && src_tile != 32 &&
      src_tile != 64)
    return false;
  return true;
}

static void drop_graphs(mg_mesh* M) {
  DeviceGuard g(M->device);
  for (auto& kv : M->graphs) cudaGraphExecDestroy(kv.second);
  M->graphs.clear();
}

// A setter of one launch-shape field: another value than the one on the handle
// asks for the shape, the same one asks for nothing.
static void set_field(mg_mesh::Tuning& t, int mg_mesh::Tuning::* field, int value) {
  if (t.*field == value) return;
  t.*field = value;
  t.path = MG_PATH_SHAPE;
}

static void apply_tuning(mg_mesh::Tuning& t, int batch, int tile_rows, int src_tile) {
  if (batch != -1 || tile_rows != -1 || src_tile != -1) t.path = MG_PATH_SHAPE;
  if (batch != -1) t.batch = batch;
  if (tile_rows != -1) t.tile_rows = tile_rows;
  if (src_tile != -1) t.src_tile = src_tile;
}

int mg_mesh_set_tuning(mg_mesh* M, int chunk, int batch, int tile_rows, int src_tile) {
  if (!M) return MG_ERR_ARG;
  if (chunk != -1 && (chunk < 0 || chunk == 1 || chunk % 2 != 0 || chunk > 4096)) return MG_ERR_ARG;
  if (!tuning_ok(batch, tile_rows, src_tile)) return MG_ERR_ARG;
  drop_graphs(M);
  if (chunk != -1) M->chunk = chunk;
  for (auto& t : M->tune) apply_tuning(t, batch, tile_rows, src_tile);
  return MG_OK;
}

int mg_mesh_set_kernel_tuning(mg_mesh* M, int kind, int batch, int tile_rows, int src_tile) {
  if (!M || kind < 0 || kind > 2 || !tuning_ok(batch, tile_rows, src_tile)) return MG_ERR_ARG;
  drop_graphs(M);
  apply_tuning(M->tune[kind], batch, tile_rows, src_tile);
  return MG_OK;
}

int mg_mesh_set_shot_groups(mg_mesh* M, int kind, int groups) {
  if (!M || kind < -1 || kind > 2 || (groups != 1 && groups != 2 && groups != 4 && groups != 8))
    return MG_ERR_ARG;
  drop_graphs(M);
  for (int k = 0; k < 3; ++k)
    if (kind == -1 || kind == k) set_field(M->tune[k], &mg_mesh::Tuning::groups, groups);
  return MG_OK;
}

int mg_mesh_set_cache_hints(mg_mesh* M, int on) {
  if (!M || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  M->cache_hints = on;
  return MG_OK;
}

int mg_mesh_set_uniform_ell(mg_mesh* M, int on) {
  if (!M || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  if (!on) {
    M->uniform_ell = false;
    return MG_OK;
  }
  if (!M->ellu.p) {
    const mg::HostMesh& h = M->hm;
    int w = 0;
    for (int32_t x : h.slice_w) w = std::max(w, (int)x);
    const size_t total = (size_t)h.n_slices * w * mg::kSliceH;
    const size_t stored = h.slice_off.empty() ? 0 : (size_t)h.slice_off.back();
    if (stored == 0 || total > 2 * stored) return MG_ERR_UNSUPPORTED;   // padding would double K
    DeviceGuard g(M->device);
    if (!g.ok) return MG_ERR_CUDA;
    // the host copy of the entries is released after upload: read them back
    std::vector<mg::EllEntry> ell(stored);
    if (cudaMemcpy(ell.data(), M->ell.p, stored * sizeof(mg::EllEntry),
                   cudaMemcpyDeviceToHost) != cudaSuccess)
      return MG_ERR_CUDA;
    std::vector<int32_t> u(2 * total);
    for (int64_t s = 0; s < h.n_slices; ++s)
      for (int k = 0; k < w; ++k)
        for (int r = 0; r < mg::kSliceH; ++r) {
          const size_t o = ((size_t)s * w + k) * mg::kSliceH + r;
          if (k < h.slice_w[s]) {
            const mg::EllEntry& e = ell[h.slice_off[s] + (size_t)k * mg::kSliceH + r];
            std::memcpy(&u[2 * o], &e, sizeof(e));
          } else {
            const float zero = 0.0f;
            u[2 * o] = (int32_t)(s * mg::kSliceH + r);
            std::memcpy(&u[2 * o + 1], &zero, sizeof(zero));
          }
        }
    MG_TRY(upload(M->ellu, u));
    M->wu = w;
  }
  M->uniform_ell = true;
  return MG_OK;
}

int mg_mesh_set_chunked_ell(mg_mesh* M, int chunk) {
  if (!M || (chunk != 0 && chunk != 2 && chunk != 4 && chunk != 8 && chunk != 16))
    return MG_ERR_ARG;
  drop_graphs(M);
  if (!chunk) {
    M->chunked_ell = false;
    return MG_OK;
  }
  if (!M->ellc.p || M->cchunk != chunk) {
    const mg::HostMesh& h = M->hm;
    int w = 0;
    for (int32_t x : h.slice_w) w = std::max(w, (int)x);
    const size_t stored = h.slice_off.empty() ? 0 : (size_t)h.slice_off.back();
    if (stored == 0) return MG_ERR_UNSUPPORTED;
    const int64_t nch = (w + chunk - 1) / chunk;
    const int64_t stride = nch * mg::kSliceH * chunk;
    const size_t total = (size_t)h.n_slices * stride;
    DeviceGuard g(M->device);
    if (!g.ok) return MG_ERR_CUDA;
    // the host copy of the entries is released after upload: read them back
    std::vector<mg::EllEntry> ell(stored);
    if (cudaMemcpy(ell.data(), M->ell.p, stored * sizeof(mg::EllEntry),
                   cudaMemcpyDeviceToHost) != cudaSuccess)
      return MG_ERR_CUDA;
    // slots past a slice's width are never read: zero-filled
    std::vector<int32_t> c(2 * total, 0);
    for (int64_t s = 0; s < h.n_slices; ++s)
      for (int k = 0; k < h.slice_w[s]; ++k)
        for (int r = 0; r < mg::kSliceH; ++r) {
          const size_t o = (size_t)s * stride + ((size_t)(k / chunk) * mg::kSliceH + r) * chunk +
                           k % chunk;
          std::memcpy(&c[2 * o], &ell[h.slice_off[s] + (size_t)k * mg::kSliceH + r],
                      sizeof(mg::EllEntry));
        }
    if (M->ellc.p) {
      cudaFree(M->ellc.p);
      M->ellc = Buf{};
    }
    MG_TRY(upload(M->ellc, c));
    M->cchunk = chunk;
    M->cstride = stride;
  }
  M->chunked_ell = true;
  return MG_OK;
}

int mg_mesh_set_dependent_launch(mg_mesh* M, int on) {
  if (!M || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  M->dep_launch = on;
  return MG_OK;
}

int mg_mesh_set_bulk_copies(mg_mesh* M, int on) {
  if (!M || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  set_field(M->tune[0], &mg_mesh::Tuning::bulk, on);
  return MG_OK;
}

int mg_mesh_device_status(mg_mesh* M) {
  if (!M) return MG_ERR_ARG;
  if (!M->errbuf.p) return MG_OK;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  int word = 0;
  if (cudaMemcpy(&word, M->errbuf.p, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemset(M->errbuf.p, 0, sizeof(int)) != cudaSuccess)
    return MG_ERR_CUDA;
  return word == 0 ? MG_OK : word == 1 ? MG_ERR_TIMEOUT : MG_ERR_ARG;
}

int mg_mesh_set_gather_ring(mg_mesh* M, int kind, int depth) {
  if (!M || kind < -1 || kind > 2 || (depth != 0 && depth != 4 && depth != 8)) return MG_ERR_ARG;
  drop_graphs(M);
  for (int k = 0; k < 3; ++k)
    if (kind == -1 || kind == k) set_field(M->tune[k], &mg_mesh::Tuning::ring, depth);
  return MG_OK;
}

int mg_mesh_set_row_sweep(mg_mesh* M, int blocks) {
  if (!M || blocks < 0 || blocks > 65536) return MG_ERR_ARG;
  drop_graphs(M);
  set_field(M->tune[0], &mg_mesh::Tuning::sweep, blocks);
  return MG_OK;
}

int mg_mesh_get_row_sweep(const mg_mesh* M) { return M ? M->tune[0].sweep : MG_ERR_ARG; }

int mg_mesh_set_late_prefetch(mg_mesh* M, int kind, int level) {
  if (!M || kind < -1 || kind > 2 || level < 0 || level > 3 || (level == 3 && kind != 0))
    return MG_ERR_ARG;
  drop_graphs(M);
  for (int k = 0; k < 3; ++k)
    if (kind == -1 || kind == k) M->tune[k].prefetch = level;
  return MG_OK;
}

int mg_mesh_set_wide_lanes(mg_mesh* M, int on) {
  if (!M || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  M->tune[0].wide = on;
  return MG_OK;
}

int mg_mesh_get_wide_lanes(const mg_mesh* M) { return M ? M->tune[0].wide : MG_ERR_ARG; }

int mg_mesh_get_late_prefetch(const mg_mesh* M, int32_t* out) {
  if (!M || !out) return MG_ERR_ARG;
  for (int k = 0; k < 3; ++k) out[k] = M->tune[k].prefetch;
  return MG_OK;
}

int mg_mesh_set_l1_streaming(mg_mesh* M, int kind, int on) {
  if (!M || kind < -1 || kind > 2 || (on != 0 && on != 1)) return MG_ERR_ARG;
  drop_graphs(M);
  for (int k = 0; k < 3; ++k)
    if (kind == -1 || kind == k) M->tune[k].stream = on;
  return MG_OK;
}

int mg_mesh_get_l1_streaming(const mg_mesh* M, int32_t* out) {
  if (!M || !out) return MG_ERR_ARG;
  for (int k = 0; k < 3; ++k) out[k] = M->tune[k].stream;
  return MG_OK;
}

int mg_mesh_set_tma_tiles(mg_mesh* M, int rows) {
  if (!M || rows < 0 || rows > 1024 || rows % mg::kSliceH) return MG_ERR_ARG;
  drop_graphs(M);
  set_field(M->tune[0], &mg_mesh::Tuning::tma, rows);
  return MG_OK;
}

int mg_mesh_get_tma_tiles(const mg_mesh* M) { return M ? M->tune[0].tma : MG_ERR_ARG; }

int64_t mg_mesh_checkpoint_generation(const mg_mesh* M) { return M ? M->ck_gen : MG_ERR_ARG; }

int mg_mesh_set_persistent(mg_mesh* M, int steps, long long wait_cycles, int extra_arrivals) {
  if (!M || steps < 1 || steps > (1 << 20) || wait_cycles < 1000 || extra_arrivals < 0 ||
      extra_arrivals > (1 << 20))
    return MG_ERR_ARG;
  M->persist_steps = steps;
  M->persist_budget = wait_cycles;
  M->persist_extra = extra_arrivals;
  return MG_OK;
}

int mg_mesh_get_gather_ring(const mg_mesh* M, int32_t* out) {
  if (!M || !out) return MG_ERR_ARG;
  for (int k = 0; k < 3; ++k) out[k] = M->tune[k].ring;
  return MG_OK;
}

int mg_mesh_set_min_blocks(mg_mesh* M, int min_blocks) {
  if (!M || (min_blocks != 0 && min_blocks != 5)) return MG_ERR_ARG;
  drop_graphs(M);
  set_field(M->tune[0], &mg_mesh::Tuning::min_blocks, min_blocks);
  return MG_OK;
}

int mg_mesh_set_kernel_min_blocks(mg_mesh* M, int kind, int min_blocks) {
  if (!M || kind < 0 || kind > 2 ||
      (min_blocks != 0 && min_blocks != 5 && (min_blocks != 6 || kind != 2)))
    return MG_ERR_ARG;
  drop_graphs(M);
  set_field(M->tune[kind], &mg_mesh::Tuning::min_blocks, min_blocks);
  return MG_OK;
}

int mg_mesh_set_kernel_path(mg_mesh* M, int kind, int path) {
  if (!M || kind < -1 || kind > 2 || path < MG_PATH_AUTO || path > MG_PATH_ROWS)
    return MG_ERR_ARG;
  drop_graphs(M);
  for (int k = 0; k < 3; ++k)
    if (kind == -1 || kind == k) M->tune[k].path = path;
  return MG_OK;
}

int mg_mesh_get_kernel_path(const mg_mesh* M, int32_t* out) {
  if (!M || !out) return MG_ERR_ARG;
  for (int k = 0; k < 3; ++k) out[k] = M->tune[k].path;
  return MG_OK;
}

int mg_mesh_get_tuning(const mg_mesh* M, int32_t* out) {
  if (!M || !out) return MG_ERR_ARG;
  out[0] = M->chunk;
  for (int k = 0; k < 3; ++k) {
    out[1 + 5 * k] = M->tune[k].batch;
    out[2 + 5 * k] = M->tune[k].tile_rows;
    out[3 + 5 * k] = M->tune[k].src_tile;
    out[4 + 5 * k] = M->tune[k].groups;
    out[5 + 5 * k] = M->tune[k].min_blocks;
  }
  out[16] = M->tune[0].bulk;
  return MG_OK;
}

int mg_mesh_get_info(const mg_mesh* M, mg_mesh_info_t* info) {
  if (!M || !info) return MG_ERR_ARG;
  const mg::HostMesh& h = M->hm;
  info->dim = h.dim;
  info->n_levels = h.n_levels;
  info->n_nodes = h.n;
  info->n_cells = h.m;
  info->n_bnd = h.nb;
  info->nnz = h.rowptr.empty() ? 0 : h.rowptr.back();
  info->ell_entries = h.slice_off.empty() ? 0 : h.slice_off.back();
  info->slice_height = mg::kSliceH;
  info->max_row_nnz = h.max_row_nnz;
  int64_t bytes = 0;
  const Buf* all[] = {&M->ell, &M->slice_off, &M->slice_w, &M->nc_ptr, &M->nc_cell, &M->nc_w,
                      &M->nf_ptr, &M->nf_cell, &M->nf_w, &M->is_bnd, &M->row_abs, &M->cells,
                      &M->vol, &M->cf_ptr, &M->cf_facet, &M->bnd, &M->bnd_meas, &M->eps_h,
                      &M->wav_h, &M->wavf, &M->coef, &M->tcoef, &M->mass, &M->scal, &M->stA,
                      &M->stB, &M->stC, &M->stD, &M->out_h, &M->w_h, &M->v_h, &M->g_h, &M->ev,
                      &M->G, &M->ckpt, &M->seg, &M->gfine, &M->step_base, &M->tr, &M->trf,
                      &M->xbuf};
  for (const Buf* b : all) bytes += (int64_t)b->bytes;
  for (const auto& kv : M->auto_ellc) bytes += (int64_t)kv.second.bytes;
  for (const auto& kv : M->patches)
    for (const auto& g : kv.second.groups)
      for (const Buf& b : g.second.buf) bytes += (int64_t)b.bytes;
  {
    std::lock_guard<std::mutex> lock(M->flux_mu);
    for (const Buf* b : {&M->flux_cell, &M->flux_ptr, &M->flux_inc, &M->flux_pinc})
      bytes += (int64_t)b->bytes;
    for (const Buf& b : M->flux_tab) bytes += (int64_t)b.bytes;
    for (const mg::FluxBuffer& b : M->flux_scratch) bytes += (int64_t)b.bytes;
  }
  info->device_bytes = bytes;
  return MG_OK;
}

int mg_mesh_get_permutation(const mg_mesh* M, int32_t* perm) {
  if (!M || !perm) return MG_ERR_ARG;
  std::copy(M->hm.perm.begin(), M->hm.perm.end(), perm);
  return MG_OK;
}

int64_t mg_launch_count(const mg_mesh* M) { return M ? M->launches : 0; }

int mg_cfl_dt(mg_mesh* M, const double* eps, int flags, void* stream, double* dt_out) {
  if (!M || !eps || !dt_out) return MG_ERR_ARG;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const void* d;
  MG_TRY(stage_in(M->eps_h, eps, M->hm.m * sizeof(double), flags, st, &d));
  double lam = 0.0;
  MG_TRY(cfl_lambda(M, static_cast<const double*>(d), st, &lam));
  if (!(lam > 0.0) || !std::isfinite(lam)) return MG_ERR_ARG;
  *dt_out = 2.0 / std::sqrt(lam);
  return MG_OK;
}

int mg_forward(mg_mesh* M, const double* eps, const mg_shots* shots, const double* wavelet,
               double dt, int nt, float* traces, int ckpt_every, void* stream, int flags) {
  if (!M || !traces) return MG_ERR_ARG;
  if (flags & ~(kCommonFlags | MG_SINGLE_SOURCE | MG_PERSISTENT | MG_KEEP_CHECKPOINTS |
                MG_KEEP_STATES))
    return MG_ERR_UNSUPPORTED;
  if ((flags & MG_KEEP_CHECKPOINTS) && (ckpt_every < 1 || (flags & MG_SINGLE_SOURCE)))
    return MG_ERR_ARG;
  if ((flags & MG_KEEP_STATES) && (flags & (MG_KEEP_CHECKPOINTS | MG_SINGLE_SOURCE)))
    return MG_ERR_ARG;
  if ((flags & MG_PERSISTENT) && (flags & (MG_SINGLE_SOURCE | MG_KEEP_STATES)))
    return MG_ERR_UNSUPPORTED;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Prep pp;
  MG_TRY(prepare(M, eps, shots, wavelet, dt, nt, flags, st, pp));
  const size_t tbytes = (size_t)pp.R * nt * sizeof(float);
  MG_TRY(ensure(M->tr, tbytes));
  float* tr = P<float>(M->tr);
  if (flags & MG_SINGLE_SOURCE) {
    MG_TRY(run_forward_single(M, pp, nt, tr, st));
  } else if (flags & MG_KEEP_STATES) {
    M->ck_valid = false;  M->ck_gen++;
    M->seg_full = false;
    const size_t state = (size_t)M->hm.n * pp.S_pad;
    MG_TRY(ensure(M->seg, (size_t)(nt + 2) * state * sizeof(float)));
    MG_TRY(run_forward_states(M, pp, nt, tr, P<float>(M->seg), st, flags));
    MG_TRY(note_kept(M, st));
    M->ck_valid = true;  M->ck_gen++;
    M->seg_full = true;
    M->ck_every = nt;
    M->ck_nt = nt;
    M->ck_S_pad = pp.S_pad;
    M->ck_nshots = pp.S;
    M->ck_dt = dt;
    M->ck_ev_gen = M->ev_gen;
  } else {
    float* ck = nullptr;
    M->ck_valid = false;  M->ck_gen++;
    M->seg_full = false;
    if (flags & MG_KEEP_CHECKPOINTS) {
      const int nck = (nt + ckpt_every - 1) / ckpt_every;
      MG_TRY(ensure(M->ckpt, (size_t)nck * 2 * M->hm.n * pp.S_pad * sizeof(float)));
      ck = P<float>(M->ckpt);
    }
    MG_TRY(run_forward(M, pp, nt, tr, ckpt_every, ck, st, flags));
    // the barrier waits are bounded: read (and clear) the status word
    if (flags & MG_PERSISTENT) MG_TRY(persist_status(M, st));
    if (ck) {
      MG_TRY(note_kept(M, st));
      M->ck_valid = true;  M->ck_gen++;
      M->ck_every = ckpt_every;
      M->ck_nt = nt;
      M->ck_S_pad = pp.S_pad;
      M->ck_nshots = pp.S;
      M->ck_dt = dt;
      M->ck_ev_gen = M->ev_gen;
    }
  }
  return deliver(M->tr, traces, tbytes, flags, st);
}

int mg_jacobian_apply(mg_mesh* M, int level, const double* eps, const mg_shots* shots,
                      const double* wavelet, double dt, int nt, const double* v, float* jv,
                      void* stream, int flags) {
  if (!M || !v || !jv) return MG_ERR_ARG;
  if (level < 0 || level >= M->hm.n_levels) return MG_ERR_ARG;
  if (flags & ~(kCommonFlags | MG_REUSE_CHECKPOINTS)) return MG_ERR_UNSUPPORTED;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Prep pp;
  MG_TRY(prepare(M, eps, shots, wavelet, dt, nt, flags, st, pp));
  MG_TRY(ensure_level(M, level));
  const void* d;
  MG_TRY(stage_in(M->v_h, v, M->hm.n_cells_level[level] * sizeof(double), flags, st, &d));
  MG_TRY(ensure(M->tcoef, M->hm.n * sizeof(float2)));
  mg::TangentCoefArgs tca;
  tca.c = coef_args(M, pp.eps, dt);
  tca.v = static_cast<const double*>(d);
  tca.anc = P<int32_t>(M->anc[level]);
  tca.tcoef = P<float2>(M->tcoef);
  MG_TRY(mg::launch_tangent_coefs(tca, st));
  M->launches += 1;
  const size_t tbytes = (size_t)pp.R * nt * sizeof(float);
  MG_TRY(ensure(M->tr, tbytes));
  float* tr = P<float>(M->tr);
  const int64_t n = M->hm.n;
  const size_t state = (size_t)n * pp.S_pad;
  if (!(flags & MG_REUSE_CHECKPOINTS)) {
    mg::DevPatches D;
    mg::ResidentShape shape;
    MG_TRY(resident_shape(M, 1, pp.S_pad, nt, D, shape));
    if (shape.lpr) {
      const int rc = run_tangent_resident(M, pp, nt, nullptr, tr, nullptr, D, shape, st);
      if (rc == MG_OK) return deliver(M->tr, jv, tbytes, flags, st);
      if (rc != MG_ERR_UNSUPPORTED) return rc;
    }
  }
  MG_TRY(ensure_auto_entries(M, 1, group_cols(M, 1, pp.S_pad), st));
  Buf* bufs[] = {&M->stA, &M->stB, &M->stC, &M->stD};
  for (Buf* b : bufs) {
    MG_TRY(ensure(*b, state * sizeof(float)));
    MG_CU(cudaMemsetAsync(b->p, 0, state * sizeof(float), st));
  }
  float *p = P<float>(M->stA), *pm = P<float>(M->stB), *q = P<float>(M->stC),
        *qm = P<float>(M->stD);
  mg::TangentArgs a{};
  a.f = step_args(M, pp, pp.S_pad, nt);
  a.tcoef = P<const float2>(M->tcoef);
  a.dtraces = tr;
  if (flags & MG_REUSE_CHECKPOINTS) {
    // the states kept by the last mg_forward (MG_KEEP_STATES) are read: slot
    // j of the segment buffer holds p_{j-1}; only dp is advanced
    const bool kept = M->ck_valid && M->seg_full && M->ck_every == nt && M->ck_nt == nt &&
                      M->ck_S_pad == pp.S_pad && M->ck_nshots == pp.S && M->ck_dt == dt &&
                      M->ck_ev_gen == M->ev_gen;
    if (!kept) return MG_ERR_ARG;
    float* seg = P<float>(M->seg);
    const mg_mesh::Tuning t = in_force(M, 1);
    a.f.batch = t.batch;
    a.f.ring = t.ring;
    a.f.stream = t.stream;
    a.f.pdl = M->dep_launch;
    a.f.hint = M->cache_hints;
    const int W = group_cols(M, 1, pp.S_pad), NG = pp.S_pad / W;
    int32_t* base = nullptr;
    const bool graph = graphs_on(M, flags);
    if (graph) {
      MG_TRY(ensure(M->step_base, 16));
      base = P<int32_t>(M->step_base);
      MG_TRY(mg::launch_set_int(base, 0, st));
      M->launches += 1;
    }
    auto record = [&](cudaStream_t cs) -> int {
      mg::TangentArgs b = a;
      b.f.step_base = base;
      b.f.cols = W;
      for (int g = 0; g < NG; ++g) {   // each shot group runs the whole history
        b.f.col0 = g * W;
        float *u = q, *z = qm;
        for (int j = 0; j < nt; ++j) {
          b.f.p = seg + (size_t)(j + 1) * state;
          b.f.pm = seg + (size_t)j * state;
          b.pk1 = seg + (size_t)(j + 2) * state;
          b.q = u;
          b.qm = z;
          b.f.step = j;
          MG_TRY(mg::launch_tangent_kept(b, pp.S_pad, cs));
          std::swap(u, z);
        }
      }
      return MG_OK;
    };
    if (graph) {
      const std::string key = key_of("tankept", {seg, q, qm, tr, a.f.coef, a.tcoef,
                                                 a.f.ev.rec_ptr, base},
                                     {pp.S_pad, pp.S, pp.R, nt, n, W});
      MG_TRY(run_graph(M, key, NG * nt, st, record));
    } else {
      MG_TRY(record(st));
      M->launches += (int64_t)NG * nt;
    }
    MG_TRY(poison(M, tr, pp.R * nt, true, st));
    return deliver(M->tr, jv, tbytes, flags, st);
  }
  int l = 0;
  const int C = M->chunk;
  if (graphs_on(M, flags) && nt >= C) {
    MG_TRY(ensure(M->step_base, 16));
    int32_t* base = P<int32_t>(M->step_base);
    MG_TRY(mg::launch_set_int(base, 0, st));
    M->launches += 1;
    const int W = group_cols(M, 1, pp.S_pad), NG = pp.S_pad / W;
    const std::string key = key_of("tan", {p, pm, q, qm, tr, a.f.wavelet, a.f.coef, a.tcoef,
                                           a.f.ev.src_ptr, base},
                                   {pp.S_pad, pp.S, pp.R, nt, C, n, W});
    for (; l + C <= nt; l += C) {
      MG_TRY(run_graph(M, key, NG * C + 1, st, [&](cudaStream_t cs) {
        mg::TangentArgs b = a;
        b.f.step_base = base;
        b.f.cols = W;
        for (int g = 0; g < NG; ++g) {   // each shot group runs the whole chunk
          b.f.col0 = g * W;
          float *x = p, *y = pm, *u = q, *z = qm;
          for (int j = 0; j < C; ++j) {
            b.f.p = x;
            b.f.pm = y;
            b.f.pout = y;
            b.q = u;
            b.qm = z;
            b.f.step = j;
            MG_TRY(do_tangent(M, b, pp.S_pad, cs));
            std::swap(x, y);
            std::swap(u, z);
          }
        }
        return mg::launch_add_int(base, C, cs);
      }));
    }
  }
  for (; l < nt; ++l) {
    a.f.p = p;
    a.f.pm = pm;
    a.f.pout = pm;
    a.q = q;
    a.qm = qm;
    a.f.step = l;
    MG_TRY(do_tangent(M, a, pp.S_pad, st));
    M->launches += 1;
    std::swap(p, pm);
    std::swap(q, qm);
  }
  return deliver(M->tr, jv, tbytes, flags, st);
}

int mg_forward_jacobian_apply(mg_mesh* M, int level, const double* eps, const mg_shots* shots,
                              const double* wavelet, double dt, int nt, const double* v,
                              float* traces, float* jv, void* stream, int flags) {
  if (!M || !v || !jv || !traces) return MG_ERR_ARG;
  if (level < 0 || level >= M->hm.n_levels) return MG_ERR_ARG;
  if (flags & ~(kCommonFlags | MG_KEEP_STATES | MG_PERSISTENT)) return MG_ERR_UNSUPPORTED;
  if ((flags & MG_PERSISTENT) && !(flags & MG_KEEP_STATES)) return MG_ERR_UNSUPPORTED;
  DeviceGuard g(M->device);
  if (!g.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Prep pp;
  MG_TRY(prepare(M, eps, shots, wavelet, dt, nt, flags, st, pp));
  MG_TRY(ensure_level(M, level));
  const void* d;
  MG_TRY(stage_in(M->v_h, v, M->hm.n_cells_level[level] * sizeof(double), flags, st, &d));
  MG_TRY(ensure(M->tcoef, M->hm.n * sizeof(float2)));
  mg::TangentCoefArgs tca;
  tca.c = coef_args(M, pp.eps, dt);
  tca.v = static_cast<const double*>(d);
  tca.anc = P<int32_t>(M->anc[level]);
  tca.tcoef = P<float2>(M->tcoef);
  MG_TRY(mg::launch_tangent_coefs(tca, st));
  M->launches += 1;
  const size_t tbytes = (size_t)pp.R * nt * sizeof(float);
  MG_TRY(ensure(M->tr, tbytes));
  MG_TRY(ensure(M->trf, tbytes));
  float* tr = P<float>(M->tr);
  float* trf = P<float>(M->trf);
  const int64_t n = M->hm.n;
  const size_t state = (size_t)n * pp.S_pad;
  const bool keep = flags & MG_KEEP_STATES;
  M->ck_valid = false;  M->ck_gen++;
  M->seg_full = false;
  float *p = nullptr, *pm = nullptr, *seg = nullptr;
  if (keep) {
    MG_TRY(ensure(M->seg, (size_t)(nt + 2) * state * sizeof(float)));
    seg = P<float>(M->seg);
    MG_CU(cudaMemsetAsync(seg, 0, 2 * state * sizeof(float), st));
  }
  auto finish = [&]() -> int {
    if (keep) {
      MG_TRY(note_kept(M, st));
      M->ck_valid = true;  M->ck_gen++;
      M->seg_full = true;
      M->ck_every = nt;
      M->ck_nt = nt;
      M->ck_S_pad = pp.S_pad;
      M->ck_nshots = pp.S;
      M->ck_dt = dt;
      M->ck_ev_gen = M->ev_gen;
    }
    MG_TRY(deliver(M->trf, traces, tbytes, flags, st));
    return deliver(M->tr, jv, tbytes, flags, st);
  };
  if (!(flags & MG_PERSISTENT)) {
    mg::DevPatches D;
    mg::ResidentShape shape;
    MG_TRY(resident_shape(M, 1, pp.S_pad, nt, D, shape, keep));
    if (shape.lpr) {
      const int rc = run_tangent_resident(M, pp, nt, trf, tr, keep ? seg + 2 * state : nullptr, D,
                                          shape, st);
      if (rc == MG_OK) return finish();
      if (rc != MG_ERR_UNSUPPORTED) return rc;
    }
  }
  MG_TRY(ensure_auto_entries(M, 1, group_cols(M, 1, pp.S_pad), st));
  if (!keep) {
    for (Buf* b : {&M->stA, &M->stB}) {
      MG_TRY(ensure(*b, state * sizeof(float)));
      MG_CU(cudaMemsetAsync(b->p, 0, state * sizeof(float), st));
    }
    p = P<float>(M->stA);
    pm = P<float>(M->stB);
  }
  for (Buf* b : {&M->stC, &M->stD}) {
    MG_TRY(ensure(*b, state * sizeof(float)));
    MG_CU(cudaMemsetAsync(b->p, 0, state * sizeof(float), st));
  }
  float *q = P<float>(M->stC), *qm = P<float>(M->stD);
  mg::TangentArgs a{};
  a.f = step_args(M, pp, pp.S_pad, nt);
  a.f.traces = trf;
  a.f.batch = in_force(M, 1).batch;   // MG_PERSISTENT
  a.f.hint = keep ? M->cache_hints : 0;   // p_{l-1} is last read here only when kept
  a.tcoef = P<const float2>(M->tcoef);
  a.dtraces = tr;
  const int W = group_cols(M, 1, pp.S_pad), NG = pp.S_pad / W;
  int32_t* base = nullptr;
  const bool graph = graphs_on(M, flags);
  if (graph) {
    MG_TRY(ensure(M->step_base, 16));
    base = P<int32_t>(M->step_base);
    MG_TRY(mg::launch_set_int(base, 0, st));
    M->launches += 1;
  }
  auto record = [&](cudaStream_t cs) -> int {
    mg::TangentArgs b = a;
    b.f.step_base = base;
    b.f.cols = W;
    for (int g = 0; g < NG; ++g) {   // each shot group runs the whole history
      b.f.col0 = g * W;
      float *x = p, *y = pm, *u = q, *z = qm;
      for (int j = 0; j < nt; ++j) {
        if (keep) {
          b.f.p = seg + (size_t)(j + 1) * state;
          b.f.pm = seg + (size_t)j * state;
          b.f.pout = seg + (size_t)(j + 2) * state;
        } else {
          b.f.p = x;
          b.f.pm = y;
          b.f.pout = y;
          std::swap(x, y);
        }
        b.q = u;
        b.qm = z;
        b.f.step = j;
        row_tangent_args(M, W, b);
        MG_TRY(mg::launch_tangent(b, pp.S_pad, cs));
        std::swap(u, z);
      }
    }
    return MG_OK;
  };
  if (flags & MG_PERSISTENT) {
    // each shot group: cooperative launches of up to persist_steps steps
    // with grid barriers between the steps, writing the kept history
    mg::PersistArgs pa{};
    MG_TRY(persist_args(M, st, seg, state, pa));
    for (int g = 0; g < NG; ++g) {
      mg::TangentArgs b = a;
      b.f.step_base = nullptr;
      b.f.col0 = g * W;
      b.f.cols = W;
      float *u = q, *z = qm;
      for (int l = 0; l < nt;) {
        pa.steps = std::min(nt - l, M->persist_steps);
        b.f.step = l;
        b.q = u;
        b.qm = z;
        MG_TRY(mg::launch_tangent_persist(b, pp.S_pad, pa, st));
        M->launches += 1;
        if (pa.steps % 2) std::swap(u, z);
        l += pa.steps;
      }
    }
    MG_TRY(persist_status(M, st));
  } else if (graph) {
    const std::string key = key_of("fwdtan", {seg, p, pm, q, qm, tr, trf, a.f.wavelet, a.f.coef,
                                              a.tcoef, a.f.ev.src_ptr, base},
                                   {pp.S_pad, pp.S, pp.R, nt, n, W, keep ? 1 : 0});
    MG_TRY(run_graph(M, key, NG * nt, st, record));
  } else {
    MG_TRY(record(st));
    M->launches += (int64_t)NG * nt;
  }
  return finish();
}

int mg_jacobian_T_apply(mg_mesh* M, int level, const double* eps, const mg_shots* shots,
                        const double* wavelet, double dt, int nt, const float* w, double* g,
                        int ckpt_every, void* stream, int flags) {
  if (!M || !w || !g || ckpt_every < 1) return MG_ERR_ARG;
  if (level < 0 || level >= M->hm.n_levels) return MG_ERR_ARG;
  if (flags & ~(kCommonFlags | MG_REUSE_CHECKPOINTS | MG_PERSISTENT)) return MG_ERR_UNSUPPORTED;
  DeviceGuard guard(M->device);
  if (!guard.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Prep pp;
  MG_TRY(prepare(M, eps, shots, wavelet, dt, nt, flags, st, pp));
  MG_TRY(ensure_level(M, level));
  const int64_t n = M->hm.n;
  const size_t state = (size_t)n * pp.S_pad;
  // trace weights into the handle's buffer (stable address for the graphs)
  const size_t wbytes = (size_t)pp.R * nt * sizeof(float);
  MG_TRY(ensure(M->w_h, wbytes));
  MG_CU(cudaMemcpyAsync(M->w_h.p, w, wbytes,
                        (flags & MG_HOST_PTRS) ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                        st));
  const float* wd = P<const float>(M->w_h);
  // checkpoints
  const bool reuse = (flags & MG_REUSE_CHECKPOINTS) && M->ck_valid && M->ck_every == ckpt_every &&
                     M->ck_nt == nt && M->ck_S_pad == pp.S_pad && M->ck_nshots == pp.S &&
                     M->ck_dt == dt && M->ck_ev_gen == M->ev_gen;
  if ((flags & MG_REUSE_CHECKPOINTS) && !reuse) return MG_ERR_ARG;
  // every state of the forward kept (MG_KEEP_STATES): one segment, no recompute
  const bool states = reuse && M->seg_full && ckpt_every == nt;
  // several reverse steps per cooperative launch: on the kept history only
  if ((flags & MG_PERSISTENT) && !states) return MG_ERR_UNSUPPORTED;
  if (!states) M->seg_full = false;   // the segment buffer is rewritten below
  const int nck = (nt + ckpt_every - 1) / ckpt_every;
  if (!reuse) {
    M->ck_valid = false;  M->ck_gen++;
    MG_TRY(ensure(M->ckpt, (size_t)nck * 2 * state * sizeof(float)));
    MG_TRY(run_forward(M, pp, nt, nullptr, ckpt_every, P<float>(M->ckpt), st, flags));
  }
  float* ck = P<float>(M->ckpt);
  // segment buffer: slot j holds p_{l0-1+j}, j = 0..K+1
  const int K = std::min(ckpt_every, nt);
  MG_TRY(ensure(M->seg, (size_t)(K + 2) * state * sizeof(float)));
  float* seg = P<float>(M->seg);
  // adjoint states and accumulators
  MG_TRY(ensure(M->stC, state * sizeof(float)));
  MG_TRY(ensure(M->stD, state * sizeof(float)));
  float* mu = P<float>(M->stC);
  float* mu1 = P<float>(M->stD);
  MG_CU(cudaMemsetAsync(mu, 0, state * sizeof(float), st));
  MG_CU(cudaMemsetAsync(mu1, 0, state * sizeof(float), st));
  // Shot groups: every recompute and reverse launch covers the columns of
  // one group; each group runs a whole segment before the next one (the
  // forward kind's grouping for the recompute, the adjoint's for the
  // reverse steps).
  const int Wf = group_cols(M, 0, pp.S_pad), NGf = pp.S_pad / Wf;
  const int Wa = group_cols(M, 2, pp.S_pad), NGa = pp.S_pad / Wa;
  // resident kernels for the recompute and the reverse steps of a segment (not
  // for one too short; MG_PERSISTENT asks for its own kernels)
  mg::DevPatches Df, Da;
  mg::ResidentShape shf, sha;
  if (!(flags & MG_PERSISTENT)) {
    MG_TRY(resident_shape(M, 0, pp.S_pad, std::min(ckpt_every, nt), Df, shf, true));
    MG_TRY(resident_shape(M, 2, pp.S_pad, std::min(ckpt_every, nt), Da, sha));
  }
  // accumulators: one set per source tile of the untiled kernel; the tiled
  // kernel sums all shots of a row inside its CTA; the resident kernel, which
  // either of them may share the segments with, one per source tile
  int acc_sets = adjoint_sets(M, pp.S_pad, Wa);
  if (sha.lpr) acc_sets = std::max(acc_sets, pp.S_pad / (4 * sha.lpr));
  const size_t acc = (size_t)acc_sets * n;
  MG_TRY(ensure(M->G, 4 * acc * sizeof(float)));
  MG_CU(cudaMemsetAsync(M->G.p, 0, 4 * acc * sizeof(float), st));
  float* G = P<float>(M->G);
  mg::StepArgs fa = step_args(M, pp, pp.S_pad, nt);
  fa.traces = nullptr;
  mg::AdjointArgs aa{};
  aa.K = dev_ell(M);
  aa.ev = pp.ev;
  aa.coef = P<const float4>(M->coef);
  aa.ld = pp.S_pad;
  aa.w = wd;
  aa.nt = nt;
  aa.step_base = nullptr;
  const mg_mesh::Tuning ta = in_force(M, 2);
  aa.batch = ta.batch;
  aa.ring = ta.ring;
  aa.stream = ta.stream;
  aa.prefetch = ta.prefetch;
  aa.min_blocks = ta.min_blocks;
  aa.G = G;
  aa.Gc = G + acc;
  aa.H = G + 2 * acc;
  aa.Hc = G + 3 * acc;
  aa.hint = states ? M->cache_hints : 0;
  const bool use_graph = graphs_on(M, flags) && ckpt_every % 2 == 0 && ckpt_every <= nt;
  int32_t* base = nullptr;
  if (use_graph) {
    MG_TRY(ensure(M->step_base, 16));
    base = P<int32_t>(M->step_base);
  }
  if (!shf.lpr && !states) MG_TRY(ensure_auto_entries(M, 0, Wf, st));
  if (!sha.lpr) MG_TRY(ensure_auto_entries(M, 2, Wa, st));
  mg::ResidentAdjArgs ra{};
  if (sha.lpr) {
    ra.P = Da;
    ra.ev = pp.ev;
    ra.coef = aa.coef;
    ra.w = wd;
    ra.nt = nt;
    ra.ld = pp.S_pad;
    ra.state = (int64_t)state;
  }
  // false: not on the resident kernel (rc says whether something failed)
  auto resident_recompute = [&](int a, int l0, int l1, int& rc) {
    rc = MG_OK;
    if (!shf.lpr || l1 - l0 < 16) return false;
    const float* slot = ck + (size_t)a * 2 * state;
    rc = run_recompute_resident(M, pp, nt, l0, l1 - l0, slot, slot + state, seg + 2 * state, Df,
                                shf, st);
    if (rc != MG_ERR_UNSUPPORTED) return true;
    rc = MG_OK;
    shf.lpr = 0;
    return false;
  };
  auto resident_reverse = [&](int l0, int l1, int& rc) {
    rc = MG_OK;
    if (!sha.lpr || l1 - l0 < 16) return false;
    rc = resident_buffers(M, Da, sha.lpr, st, ra);
    ra.mu = mu;
    ra.mu1 = mu1;
    ra.k = l1;
    ra.steps = l1 - l0;
    ra.pk = seg + (size_t)(l1 - l0 + 1) * state;
    for (int set = 0; rc == MG_OK && set * 4 * sha.lpr < pp.S_pad; ++set) {
      ra.col0 = set * 4 * sha.lpr;
      ra.G = aa.G + (size_t)set * n;
      ra.Gc = aa.Gc + (size_t)set * n;
      ra.H = aa.H + (size_t)set * n;
      ra.Hc = aa.Hc + (size_t)set * n;
      rc = mg::launch_resident_adjoint(ra, sha, st);
      M->launches += 1;
    }
    if (rc != MG_ERR_UNSUPPORTED) return true;   // refused before its first launch only
    rc = MG_OK;
    sha.lpr = 0;
    return false;
  };
  for (int a = nck - 1; a >= 0; --a) {
    const int l0 = a * ckpt_every;
    const int l1 = std::min(nt, l0 + ckpt_every);
    int rc = MG_OK;
    const bool recomputed = !states && resident_recompute(a, l0, l1, rc);
    MG_TRY(rc);
    if (!states && !recomputed) {
      MG_TRY(mg::launch_copy_f4(ck + (size_t)a * 2 * state, seg + state, (int64_t)state, st));
      MG_TRY(mg::launch_copy_f4(ck + (size_t)a * 2 * state + state, seg, (int64_t)state, st));
      M->launches += 2;
    }
    if (flags & MG_PERSISTENT) {   // kept history: one segment, l0 = 0, l1 = nt
      mg::PersistArgs pa{};
      MG_TRY(persist_args(M, st, seg, state, pa));
      for (int g = 0; g < NGa; ++g) {
        mg::AdjointArgs b = aa;
        b.col0 = g * Wa;
        b.cols = Wa;
        float* x = mu;
        float* y = mu1;
        for (int k = l1; k > l0;) {
          pa.steps = std::min(k - l0, M->persist_steps);
          b.mu = x;
          b.mu1 = y;
          b.k = k;
          MG_TRY(mg::launch_adjoint_persist(b, pp.S_pad, pa, st));
          M->launches += 1;
          if (pa.steps % 2) std::swap(x, y);
          k -= pa.steps;
        }
      }
      if ((l1 - l0) % 2) std::swap(mu, mu1);
      MG_TRY(persist_status(M, st));
      continue;
    }
    if (use_graph && l1 - l0 == ckpt_every) {
      // whole segment: recompute p_{l0+1..l1}, then reverse steps k = l1..l0+1,
      // each as one graph; indices relative to *base = l0
      MG_TRY(mg::launch_set_int(base, l0, st));
      M->launches += 1;
      const std::string kr = key_of("rec", {seg, fa.wavelet, fa.coef, fa.ev.src_ptr, base},
                                    {pp.S_pad, pp.S, pp.R, nt, ckpt_every, n, Wf});
      if (!states && !recomputed) MG_TRY(run_graph(M, kr, NGf * ckpt_every, st, [&](cudaStream_t cs) {
        mg::StepArgs b = fa;
        b.step_base = base;
        b.cols = Wf;
        for (int g = 0; g < NGf; ++g) {
          b.col0 = g * Wf;
          for (int j = 1; j <= ckpt_every; ++j) {
            b.p = seg + (size_t)j * state;
            b.pm = seg + (size_t)(j - 1) * state;
            b.pout = seg + (size_t)(j + 1) * state;
            b.step = j - 1;
            MG_TRY(do_step(M, b, pp.S_pad, cs));
          }
        }
        return MG_OK;
      }));
      if (resident_reverse(l0, l1, rc)) {
        MG_TRY(rc);
        continue;
      }
      const std::string ka = key_of("adj", {seg, mu, mu1, wd, aa.coef, aa.ev.rec_ptr, G, base},
                                    {pp.S_pad, pp.S, pp.R, nt, ckpt_every, n, Wa});
      MG_TRY(run_graph(M, ka, NGa * ckpt_every, st, [&](cudaStream_t cs) {
        mg::AdjointArgs b = aa;
        b.step_base = base;
        b.cols = Wa;
        for (int g = 0; g < NGa; ++g) {
          b.col0 = g * Wa;
          float* x = mu;
          float* y = mu1;
          for (int r = ckpt_every; r >= 1; --r) {   // k = l0 + r
            b.mu = x;
            b.mu1 = y;
            b.pk = seg + (size_t)(r + 1) * state;
            b.k = r;
            MG_TRY(do_adjoint(M, b, pp.S_pad, cs));
            std::swap(x, y);
          }
        }
        return MG_OK;
      }));
      continue;   // even segment length: mu / mu1 are back in place
    }
    for (int l = l0; l < l1 && !states && !recomputed; ++l) {
      const int j = l - l0 + 1;  // slot of p_l
      fa.p = seg + (size_t)j * state;
      fa.pm = seg + (size_t)(j - 1) * state;
      fa.pout = seg + (size_t)(j + 1) * state;
      fa.step = l;
      MG_TRY(do_step(M, fa, pp.S_pad, st));
      M->launches += 1;
    }
    if (resident_reverse(l0, l1, rc)) {
      MG_TRY(rc);
      continue;
    }
    for (int g = 0; g < NGa; ++g) {
      mg::AdjointArgs b = aa;
      b.col0 = g * Wa;
      b.cols = Wa;
      float* x = mu;
      float* y = mu1;
      for (int k = l1; k > l0; --k) {
        b.mu = x;
        b.mu1 = y;
        b.pk = seg + (size_t)(k - l0 + 1) * state;
        b.k = k;
        MG_TRY(do_adjoint(M, b, pp.S_pad, st));
        M->launches += 1;
        std::swap(x, y);
      }
    }
    if ((l1 - l0) % 2) std::swap(mu, mu1);
  }
  // per-cell gradient (FP64), then restriction to the level
  MG_TRY(ensure(M->gfine, M->hm.m * sizeof(double)));
  mg::GradArgs ga;
  ga.m = M->hm.m;
  ga.k = M->hm.dim + 1;
  ga.dim = M->hm.dim;
  ga.cells = P<int32_t>(M->cells);
  ga.vol = P<double>(M->vol);
  ga.cf_ptr = P<int64_t>(M->cf_ptr);
  ga.cf_facet = P<int32_t>(M->cf_facet);
  ga.bnd = P<int32_t>(M->bnd);
  ga.bnd_meas = P<double>(M->bnd_meas);
  ga.eps = pp.eps;
  ga.dt = dt;
  ga.bc = M->hm.bc;
  ga.n = (int32_t)n;
  ga.tiles = acc_sets;
  ga.G = aa.G; ga.Gc = aa.Gc; ga.H = aa.H; ga.Hc = aa.Hc;
  ga.g_fine = P<double>(M->gfine);
  MG_TRY(mg::launch_cell_gradient(ga, st));
  const int64_t nc = M->hm.n_cells_level[level];
  MG_TRY(ensure(M->g_h, nc * sizeof(double)));
  MG_TRY(mg::launch_restrict(nc, P<int64_t>(M->lvl_ptr[level]), P<int32_t>(M->lvl_idx[level]),
                             ga.g_fine, P<double>(M->g_h), st));
  M->launches += 2;
  MG_TRY(poison(M, P<float>(M->g_h), 2 * nc, reuse, st));
  return deliver(M->g_h, g, nc * sizeof(double), flags, st);
}

int mg_autotune(mg_mesh* M, const double* eps, const mg_shots* shots, const double* wavelet,
                double dt, int steps, int level, void* stream, int flags, int32_t* chosen) {
  if (!M || !eps || !shots || !wavelet || steps < 2 || level < 0 || level >= M->hm.n_levels)
    return MG_ERR_ARG;
  if (flags & ~MG_ALLOW_CFL) return MG_ERR_UNSUPPORTED;
  MG_TRY(validate_shots(M, shots));
  DeviceGuard guard(M->device);
  if (!guard.ok) return MG_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int S_pad = round_pad(shots->n_shots);
  auto hit = M->tuned.find(S_pad);
  if (hit != M->tuned.end()) {
    drop_graphs(M);
    for (int k = 0; k < 3; ++k) M->tune[k] = hit->second[k];
    return chosen ? mg_mesh_get_tuning(M, chosen) : MG_OK;
  }
  // scratch: traces / weights [R][steps] and level vectors
  const int64_t R = shots->rec_ptr[shots->n_shots];
  const int64_t nl = M->hm.n_cells_level[level];
  const size_t tb = ((size_t)R * steps * sizeof(float) + 255) / 256 * 256;
  const size_t vb = ((size_t)nl * sizeof(double) + 255) / 256 * 256;
  MG_TRY(ensure(M->tune_scratch, 2 * tb + 2 * vb));
  unsigned char* base = P<unsigned char>(M->tune_scratch);
  MG_CU(cudaMemsetAsync(base, 0, 2 * tb + 2 * vb, st));
  float* tr = reinterpret_cast<float*>(base);
  const float* w0 = reinterpret_cast<const float*>(base + tb);
  const double* v0 = reinterpret_cast<const double*>(base + 2 * tb);
  double* g0 = reinterpret_cast<double*>(base + 2 * tb + vb);
  const int K = steps;  // one checkpoint segment
  auto run = [&](int kind) -> int {
    switch (kind) {
      case 0: return mg_forward(M, eps, shots, wavelet, dt, steps, tr, 0, stream, flags);
      case 1: return mg_jacobian_apply(M, level, eps, shots, wavelet, dt, steps, v0, tr, stream,
                                       flags);
      default: return mg_jacobian_T_apply(M, level, eps, shots, wavelet, dt, steps, w0, g0, K,
                                          stream, flags);
    }
  };
  // the register-capped shapes (5 CTAs per SM) and the row sweeps of 4
  // blocks per CTA (mg_mesh_set_row_sweep) apply to the forward only;
  // the row kernels with a gather ring of 4 or 8 slots to every kind (a
  // ring that exceeds a CTA's shared memory is skipped); the bulk-copy
  // kernel and the bulk-copy tiled kernel are not candidates (measured
  // slower on every workload: 2D 41.6 and 92.7 vs 19.7 us, 3D 769 and
  // 2620 vs 532 us per step)
  const mg_mesh::Tuning shapes[] = {
      {1, 0, 32},          {2, 0, 32},          {4, 0, 32},          {1, 64, 32},
      {1, 64, 16},         {1, 128, 32},        {1, 128, 16},        {1, 256, 32},
      {1, 256, 16},        {2, 0, 32, 1, 5},    {4, 0, 32, 1, 5},    {1, 0, 32, 1, 0, 0, 4},
      {2, 0, 32, 1, 0, 0, 4}, {4, 0, 32, 1, 0, 0, 4}, {1, 0, 32, 1, 0, 0, 8},
      {2, 0, 32, 1, 0, 0, 8}, {4, 0, 32, 1, 0, 0, 8}, {1, 0, 32, 1, 0, 0, 0, 4},
      {2, 0, 32, 1, 5, 0, 0, 4}, {4, 0, 32, 1, 5, 0, 0, 4}, {1, 0, 32, 1, 5},
      {1, 0, 32, 1, 6},    {2, 0, 32, 1, 6},    {2, 0, 32, 1, 5}};
  const int n_shapes = (int)(sizeof(shapes) / sizeof(shapes[0]));
  cudaEvent_t e0, e1;
  MG_CU(cudaEventCreate(&e0));
  MG_CU(cudaEventCreate(&e1));
  int rc = MG_OK;
  // bring the clocks up before anything is timed: a GPU coming out of idle
  // would otherwise bias against the first candidates
  for (int i = 0; i < 4 && rc == MG_OK; ++i) rc = run(2);
  if (rc == MG_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = MG_ERR_CUDA;
  // the L1 policy is the caller's setting, not a candidate
  const int l1[3] = {M->tune[0].stream, M->tune[1].stream, M->tune[2].stream};
  auto time_of = [&](int kind, mg_mesh::Tuning c, float* out, int path = MG_PATH_SHAPE) -> int {
    drop_graphs(M);
    c.stream = l1[kind];
    c.path = path;
    M->tune[kind] = c;
    int r = run(kind);  // warm-up: tile tables, buffers, graphs
    float cand = 1e30f;
    for (int rep = 0; rep < 3 && r == MG_OK; ++rep) {  // best of three
      cudaEventRecord(e0, st);
      r = run(kind);
      cudaEventRecord(e1, st);
      if (r != MG_OK) break;
      if (cudaEventSynchronize(e1) != cudaSuccess) { r = MG_ERR_CUDA; break; }
      float ms = 0.0f;
      cudaEventElapsedTime(&ms, e0, e1);
      cand = std::min(cand, ms);
    }
    *out = cand;
    return r == MG_ERR_UNSUPPORTED ? MG_OK : r;   // a ring too large for the shape: skipped
  };
  for (int kind = 0; kind < 3 && rc == MG_OK; ++kind) {
    // launch shapes with one shot group, then 2, 4 and 8 groups on the two
    // fastest shapes (groups that do not give a valid width are skipped)
    float ms[n_shapes];
    for (int i = 0; i < n_shapes && rc == MG_OK; ++i) {
      ms[i] = 1e30f;
      // register caps: 5 CTAs per SM for every kind, 6 for the adjoint;
      // the other variants apply to the forward only
      if (((shapes[i].bulk || shapes[i].sweep || shapes[i].tma) && kind != 0) ||
          (shapes[i].min_blocks == 6 && kind != 2))
        continue;
      rc = time_of(kind, shapes[i], &ms[i]);
    }
    if (rc != MG_OK) break;
    int order[n_shapes];
    for (int i = 0; i < n_shapes; ++i) order[i] = i;
    std::stable_sort(order, order + n_shapes, [&](int x, int y) { return ms[x] < ms[y]; });
    // candidates within 1% of the fastest count as equal (run-to-run noise
    // is of that size): the earliest in the list wins, so repeated tuning
    // of the same problem settles on the same shape
    int first = order[0];
    for (int i = 0; i < n_shapes; ++i)
      if (ms[i] <= ms[order[0]] * 1.01f) { first = i; break; }
    float best = ms[first];
    mg_mesh::Tuning pick = shapes[first];
    pick.stream = l1[kind];
    // groups act only inside graph chunks (forward, tangent: runs of at
    // least `chunk` steps) and graph segments (adjoint: even segments), so
    // they are timed only when the timed runs use them
    const bool grouped = M->chunk >= 2 && (kind == 2 ? steps % 2 == 0 : steps >= M->chunk);
    for (int top = 0; top < 2 && rc == MG_OK && grouped; ++top) {
      for (int G : {2, 4, 8}) {
        mg_mesh::Tuning c = shapes[order[top]];
        c.groups = G;
        c.stream = l1[kind];
        c.path = MG_PATH_SHAPE;
        M->tune[kind] = c;
        if (group_cols(M, kind, S_pad) == S_pad) continue;
        float t = 0.0f;
        rc = time_of(kind, c, &t);
        if (rc != MG_OK) break;
        if (t < best * 0.99f) { best = t; pick = c; }   // groups must win by more than 1%
      }
    }
    pick.path = MG_PATH_SHAPE;
    // the library's own row shape and, wherever the problem fits it, the resident
    // kernel against the best of these; MG_PATH_AUTO where its estimate chooses the
    // winner by itself (it chooses anew for other shot counts)
    mg::DevPatches D;
    mg::ResidentShape shape;
    auto fits = [&](int path) {
      M->tune[kind].path = path;
      rc = resident_shape(M, kind, S_pad, steps, D, shape);
      return rc == MG_OK && shape.lpr > 0;
    };
    float t = 0.0f;
    if (rc == MG_OK) rc = time_of(kind, pick, &t, MG_PATH_ROWS);
    if (rc == MG_OK && t < best * 0.99f) {
      best = t;
      pick.path = MG_PATH_ROWS;
    }
    if (rc == MG_OK && fits(MG_PATH_RESIDENT)) {
      rc = time_of(kind, pick, &t, MG_PATH_RESIDENT);
      if (rc == MG_OK && t < best) pick.path = MG_PATH_RESIDENT;
    }
    if (rc == MG_OK && pick.path != MG_PATH_SHAPE) {
      const bool resident = fits(MG_PATH_AUTO);
      if (rc == MG_OK && resident == (pick.path == MG_PATH_RESIDENT)) pick.path = MG_PATH_AUTO;
    }
    M->tune[kind] = pick;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  drop_graphs(M);
  if (rc != MG_OK) return rc;
  M->tuned[S_pad] = {M->tune[0], M->tune[1], M->tune[2]};
  return chosen ? mg_mesh_get_tuning(M, chosen) : MG_OK;
}

}  // extern "C"

namespace mg {

int padded_shots(int S) { return round_pad(S); }
const HostMesh* host_mesh(const mg_mesh* M) { return M ? &M->hm : nullptr; }
int mesh_device(const mg_mesh* M) { return M->device; }
int mesh_graph_chunk(const mg_mesh* M) { return M->chunk; }
void add_launches(mg_mesh* M, int64_t n) { M->launches += n; }

int mesh_poisoned(mg_mesh* M, cudaStream_t st, int* count) {
  *count = 0;
  if (!M->errbuf.p) return MG_OK;
  MG_CU(cudaMemcpyAsync(count, P<int>(M->errbuf) + kWordPoisoned, sizeof(int),
                        cudaMemcpyDeviceToHost, st));
  MG_CU(cudaStreamSynchronize(st));
  return MG_OK;
}

void mesh_take_scratch(mg_mesh* M, std::vector<FluxBuffer>& bufs) {
  std::lock_guard<std::mutex> lock(M->flux_mu);
  bufs.clear();
  bufs.swap(M->flux_scratch);
}

bool mesh_keep_scratch(mg_mesh* M, std::vector<FluxBuffer>& bufs) {
  std::lock_guard<std::mutex> lock(M->flux_mu);
  if (!M->flux_scratch.empty()) return false;
  bufs.swap(M->flux_scratch);
  return true;
}

long long mesh_wait_budget(const mg_mesh* M) { return M->persist_budget; }
std::mutex& mesh_flux_mutex(mg_mesh* M) { return M->flux_mu; }

bool mesh_flux_geometry(mg_mesh* M, FluxGeometry* g) {
  if (!M->flux_inc.p) return false;
  g->cell = P<const float4>(M->flux_cell);
  g->inc_ptr = P<const int32_t>(M->flux_ptr);
  g->inc = P<const int4>(M->flux_inc);
  g->cells = P<const int32_t>(M->cells);
  g->patches = M->flux_patches;
  return true;
}

int mesh_set_flux_geometry(mg_mesh* M, const std::vector<float>& cell,
                           const std::vector<int32_t>& ptr, const std::vector<int4>& inc,
                           const HostFluxPatches& H, FluxGeometry* g) {
  if (H.B) {
    DevFluxPatches D{};
    int k = 0, rc = MG_OK;
    auto put = [&](const std::vector<int32_t>& v, const int32_t*& to) {
      Buf& b = M->flux_tab[k++];
      if (rc == MG_OK) rc = upload(b, v);
      to = P<const int32_t>(b);
    };
    put(H.own_off, D.own_off);
    put(H.border, D.border);
    put(H.halo_off, D.halo_off);
    put(H.x_off, D.x_off);
    put(H.cell_off, D.cell_off);
    put(H.inner, D.inner);
    put(H.inc_off, D.inc_off);
    put(H.row, D.row);
    put(H.row_inc, D.row_inc);
    put(H.halo, D.halo);
    put(H.halo_x, D.halo_x);
    put(H.cell, D.cell);
    put(H.cell_slot, D.cell_slot);
    if (rc == MG_OK) rc = upload(M->flux_pinc, H.inc);
    D.inc = P<const int4>(M->flux_pinc);
    D.n_x = H.x_off[H.B];
    D.max_own = H.max_own;
    D.max_halo = H.max_halo;
    D.max_slots = H.max_slots;
    D.max_cells = H.max_cells;
    D.max_inc = H.max_inc;
    D.B = H.B;
    if (rc == MG_OK) {
      M->flux_patches = D;
    } else {   // no memory for them: launches per step
      for (Buf* b = M->flux_tab.data(); b != M->flux_tab.data() + M->flux_tab.size(); ++b) {
        if (b->p) cudaFree(b->p);
        *b = Buf{};
      }
      if (M->flux_pinc.p) cudaFree(M->flux_pinc.p);
      M->flux_pinc = Buf{};
      if (rc != MG_ERR_OOM) return rc;
    }
  }
  MG_TRY(upload(M->flux_cell, cell));
  MG_TRY(upload(M->flux_ptr, ptr));
  MG_TRY(upload(M->flux_inc, inc));   // last: its presence marks the set
  MG_CU(cudaStreamSynchronize(cudaStreamLegacy));   // as in upload_groups
  mesh_flux_geometry(M, g);
  return MG_OK;
}

int mesh_view(mg_mesh* M, MeshView* v) {
  if (!M || !v) return MG_ERR_ARG;
  v->device = M->device;
  v->bc = M->hm.bc;
  v->n = M->hm.n;
  v->m = M->hm.m;
  v->K = dev_ell(M);
  v->coef_base = coef_args(M, nullptr, 0.0);
  v->coef_base.coef = nullptr;
  v->row_abs = P<const double>(M->row_abs);
  v->perm_host = M->hm.perm.data();
  v->launches = &M->launches;
  v->batch = in_force(M, 0).batch;
  return MG_OK;
}

int prepare_instance(mg_mesh* M, const double* eps, const mg_shots* shots, const double* wavelet,
                     double dt, int nt, int flags, void* stream, int ckpt_every, const float* w,
                     InstanceView* v) {
  if (!M || !v) return MG_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Prep pp;
  MG_TRY(prepare(M, eps, shots, wavelet, dt, nt, flags, st, pp));
  const int64_t n = M->hm.n;
  const size_t state = (size_t)n * pp.S_pad;
  for (Buf* b : {&M->stA, &M->stB, &M->stC, &M->stD}) MG_TRY(ensure(*b, state * sizeof(float)));
  MG_TRY(ensure(M->tr, (size_t)pp.R * nt * sizeof(float)));
  v->K = dev_ell(M);
  v->ev = pp.ev;
  v->coef = P<const float4>(M->coef);
  v->wavelet = P<const float>(M->wavf);
  v->eps = pp.eps;
  v->S = pp.S;
  v->S_pad = pp.S_pad;
  v->tiles = pp.tiles;
  v->R = pp.R;
  v->n = n;
  v->A = P<float>(M->stA);
  v->B = P<float>(M->stB);
  v->C = P<float>(M->stC);
  v->D = P<float>(M->stD);
  v->tr = P<float>(M->tr);
  v->ckpt = v->seg = nullptr;
  v->G = nullptr;
  v->w = nullptr;
  if (ckpt_every > 0) {
    const int nck = (nt + ckpt_every - 1) / ckpt_every;
    MG_TRY(ensure(M->ckpt, (size_t)nck * 2 * state * sizeof(float)));
    MG_TRY(ensure(M->seg, (size_t)(std::min(ckpt_every, nt) + 2) * state * sizeof(float)));
    MG_TRY(ensure(M->G, 4 * (size_t)pp.tiles * n * sizeof(float)));
    v->ckpt = P<float>(M->ckpt);
    v->seg = P<float>(M->seg);
    v->G = P<float>(M->G);
    M->ck_valid = false;  M->ck_gen++;
    M->seg_full = false;
  }
  if (w) {
    const size_t wbytes = (size_t)pp.R * nt * sizeof(float);
    MG_TRY(ensure(M->w_h, wbytes));
    MG_CU(cudaMemcpyAsync(M->w_h.p, w, wbytes,
                          (flags & MG_HOST_PTRS) ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice,
                          st));
    v->w = P<const float>(M->w_h);
  }
  v->launches = &M->launches;
  return MG_OK;
}

int finish_gradient(mg_mesh* M, int level, const double* eps_dev, double dt, int tiles, double* g,
                    int flags, void* stream) {
  if (!M || !g || level < 0 || level >= M->hm.n_levels) return MG_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  MG_TRY(ensure_level(M, level));
  MG_TRY(ensure(M->gfine, M->hm.m * sizeof(double)));
  const size_t acc = (size_t)tiles * M->hm.n;
  float* G = P<float>(M->G);
  mg::GradArgs ga;
  ga.m = M->hm.m;
  ga.k = M->hm.dim + 1;
  ga.dim = M->hm.dim;
  ga.cells = P<int32_t>(M->cells);
  ga.vol = P<double>(M->vol);
  ga.cf_ptr = P<int64_t>(M->cf_ptr);
  ga.cf_facet = P<int32_t>(M->cf_facet);
  ga.bnd = P<int32_t>(M->bnd);
  ga.bnd_meas = P<double>(M->bnd_meas);
  ga.eps = eps_dev;
  ga.dt = dt;
  ga.bc = M->hm.bc;
  ga.n = (int32_t)M->hm.n;
  ga.tiles = tiles;
  ga.G = G; ga.Gc = G + acc; ga.H = G + 2 * acc; ga.Hc = G + 3 * acc;
  ga.g_fine = P<double>(M->gfine);
  MG_TRY(mg::launch_cell_gradient(ga, st));
  const int64_t nc = M->hm.n_cells_level[level];
  MG_TRY(ensure(M->g_h, nc * sizeof(double)));
  MG_TRY(mg::launch_restrict(nc, P<int64_t>(M->lvl_ptr[level]), P<int32_t>(M->lvl_idx[level]),
                             ga.g_fine, P<double>(M->g_h), st));
  M->launches += 2;
  return deliver(M->g_h, g, nc * sizeof(double), flags, st);
}

}  // namespace mg
