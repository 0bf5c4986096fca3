// Patch tables of the flux path's resident kernels (resident_flux.h).
#include <algorithm>

#include "resident_flux.h"

namespace mg {

int build_flux_patches(const HostMesh& hm, int B, const std::vector<int4>& geo_inc,
                       HostFluxPatches& F) {
  HostPatches P;
  const int rc = build_patches(hm, B, P);
  if (rc != MG_OK) return rc;
  const int k1 = hm.dim + 1;
  F = HostFluxPatches();
  F.B = B;
  std::vector<int32_t> slot(hm.n), xrow(hm.n, -1);   // slot in its patch, exchange row
  std::vector<std::vector<int32_t>> cells(B);
  F.border = P.n_border;
  F.inner.assign(B, 0);
  for (auto* v : {&F.halo_off, &F.x_off, &F.cell_off, &F.inc_off}) v->assign(B + 1, 0);
  F.own_off = P.own_off;
  F.row = P.row;
  for (int b = 0; b < B; ++b) {
    F.x_off[b + 1] = F.x_off[b] + P.n_border[b];
    F.halo_off[b + 1] = F.halo_off[b] + (int)P.halo[b].size();
    for (int i = P.own_off[b]; i < P.own_off[b + 1]; ++i) {
      const int s = i - P.own_off[b];
      slot[P.row[i]] = s;
      if (s < P.n_border[b]) xrow[P.row[i]] = F.x_off[b] + s;
    }
  }
  int bad = 0, oom = 0;
#pragma omp parallel reduction(+ : oom)
  {
    Stamps seen(hm.m);
#pragma omp for schedule(dynamic, 4)
    for (int b = 0; b < B; ++b) no_throw(oom, [&] {
      seen.need();
      std::vector<int32_t>& c = cells[b];
      for (int i = P.own_off[b]; i < P.own_off[b + 1]; ++i)
        for (int64_t q = hm.nc_ptr[P.row[i]]; q < hm.nc_ptr[P.row[i] + 1]; ++q) {
          if (!seen[hm.nc_cell[q]]) c.push_back(hm.nc_cell[q]);
          seen[hm.nc_cell[q]] = 1;
        }
      for (int32_t e : c) seen[e] = 0;
      auto inner = [&](int32_t e) {
        for (int a = 0; a < k1; ++a)
          if (P.part[hm.cells[(size_t)e * k1 + a]] != b) return false;
        return true;
      };
      F.inner[b] = (int)(std::stable_partition(c.begin(), c.end(), inner) - c.begin());
    });
  }
  if (oom) return MG_ERR_OOM;
  for (int b = 0; b < B; ++b) {
    int inc = 0;
    for (int i = P.own_off[b]; i < P.own_off[b + 1]; ++i)
      inc += (int)(hm.nc_ptr[P.row[i] + 1] - hm.nc_ptr[P.row[i]]);
    const int own = P.own_off[b + 1] - P.own_off[b], h = (int)P.halo[b].size();
    F.cell_off[b + 1] = F.cell_off[b] + (int)cells[b].size();
    F.inc_off[b + 1] = F.inc_off[b] + inc;
    F.max_own = std::max(F.max_own, own);
    F.max_halo = std::max(F.max_halo, h);
    F.max_slots = std::max(F.max_slots, own + h);
    F.max_cells = std::max(F.max_cells, (int)cells[b].size());
    F.max_inc = std::max(F.max_inc, inc);
  }
  if (F.max_inc >= 1 << kIncShift) return MG_ERR_UNSUPPORTED;
  F.row_inc.resize(hm.n);
  F.halo.resize(F.halo_off[B]);
  F.halo_x.resize(F.halo_off[B]);
  F.cell.resize(F.cell_off[B]);
  F.cell_slot.assign((size_t)F.cell_off[B] * 4, 0);
  F.inc.resize(F.inc_off[B]);
#pragma omp parallel reduction(+ : bad, oom)
  {
    Stamps at(hm.m), halo(hm.n);   // place of a cell, slot of a halo row, plus 1
#pragma omp for schedule(dynamic, 4)
    for (int b = 0; b < B; ++b) no_throw(oom, [&] {
      at.need();
      halo.need();
      const std::vector<int32_t>&c = cells[b], &h = P.halo[b];
      const int own = P.own_off[b + 1] - P.own_off[b];
      for (size_t i = 0; i < h.size(); ++i) {
        F.halo[F.halo_off[b] + i] = h[i];
        F.halo_x[F.halo_off[b] + i] = xrow[h[i]];
        halo[h[i]] = own + (int32_t)i + 1;
      }
      for (size_t i = 0; i < c.size(); ++i) {
        const int32_t* v = hm.cells.data() + (size_t)c[i] * k1;
        at[c[i]] = (int32_t)i + 1;
        F.cell[F.cell_off[b] + i] = P.part[v[0]] == b ? c[i] : ~c[i];
        for (int a = 0; a < k1; ++a) {
          // the rows of a cell couple with one another: a foreign one is a halo row
          const int32_t s = P.part[v[a]] == b ? slot[v[a]] : halo[v[a]] - 1;
          if (s < 0) ++bad;
          F.cell_slot[(size_t)(F.cell_off[b] + i) * 4 + a] = s;
        }
      }
      int k = 0;
      for (int i = P.own_off[b]; i < P.own_off[b + 1]; ++i) {
        const int32_t r = P.row[i];
        const int cnt = (int)(hm.nc_ptr[r + 1] - hm.nc_ptr[r]);
        if (cnt >= 1 << (31 - kIncShift)) ++bad;
        F.row_inc[i] = k | cnt << kIncShift;
        for (int64_t s = hm.nc_ptr[r]; s < hm.nc_ptr[r + 1]; ++s) {
          int4 q = geo_inc[s];
          q.x = at[q.x] - 1;
          F.inc[F.inc_off[b] + k++] = q;
        }
      }
      for (int32_t r : h) halo[r] = 0;
      for (int32_t e : c) at[e] = 0;
    });
  }
  return oom ? MG_ERR_OOM : bad ? MG_ERR_UNSUPPORTED : MG_OK;
}

}  // namespace mg
