// Partition of a mesh's rows over the CTAs of the resident kernels
// (resident_common.cuh) and the patch-local form of the stiffness: recursive
// coordinate bisection into compact patches, whichever order the rows are
// numbered in.
#include <algorithm>
#include <numeric>

#include "resident.h"

namespace mg {
namespace {

// A row with its point, moved together: the bisection walks memory in order.
struct Pt {
  double x[3];
  int32_t row;
};

// Cuts [p, p + n) into the patches b0 .. b1-1 along the longest extent; ties in
// the coordinate go by row number, so the partition depends on the mesh alone.
void bisect(Pt* p, int64_t n, int dim, int b0, int b1, std::vector<int32_t>& part) {
  if (b1 - b0 == 1) {
    for (int64_t i = 0; i < n; ++i) part[p[i].row] = b0;
    return;
  }
  int axis = 0;
  double best = -1.0;
  for (int a = 0; a < dim; ++a) {
    double lo = 1e300, hi = -1e300;
    for (int64_t i = 0; i < n; ++i) {
      lo = std::min(lo, p[i].x[a]);
      hi = std::max(hi, p[i].x[a]);
    }
    if (hi - lo > best) {
      best = hi - lo;
      axis = a;
    }
  }
  const int bm = b0 + (b1 - b0) / 2;
  const int64_t k = n * (bm - b0) / (b1 - b0);
  if (k < n)
    std::nth_element(p, p + k, p + n, [axis](const Pt& u, const Pt& v) {
      return u.x[axis] != v.x[axis] ? u.x[axis] < v.x[axis] : u.row < v.row;
    });
#pragma omp task shared(part) if (n > 4096)
  bisect(p, k, dim, b0, bm, part);
  bisect(p + k, n - k, dim, bm, b1, part);
#pragma omp taskwait
}

}  // namespace

int build_patches(const HostMesh& hm, int B, HostPatches& P) {
  const int64_t n = hm.n;
  if (B < 1 || B > n || n > 0x3fffffff) return MG_ERR_ARG;
  P = HostPatches();
  P.B = B;
  std::vector<int32_t> part(n);
  {
    std::vector<Pt> pts(n);
    for (int64_t r = 0; r < n; ++r) {
      for (int a = 0; a < hm.dim; ++a) pts[r].x[a] = hm.coords[(size_t)r * hm.dim + a];
      pts[r].row = (int32_t)r;
    }
#pragma omp parallel
#pragma omp single
    bisect(pts.data(), n, hm.dim, 0, B, part);
  }
  P.own_off.assign(B + 1, 0);
  for (int64_t r = 0; r < n; ++r) P.own_off[part[r] + 1]++;
  for (int b = 0; b < B; ++b) P.own_off[b + 1] += P.own_off[b];
  P.row.resize(n);
  {
    std::vector<int32_t> fill(P.own_off.begin(), P.own_off.end() - 1);
    for (int64_t r = 0; r < n; ++r) P.row[fill[part[r]]++] = (int32_t)r;
  }
  // border rows: coupled to a row of another patch, in either direction (the
  // pattern is symmetric patch by patch, which is checked: the exchange's two
  // halves are only safe when a patch that reads another is read by it)
  std::vector<uint8_t> border(n, 0);
  P.halo.resize(B);
  std::vector<std::vector<int32_t>> reads(B);   // patches that a patch reads
  int oom = 0;
#pragma omp parallel reduction(+ : oom)
  {
    Stamps row(n), other(B);   // halo rows and patches seen
#pragma omp for schedule(dynamic, 4)
    for (int b = 0; b < B; ++b) no_throw(oom, [&] {
      row.need();
      other.need();
      for (int i = P.own_off[b]; i < P.own_off[b + 1]; ++i)
        for (int64_t q = hm.rowptr[P.row[i]]; q < hm.rowptr[P.row[i] + 1]; ++q) {
          const int32_t c = hm.col[q], o = part[c];
          if (o == b) continue;
          border[P.row[i]] = 1;
          if (!row[c]) P.halo[b].push_back(c);
          if (!other[o]) reads[b].push_back(o);
          row[c] = other[o] = 1;
        }
      for (int32_t c : P.halo[b]) row[c] = 0;
      for (int32_t o : reads[b]) other[o] = 0;
      std::sort(P.halo[b].begin(), P.halo[b].end());
      std::sort(reads[b].begin(), reads[b].end());
    });
  }
  if (oom) return MG_ERR_OOM;
  for (int b = 0; b < B; ++b) {
    for (int32_t o : reads[b])
      if (!std::binary_search(reads[o].begin(), reads[o].end(), b)) return MG_ERR_UNSUPPORTED;
    for (int32_t r : P.halo[b]) border[r] = 1;
  }
  P.n_border.assign(B, 0);
#pragma omp parallel for schedule(dynamic, 4)
  for (int b = 0; b < B; ++b) {
    // border rows first, each kind by falling row length: a warp's rows then
    // have nearly the same length
    int32_t *r0 = P.row.data() + P.own_off[b], *r1 = P.row.data() + P.own_off[b + 1];
    std::stable_sort(r0, r1, [&](int32_t x, int32_t y) {
      if (border[x] != border[y]) return border[x] > border[y];
      return hm.rowptr[x + 1] - hm.rowptr[x] > hm.rowptr[y + 1] - hm.rowptr[y];
    });
    for (int32_t* r = r0; r < r1; ++r) P.n_border[b] += border[*r];
  }
  P.part = std::move(part);
  return MG_OK;
}

void group_rows(const HostMesh& hm, const HostPatches& P, int rpw, HostGroups& G) {
  G = HostGroups();
  const int B = P.B;
  std::vector<int32_t> slot(hm.n, -1), xrow(hm.n, -1);   // slot in its patch, exchange row
  G.grp_off.assign(B + 1, 0);
  G.border.assign(B, 0);
  G.pair_off.assign(B + 1, 0);
  G.halo_off.assign(B + 1, 0);
  G.x_off.assign(B + 1, 0);
  for (int b = 0; b < B; ++b) {
    const int n = P.own_off[b + 1] - P.own_off[b], nb = P.n_border[b];
    const int gb = (nb + rpw - 1) / rpw, gi = (n - nb + rpw - 1) / rpw;
    const int h = (int)P.halo[b].size();
    G.border[b] = gb;
    G.grp_off[b + 1] = G.grp_off[b] + gb + gi;
    G.x_off[b + 1] = G.x_off[b] + gb * rpw;
    G.halo_off[b + 1] = G.halo_off[b] + h;
    G.max_groups = std::max(G.max_groups, gi + gb);
    G.max_halo = std::max(G.max_halo, h);
    G.max_slots = std::max(G.max_slots, (gi + gb) * rpw + h);
  }
  const int ngr = G.grp_off[B];
  std::vector<int32_t> np(ngr);                          // pairs per row of every group
  G.row.resize((size_t)ngr * rpw);
  G.diag.resize((size_t)ngr * rpw);
#pragma omp parallel for schedule(dynamic, 4)
  for (int b = 0; b < B; ++b) {
    const int32_t* own = P.row.data() + P.own_off[b];
    const int n = P.own_off[b + 1] - P.own_off[b], nb = P.n_border[b], gb = G.border[b];
    for (int g = 0; g < G.grp_off[b + 1] - G.grp_off[b]; ++g) {
      int w = 0;
      for (int k = 0; k < rpw; ++k) {
        const int i = g < gb ? g * rpw + k : nb + (g - gb) * rpw + k;
        const int32_t r = i < (g < gb ? nb : n) ? own[i] : -1;
        const size_t s = (size_t)(G.grp_off[b] + g) * rpw + k;
        G.row[s] = r;
        G.diag[s] = r < 0 ? 0.0f : (float)hm.val[hm.rowptr[r]];
        if (r < 0) continue;
        slot[r] = g * rpw + k;
        if (g < gb) xrow[r] = G.x_off[b] + slot[r];
        w = std::max(w, (int)(hm.rowptr[r + 1] - hm.rowptr[r]) - 1);
      }
      np[G.grp_off[b] + g] = (w + 1) / 2;
    }
  }
  // rows of nearly equal length (triangles: 6 neighbours): the same number of
  // pairs for every row, so that the kernel's product is straight code
  const int most = *std::max_element(np.begin(), np.end());
  const int64_t total = std::accumulate(np.begin(), np.end(), (int64_t)0);
  if (most == 3 && 8 * total >= 7 * (int64_t)most * ngr) {
    G.uniform = most;
    std::fill(np.begin(), np.end(), most);
  }
  G.hdr.resize(ngr);
  for (int b = 0; b < B; ++b) {
    int at = 0;
    for (int g = G.grp_off[b]; g < G.grp_off[b + 1]; ++g) {
      G.hdr[g] = at | np[g] << kPairShift;
      at += np[g] * rpw;
    }
    G.pair_off[b + 1] = G.pair_off[b] + at;
    G.max_pairs = std::max(G.max_pairs, at);
  }
  G.pair.resize(G.pair_off[B]);
  G.halo.resize(G.halo_off[B]);
  G.halo_x.resize(G.halo_off[B]);
#pragma omp parallel for schedule(dynamic, 4)
  for (int b = 0; b < B; ++b) {
    const int own = (G.grp_off[b + 1] - G.grp_off[b]) * rpw;
    const std::vector<int32_t>& h = P.halo[b];
    for (size_t i = 0; i < h.size(); ++i) {
      G.halo[G.halo_off[b] + i] = h[i];
      G.halo_x[G.halo_off[b] + i] = xrow[h[i]];
    }
    HostGroups::Pair* at = G.pair.data() + G.pair_off[b];
    for (int g = G.grp_off[b]; g < G.grp_off[b + 1]; ++g)
      for (int p = 0; p < np[g]; ++p)
        for (int k = 0; k < rpw; ++k) {
          const int32_t r = G.row[(size_t)g * rpw + k];
          const int me = (g - G.grp_off[b]) * rpw + k;
          HostGroups::Pair q{{me, me}, {0.0f, 0.0f}};   // padding: the slot itself, value 0
          for (int e = 0; e < 2 && r >= 0; ++e) {
            const int64_t c = hm.rowptr[r] + 1 + 2 * p + e;
            if (c >= hm.rowptr[r + 1]) break;
            const int32_t cr = hm.col[c];
            q.slot[e] = P.part[cr] == b
                            ? slot[cr]
                            : own + (int)(std::lower_bound(h.begin(), h.end(), cr) - h.begin());
            q.val[e] = (float)hm.val[c];
          }
          *at++ = q;
        }
  }
}

}  // namespace mg
