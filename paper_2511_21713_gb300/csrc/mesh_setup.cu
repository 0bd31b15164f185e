// Mesh creation: validation, topology (host) and device data.
//
// The host builds integer structure only (CSR pattern of the coupled operator's sparse
// part, element-to-slot gather lists, triangle-pair classes); every floating-point
// quantity of the discretisation is computed on the device.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "host_ranges.h"
#include "pbfb_internal.cuh"
#include "quad_tables.cuh"
#include "solid_angle.h"

namespace pbfb {

namespace {

thread_local std::string g_err;

// counting sort of the values val(e), e = 0..n-1, by keys[e] in [0, nkeys): ptr (nkeys + 1) and the values, in
// ascending e within a key.  A thread takes a range of the keys and reads all of them (sequentially: a fraction of
// the scattered writes).
template <class V>
void bucket(const int* keys, int64_t n, int nkeys, V val, std::vector<int>& ptr, std::vector<int>& out) {
  ptr.assign(nkeys + 1, 0);
  out.resize(n);
  const HostRanges ranges(n < 40000 ? 1 : nkeys, n < 40000 ? 1 : std::max(1, nkeys / 16));
  auto clip = [&](int64_t& k0, int64_t& k1) {
    if (n < 40000) k0 = 0, k1 = nkeys;
  };
  ranges.run([&](int, int64_t k0, int64_t k1) {
    clip(k0, k1);
    for (int64_t e = 0; e < n; ++e)
      if (keys[e] >= k0 && keys[e] < k1) ptr[keys[e] + 1]++;
  });
  for (int i = 0; i < nkeys; ++i) ptr[i + 1] += ptr[i];
  std::vector<int> pos(ptr.begin(), ptr.end() - 1);
  ranges.run([&](int, int64_t k0, int64_t k1) {
    clip(k0, k1);
    for (int64_t e = 0; e < n; ++e)
      if (keys[e] >= k0 && keys[e] < k1) out[pos[keys[e]]++] = val(e);
  });
}

struct HostSurface {
  std::vector<int> tri;    // local ids
  std::vector<int> verts;  // shell ids
  std::vector<double> P;   // nt*9 corner coordinates
  std::vector<int> iptr, inc;  // per vertex: its triangles' entries 3 t + a, ascending
};

// Triangle-pair classification (ordered pairs: test t, trial s): touching pairs (identical, common
// edge, common vertex) from the vertex incidence, near pairs (no common vertex, centroid distance
// below 2 max(h_t, h_s), h the longest edge) from a uniform grid over the centroids with cells of
// twice the median h.  A near pair is looked for from its triangle with the larger h (ties: the
// smaller index), within radius 2 h of that triangle, so every pair is found once whatever the
// spread of triangle sizes; host threads over the triangles.  Each row (test t) lists its trial
// triangles in ascending order.
// pptr: the pairs of test t are pptr[t] .. pptr[t + 1] - 1.
void classify_pairs(const HostSurface& hs, std::vector<int>& pptr, std::vector<int>& pt, std::vector<int>& ps,
                    std::vector<int>& cls, std::vector<int>& perm) {
  const int nt = (int)hs.tri.size() / 3;
  const std::vector<int>& iptr = hs.iptr;
  const std::vector<int>& inc = hs.inc;
  std::vector<double> cen(3 * (size_t)nt), h(nt);
  double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
  for (int t = 0; t < nt; ++t) {
    const double* P = &hs.P[9 * (size_t)t];
    double hh = 0.0;
    for (int d = 0; d < 3; ++d) cen[3 * (size_t)t + d] = (P[d] + P[3 + d] + P[6 + d]) / 3.0;
    for (int k = 0; k < 3; ++k) {
      const double* A = P + 3 * k;
      const double* B = P + 3 * ((k + 1) % 3);
      const double dx = B[0] - A[0], dy = B[1] - A[1], dz = B[2] - A[2];
      hh = std::max(hh, std::sqrt(dx * dx + dy * dy + dz * dz));
    }
    h[t] = hh;
    for (int d = 0; d < 3; ++d) {
      lo[d] = std::min(lo[d], cen[3 * (size_t)t + d]);
      hi[d] = std::max(hi[d], cen[3 * (size_t)t + d]);
    }
  }
  std::vector<double> hsort(h);
  std::nth_element(hsort.begin(), hsort.begin() + nt / 2, hsort.end());
  double cell = 2.0 * std::max(hsort[nt / 2], 1e-300);
  int dims[3];
  for (;;) {
    int64_t cells = 1;
    for (int d = 0; d < 3; ++d) {
      dims[d] = std::max(1, (int)std::floor((hi[d] - lo[d]) / cell) + 1);
      cells *= dims[d];
    }
    if (cells <= 8 * (int64_t)nt + 64) break;
    cell *= 2.0;
  }
  const int64_t ncell = (int64_t)dims[0] * dims[1] * dims[2];
  auto cidx = [&](double x, int d) { return std::min(dims[d] - 1, std::max(0, (int)std::floor((x - lo[d]) / cell))); };
  std::vector<int64_t> cptr(ncell + 1, 0);
  std::vector<int> ctri(nt), cof(nt);
  for (int t = 0; t < nt; ++t) {
    const double* c = &cen[3 * (size_t)t];
    cof[t] = (int)(((int64_t)cidx(c[0], 0) * dims[1] + cidx(c[1], 1)) * dims[2] + cidx(c[2], 2));
    ++cptr[cof[t] + 1];
  }
  for (int64_t k = 0; k < ncell; ++k) cptr[k + 1] += cptr[k];
  {
    std::vector<int64_t> fill(cptr.begin(), cptr.end() - 1);
    for (int t = 0; t < nt; ++t) ctri[fill[cof[t]]++] = t;
  }
  // near pairs, both orientations, from per-thread buffers merged in thread (= triangle) order
  std::vector<int> found[HOST_THREADS];
  HostRanges(nt, 32).run([&](int k, int64_t t0, int64_t t1) {
    std::vector<int> stamp(nt, -1);
    std::vector<int>& out = found[k];
    for (int t = (int)t0; t < (int)t1; ++t) {
      for (int a = 0; a < 3; ++a) {
        const int v = hs.tri[3 * t + a];
        for (int q = iptr[v]; q < iptr[v + 1]; ++q) stamp[inc[q] / 3] = t;
      }
      const double* c = &cen[3 * (size_t)t];
      const double r = 2.0 * h[t];
      int a0[3], a1[3];
      for (int d = 0; d < 3; ++d) {
        a0[d] = cidx(c[d] - r, d);
        a1[d] = cidx(c[d] + r, d);
      }
      for (int x = a0[0]; x <= a1[0]; ++x)
        for (int y = a0[1]; y <= a1[1]; ++y)
          for (int z = a0[2]; z <= a1[2]; ++z) {
            const int64_t cc = ((int64_t)x * dims[1] + y) * dims[2] + z;
            for (int64_t q = cptr[cc]; q < cptr[cc + 1]; ++q) {
              const int u = ctri[q];
              if (stamp[u] == t) continue;  // itself and the touching triangles
              if (h[u] > h[t] || (h[u] == h[t] && u < t)) continue;  // found from u's side
              const double dx = c[0] - cen[3 * (size_t)u], dy = c[1] - cen[3 * (size_t)u + 1],
                           dz = c[2] - cen[3 * (size_t)u + 2];
              if (dx * dx + dy * dy + dz * dz < r * r) {
                out.push_back(t);
                out.push_back(u);
              }
            }
          }
    }
  });
  // rows: near partners of every triangle (both orientations), counting sort by row
  std::vector<int> nptr(nt + 1, 0);
  for (const auto& f : found)
    for (size_t q = 0; q < f.size(); q += 2) {
      ++nptr[f[q] + 1];
      ++nptr[f[q + 1] + 1];
    }
  for (int t = 0; t < nt; ++t) nptr[t + 1] += nptr[t];
  std::vector<int> near(nptr[nt]);
  {
    std::vector<int> fill(nptr.begin(), nptr.end() - 1);
    for (const auto& f : found)
      for (size_t q = 0; q < f.size(); q += 2) {
        near[fill[f[q]]++] = f[q + 1];
        near[fill[f[q + 1]]++] = f[q];
      }
  }
  struct Rows {
    std::vector<int> s, cls, perm;
  } rows[HOST_THREADS];
  pptr.assign(nt + 1, 0);
  const HostRanges ranges(nt, 64);
  ranges.run([&](int k, int64_t t0, int64_t t1) {
    std::vector<int> cnt(nt, 0), touched;
    std::vector<std::array<int, 2>> row;  // (s, class)
    Rows& out = rows[k];
    for (int t = (int)t0; t < (int)t1; ++t) {
      touched.clear();
      row.clear();
      for (int a = 0; a < 3; ++a) {
        const int v = hs.tri[3 * t + a];
        for (int q = iptr[v]; q < iptr[v + 1]; ++q) {
          const int u = inc[q] / 3;
          if (cnt[u] == 0) touched.push_back(u);
          cnt[u]++;
        }
      }
      for (int u : touched) {
        const int c = cnt[u];
        row.push_back({u, c == 3 ? PAIR_IDENTICAL : (c == 2 ? PAIR_EDGE : PAIR_VERTEX)});
      }
      for (int q = nptr[t]; q < nptr[t + 1]; ++q) row.push_back({near[q], PAIR_NEAR});
      std::sort(row.begin(), row.end());
      for (auto& e : row) {
        int u = e[0], c = e[1];
        int p[6] = {0, 1, 2, 0, 1, 2};
        const int* T = &hs.tri[3 * t];
        const int* S = &hs.tri[3 * u];
        if (c == PAIR_EDGE) {
          // shared vertices in the test triangle's order go to reference vertices 0 and 1
          int sh[2], ns = 0;
          for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
              if (T[a] == S[b]) sh[ns++] = a;
          int sb[2];
          for (int k = 0; k < 2; ++k)
            for (int b = 0; b < 3; ++b)
              if (S[b] == T[sh[k]]) sb[k] = b;
          p[0] = sh[0]; p[1] = sh[1]; p[2] = 3 - sh[0] - sh[1];
          p[3] = sb[0]; p[4] = sb[1]; p[5] = 3 - sb[0] - sb[1];
        } else if (c == PAIR_VERTEX) {
          int ia = 0, ib = 0;
          for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
              if (T[a] == S[b]) { ia = a; ib = b; }
          for (int k = 0; k < 3; ++k) {
            p[k] = (ia + k) % 3;
            p[3 + k] = (ib + k) % 3;
          }
        }
        out.s.push_back(u);
        out.cls.push_back(c);
        out.perm.insert(out.perm.end(), p, p + 6);
      }
      pptr[t + 1] = (int)row.size();
      for (int u : touched) cnt[u] = 0;
    }
  });
  for (int t = 0; t < nt; ++t) pptr[t + 1] += pptr[t];
  const int np = pptr[nt];
  pt.resize(np);
  ps.resize(np);
  cls.resize(np);
  perm.resize(6 * (size_t)np);
  ranges.run([&](int k, int64_t t0, int64_t t1) {
    const int p0 = pptr[t0];
    std::copy(rows[k].s.begin(), rows[k].s.end(), ps.begin() + p0);
    std::copy(rows[k].cls.begin(), rows[k].cls.end(), cls.begin() + p0);
    std::copy(rows[k].perm.begin(), rows[k].perm.end(), perm.begin() + 6 * (size_t)p0);
    for (int64_t t = t0; t < t1; ++t) std::fill(pt.begin() + pptr[t], pt.begin() + pptr[t + 1], (int)t);
  });
}


int build_surface(Mesh* m, Surface* s, const std::vector<int>& gtri, const std::vector<double>& xyz_h) {
  const int nt = (int)gtri.size() / 3;
  std::vector<int> verts(gtri.begin(), gtri.end());
  std::sort(verts.begin(), verts.end());
  verts.erase(std::unique(verts.begin(), verts.end()), verts.end());
  std::unordered_map<int, int> loc;
  for (int i = 0; i < (int)verts.size(); ++i) loc[verts[i]] = i;
  HostSurface hs;
  hs.verts = verts;
  hs.tri.resize(gtri.size());
  hs.P.resize(9 * (size_t)nt);
  double c[3] = {0, 0, 0};
  for (int t = 0; t < nt; ++t)
    for (int a = 0; a < 3; ++a) {
      int g = gtri[3 * t + a];
      hs.tri[3 * t + a] = loc[g];
      for (int d = 0; d < 3; ++d) hs.P[9 * t + 3 * a + d] = xyz_h[3 * (size_t)g + d];
    }
  for (int v : verts)
    for (int d = 0; d < 3; ++d) c[d] += xyz_h[3 * (size_t)v + d];
  for (int d = 0; d < 3; ++d) s->ctr[d] = c[d] / verts.size();
  {
    // largest vertex distance from the centre: the quadrature points lie within the triangles (float-float
    // coordinates, ff_grid)
    double rmax = 0.0;
    for (int v : verts) {
      double r2 = 0.0;
      for (int d = 0; d < 3; ++d) {
        const double x = xyz_h[3 * (size_t)v + d] - s->ctr[d];
        r2 += x * x;
      }
      rmax = std::max(rmax, std::sqrt(r2));
    }
    s->rmax = rmax;
  }
  s->nt = nt;
  s->nv = (int)verts.size();
  s->nq = QS * nt;
  s->tri_h = hs.tri;
  s->vmap_h = verts;
  PB_TRY(s->tri.upload(hs.tri.data(), hs.tri.size(), m->stream));
  PB_TRY(s->vmap.upload(verts.data(), verts.size(), m->stream));
  // test-reduction incidence: per vertex (t*3 + a)
  bucket(hs.tri.data(), 3 * (int64_t)nt, s->nv, [](int64_t e) { return (int)e; }, hs.iptr, hs.inc);
  PB_TRY(s->inc_ptr.upload(hs.iptr.data(), hs.iptr.size(), m->stream));
  PB_TRY(s->inc_idx.upload(hs.inc.data(), hs.inc.size(), m->stream));
  // special pairs and the correction pattern
  std::vector<int> pptr, pt, ps, cls, perm;
  classify_pairs(hs, pptr, pt, ps, cls, perm);
  s->npair = (int)pt.size();
  PB_TRY(s->pair_t.upload(pt.data(), pt.size(), m->stream));
  PB_TRY(s->pair_s.upload(ps.data(), ps.size(), m->stream));
  PB_TRY(s->pair_cls.upload(cls.data(), cls.size(), m->stream));
  PB_TRY(s->pair_perm.upload(perm.data(), perm.size(), m->stream));
  {
    // entry e = 9 p + 3 a + b of pair p couples test vertex tri[pt[p]][a] and trial vertex
    // tri[ps[p]][b]: row i's entries are those of its triangles' pairs, in ascending order
    auto entries = [&](int i, auto f) {  // f(entry, trial vertex)
      for (int q = hs.iptr[i]; q < hs.iptr[i + 1]; ++q) {
        const int t = hs.inc[q] / 3, a = hs.inc[q] % 3;
        for (int p = pptr[t]; p < pptr[t + 1]; ++p)
          for (int b = 0; b < 3; ++b) f(9 * p + 3 * a + b, hs.tri[3 * (size_t)ps[p] + b]);
      }
    };
    // sizes, and the distinct columns (a marker per column), sorted
    std::vector<int> dptr(s->nv + 1, 0), eptr(s->nv + 1, 0), cols[HOST_THREADS];
    s->c_ptr_h.assign(s->nv + 1, 0);
    const HostRanges ranges(s->nv, 32);
    ranges.run([&](int k, int64_t i0, int64_t i1) {
      std::vector<int> mark(s->nv, -1);
      for (int i = (int)i0; i < (int)i1; ++i) {
        const size_t w0 = cols[k].size();
        entries(i, [&](int, int c) {
          eptr[i + 1]++;
          if (c == i) dptr[i + 1]++;
          if (mark[c] != i) {
            mark[c] = i;
            cols[k].push_back(c);
          }
        });
        std::sort(cols[k].begin() + w0, cols[k].end());
        s->c_ptr_h[i + 1] = (int)(cols[k].size() - w0);
      }
    });
    for (int i = 0; i < s->nv; ++i) {
      s->c_ptr_h[i + 1] += s->c_ptr_h[i];
      dptr[i + 1] += dptr[i];
      eptr[i + 1] += eptr[i];
    }
    s->cnnz = s->c_ptr_h[s->nv];
    s->c_col_h.resize(s->cnnz);
    std::vector<int> cgp(s->cnnz + 1), cgi(eptr[s->nv]), dgi(dptr[s->nv]);
    cgp[s->cnnz] = eptr[s->nv];
    ranges.run([&](int k, int64_t i0, int64_t i1) {
      std::copy(cols[k].begin(), cols[k].end(), s->c_col_h.begin() + s->c_ptr_h[i0]);
      std::vector<int> rank(s->nv), pos;
      for (int i = (int)i0; i < (int)i1; ++i) {
        const int c0 = s->c_ptr_h[i], n = s->c_ptr_h[i + 1] - c0;
        pos.assign(n + 1, 0);
        for (int r = 0; r < n; ++r) rank[s->c_col_h[c0 + r]] = r;
        entries(i, [&](int, int c) { pos[rank[c] + 1]++; });
        pos[0] = eptr[i];
        for (int r = 0; r < n; ++r) {
          cgp[c0 + r] = pos[r];
          pos[r + 1] += pos[r];
        }
        int d = dptr[i];
        entries(i, [&](int e, int c) {
          cgi[pos[rank[c]]++] = e;
          if (c == i) dgi[d++] = e;
        });
      }
    });
    PB_TRY(s->cg_ptr.upload(cgp.data(), cgp.size(), m->stream));
    PB_TRY(s->cg_idx.upload(cgi.data(), cgi.size(), m->stream));
    PB_TRY(s->dg_ptr.upload(dptr.data(), dptr.size(), m->stream));
    PB_TRY(s->dg_idx.upload(dgi.data(), dgi.size(), m->stream));
    PB_TRY(s->c_ptr.upload(s->c_ptr_h.data(), s->c_ptr_h.size(), m->stream));
    PB_TRY(s->c_col.upload(s->c_col_h.data(), s->c_col_h.size(), m->stream));
  }
  PB_TRY(s->qx.alloc(3 * (size_t)s->nq));
  PB_TRY(s->qw.alloc(s->nq));
  PB_TRY(s->nrm.alloc(3 * (size_t)nt));
  PB_TRY(s->area.alloc(nt));
  PB_TRY(s->qpf.alloc(s->nq));
  PB_TRY(s->pairV.alloc(9 * (size_t)s->npair));
  PB_TRY(s->pairK.alloc(9 * (size_t)s->npair));
  PB_TRY(s->pairVfull.alloc(9 * (size_t)s->npair));
  PB_TRY(s->corrV.alloc(s->cnnz));
  PB_TRY(s->corrK.alloc(s->cnnz));
  PB_TRY(s->mass.alloc(s->cnnz));
  PB_TRY(s->diagV.alloc(s->nv));
  PB_TRY(s->spos.alloc(s->nq));
  PB_TRY(s->sdl.alloc(s->nq));
  // far-field partial-sum buffer: enough source splits for every launch shape of launch_bem_far
  PB_TRY(s->val.alloc(far_splits_max(s->nq) * (size_t)s->nq));
  return PBFB_OK;
}

uint64_t key2(int r, int c) { return ((uint64_t)(uint32_t)r << 32) | (uint32_t)c; }

}  // namespace

void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
}

const char* last_error() { return g_err.c_str(); }

// Validation of the shell mesh and its two boundary surfaces (host).
// With region (per tet 0 = Omega_m, 1 = Omega_i), Gamma_m must be the interface between the two
// regions (interior faces, normal into Omega_i) and Gamma_s the whole boundary.
static int validate(const double* xyz, int nv, const int* tets, int64_t nt, const int* gm, int ngm, const int* gs,
                    int ngs, const int* region) {
  if (!xyz || !tets || !gm || !gs || nv < 4 || nt < 1 || ngm < 4 || ngs < 4) {
    set_error("mesh_create: empty or missing arrays");
    return PBFB_ERR_INVALID;
  }
  if (nt > (int64_t(1) << 29)) {
    set_error("mesh_create: more than 2^29 tetrahedra");
    return PBFB_ERR_INVALID;
  }
  for (int64_t i = 0; i < 3 * (int64_t)nv; ++i)
    if (!std::isfinite(xyz[i])) {
      set_error("mesh_create: non-finite coordinate");
      return PBFB_ERR_INVALID;
    }
  for (int64_t i = 0; i < 4 * nt; ++i)
    if (tets[i] < 0 || tets[i] >= nv) {
      set_error("mesh_create: tet vertex id out of range");
      return PBFB_ERR_INVALID;
    }
  if (region) {
    int64_t cnt[2] = {0, 0};
    for (int64_t t = 0; t < nt; ++t) {
      if (region[t] != 0 && region[t] != 1) {
        set_error("mesh_create: tet region must be 0 (Omega_m) or 1 (Omega_i)");
        return PBFB_ERR_INVALID;
      }
      cnt[region[t]]++;
    }
    if (!cnt[0] || !cnt[1]) {
      set_error("mesh_create: both Omega_m and Omega_i need tets");
      return PBFB_ERR_INVALID;
    }
  }
  for (int i = 0; i < 3 * ngm; ++i)
    if (gm[i] < 0 || gm[i] >= nv) {
      set_error("mesh_create: Gamma_m vertex id out of range");
      return PBFB_ERR_INVALID;
    }
  for (int i = 0; i < 3 * ngs; ++i)
    if (gs[i] < 0 || gs[i] >= nv) {
      set_error("mesh_create: Gamma_s vertex id out of range");
      return PBFB_ERR_INVALID;
    }
  // boundary faces of the tets: faces used once, with the opposite vertex for orientation.
  // Face 4 t + k by its smallest vertex, then sorted by the other two (one number) within a bucket.
  struct Face {
    uint64_t key;
    int id;
    bool operator<(const Face& o) const { return key != o.key ? key < o.key : id < o.id; }
  };
  std::vector<int> fkey(4 * (size_t)nt);
  std::vector<uint64_t> fother(4 * (size_t)nt);
  int64_t degenerate[HOST_THREADS];
  std::fill(degenerate, degenerate + HOST_THREADS, nt);
  HostRanges(nt, 4096).run([&](int th, int64_t t0, int64_t t1) {
    for (int64_t t = t0; t < t1; ++t) {
      const int* T = tets + 4 * t;
      double e[3][3];
      for (int k = 0; k < 3; ++k)
        for (int d = 0; d < 3; ++d) e[k][d] = xyz[3 * T[k + 1] + d] - xyz[3 * T[0] + d];
      double det = e[0][0] * (e[1][1] * e[2][2] - e[1][2] * e[2][1]) -
                   e[0][1] * (e[1][0] * e[2][2] - e[1][2] * e[2][0]) +
                   e[0][2] * (e[1][0] * e[2][1] - e[1][1] * e[2][0]);
      double L2 = 0.0;
      for (int k = 0; k < 3; ++k) L2 = std::max(L2, e[k][0] * e[k][0] + e[k][1] * e[k][1] + e[k][2] * e[k][2]);
      if (!(std::fabs(det) > 1e-12 * L2 * std::sqrt(L2))) {
        degenerate[th] = t;
        return;
      }
      for (int k = 0; k < 4; ++k) {
        std::array<int, 3> f;
        int q = 0;
        for (int a = 0; a < 4; ++a)
          if (a != k) f[q++] = T[a];
        std::sort(f.begin(), f.end());
        fkey[4 * t + k] = f[0];
        fother[4 * t + k] = key2(f[1], f[2]);
      }
    }
  });
  const int64_t bad = *std::min_element(degenerate, degenerate + HOST_THREADS);
  if (bad < nt) {
    set_error("mesh_create: degenerate tetrahedron %lld", (long long)bad);
    return PBFB_ERR_INVALID;
  }
  std::vector<int> fptr, ford;
  bucket(fkey.data(), 4 * nt, nv, [](int64_t e) { return (int)e; }, fptr, ford);
  std::vector<Face> face(ford.size());
  // per sorted face position: multiplicity of its triple (1 boundary, 2 interior)
  std::vector<char> fcount(ford.size(), 0);
  size_t nbs[HOST_THREADS] = {}, nifs[HOST_THREADS] = {};
  bool more[HOST_THREADS] = {};
  HostRanges(nv, 512).run([&](int th, int64_t v0, int64_t v1) {
    for (size_t q = fptr[v0]; q < (size_t)fptr[v1]; ++q) face[q] = {fother[ford[q]], ford[q]};
    for (int64_t v = v0; v < v1; ++v) {
      std::sort(face.begin() + fptr[v], face.begin() + fptr[v + 1]);
      for (size_t a = fptr[v]; a < (size_t)fptr[v + 1];) {
        size_t b = a + 1;
        while (b < (size_t)fptr[v + 1] && face[b].key == face[a].key) ++b;
        if (b - a > 2) more[th] = true;
        if (b - a == 1) nbs[th]++;
        if (b - a == 2 && region && region[face[a].id / 4] != region[face[a + 1].id / 4]) nifs[th]++;
        for (size_t c = a; c < b; ++c) fcount[c] = (char)std::min<size_t>(b - a, 3);
        a = b;
      }
    }
  });
  size_t nb = 0, nif = 0;
  for (int th = 0; th < HOST_THREADS; ++th) {
    if (more[th]) {
      set_error("mesh_create: a face is shared by more than two tets");
      return PBFB_ERR_INVALID;
    }
    nb += nbs[th];
    nif += nifs[th];
  }
  if (!region && nb != (size_t)ngm + (size_t)ngs) {
    set_error("mesh_create: %zu boundary faces but %d + %d surface triangles", nb, ngm, ngs);
    return PBFB_ERR_INVALID;
  }
  if (region && (nb != (size_t)ngs || nif != (size_t)ngm)) {
    set_error("mesh_create: %zu boundary faces and %zu Omega_m/Omega_i faces but %d Gamma_s and %d Gamma_m "
              "triangles", nb, nif, ngs, ngm);
    return PBFB_ERR_INVALID;
  }
  // position of the face with this sorted triple, or -1
  auto find_face = [&](const std::array<int, 3>& f) -> long long {
    auto b = face.begin() + fptr[f[0]], e = face.begin() + fptr[f[0] + 1];
    auto it = std::lower_bound(b, e, Face{key2(f[1], f[2]), -1});
    if (it == e || it->key != key2(f[1], f[2])) return -1;
    return (long long)(it - face.begin());
  };
  std::vector<char> onm(nv, 0), ons(nv, 0);
  for (int surf = 0; surf < 2; ++surf) {
    const int* tri = surf == 0 ? gm : gs;
    int ntri = surf == 0 ? ngm : ngs;
    // directed edges (vertex pairs) in an open table of at most a quarter's load; 0 is no pair of distinct ids + 1
    size_t slots = 64;
    while (slots < 12 * (size_t)ntri) slots *= 2;
    std::vector<uint64_t> edges(slots, 0);
    auto edge = [&](int a, int b) -> uint64_t& {  // the pair's entry or the free one for it
      const uint64_t key = key2(a + 1, b + 1);
      size_t q = (key * 0x9E3779B97F4A7C15ull) >> 20 & (slots - 1);
      while (edges[q] != 0 && edges[q] != key) q = (q + 1) & (slots - 1);
      return edges[q];
    };
    for (int t = 0; t < ntri; ++t) {
      const int* F = tri + 3 * t;
      if (F[0] == F[1] || F[1] == F[2] || F[0] == F[2]) {
        set_error("mesh_create: repeated vertex in a surface triangle");
        return PBFB_ERR_INVALID;
      }
      std::array<int, 3> f = {F[0], F[1], F[2]};
      std::sort(f.begin(), f.end());
      const long long pos = find_face(f);
      const bool interface = region && surf == 0;  // Gamma_m between the regions
      if (interface) {
        if (pos < 0 || fcount[pos] != 2 || region[face[pos].id / 4] == region[face[pos + 1].id / 4]) {
          set_error("mesh_create: Gamma_m triangle %d is not a face between Omega_m and Omega_i tets", t);
          return PBFB_ERR_INVALID;
        }
      } else if (pos < 0 || fcount[pos] != 1) {
        set_error("mesh_create: surface triangle %d of %s is not a boundary face of the tets", t,
                  surf == 0 ? "Gamma_m" : "Gamma_s");
        return PBFB_ERR_INVALID;
      }
      fcount[pos] = 3;  // claimed
      // orientation: the opposite tet vertex lies on the positive side for Gamma_m (of the
      // Omega_i tet for an interface), on the negative side for Gamma_s
      const int fid = face[interface && region[face[pos].id / 4] != 1 ? pos + 1 : pos].id;
      int o = tets[fid];
      double a[3], b[3], c[3];
      for (int d = 0; d < 3; ++d) {
        a[d] = xyz[3 * F[1] + d] - xyz[3 * F[0] + d];
        b[d] = xyz[3 * F[2] + d] - xyz[3 * F[0] + d];
        c[d] = xyz[3 * o + d] - xyz[3 * F[0] + d];
      }
      double n[3] = {a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]};
      double side = n[0] * c[0] + n[1] * c[1] + n[2] * c[2];
      if ((surf == 0 && !(side > 0)) || (surf == 1 && !(side < 0))) {
        set_error("mesh_create: %s triangle %d has the wrong orientation", surf == 0 ? "Gamma_m" : "Gamma_s", t);
        return PBFB_ERR_INVALID;
      }
      for (int k = 0; k < 3; ++k) {
        uint64_t& e = edge(F[k], F[(k + 1) % 3]);
        if (e != 0) {
          set_error("mesh_create: surface is not consistently oriented / manifold");
          return PBFB_ERR_INVALID;
        }
        e = key2(F[k] + 1, F[(k + 1) % 3] + 1);
        (surf == 0 ? onm : ons)[F[k]] = 1;
      }
    }
    for (int t = 0; t < ntri; ++t)
      for (int k = 0; k < 3; ++k)
        if (edge(tri[3 * t + (k + 1) % 3], tri[3 * t + k]) == 0) {
          set_error("mesh_create: %s is not closed", surf == 0 ? "Gamma_m" : "Gamma_s");
          return PBFB_ERR_INVALID;
        }
  }
  for (int v = 0; v < nv; ++v)
    if (onm[v] && ons[v]) {
      set_error("mesh_create: Gamma_m and Gamma_s share vertex %d", v);
      return PBFB_ERR_INVALID;
    }
  return PBFB_OK;
}

// Uniform grid over the bounding boxes of the Omega_m tets (about four tets per cell), each cell
// listing, in ascending order, the tets whose box meets it: a point's candidates are its cell's.
static void build_charge_grid(Mesh* m, const std::vector<int>& tm) {
  const int64_t nt = (int64_t)tm.size() / 4;
  double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
  for (int64_t k = 0; k < 4 * nt; ++k)
    for (int d = 0; d < 3; ++d) {
      lo[d] = std::min(lo[d], m->grid_xyz[3 * (size_t)tm[k] + d]);
      hi[d] = std::max(hi[d], m->grid_xyz[3 * (size_t)tm[k] + d]);
    }
  double vol = 1.0;
  for (int d = 0; d < 3; ++d) vol *= std::max(hi[d] - lo[d], 1e-12);
  double h = std::cbrt(vol / std::max<int64_t>(1, nt / 4));
  int dim[3];
  for (int d = 0; d < 3; ++d) dim[d] = std::max(1, std::min(1024, (int)std::ceil((hi[d] - lo[d]) / h)));
  for (int d = 0; d < 3; ++d) {
    m->cell_lo[d] = lo[d];
    m->cell_dim[d] = dim[d];
  }
  m->cell_h = h;
  auto cell_range = [&](int64_t t, int* c0, int* c1) {
    for (int d = 0; d < 3; ++d) {
      double a = 1e300, b = -1e300;
      for (int v = 0; v < 4; ++v) {
        a = std::min(a, m->grid_xyz[3 * (size_t)tm[4 * t + v] + d]);
        b = std::max(b, m->grid_xyz[3 * (size_t)tm[4 * t + v] + d]);
      }
      c0[d] = std::max(0, std::min(dim[d] - 1, (int)std::floor((a - lo[d]) / h)));
      c1[d] = std::max(0, std::min(dim[d] - 1, (int)std::floor((b - lo[d]) / h)));
    }
  };
  const size_t ncell = (size_t)dim[0] * dim[1] * dim[2];
  m->cell_ptr.assign(ncell + 1, 0);
  int c0[3], c1[3];
  for (int pass = 0; pass < 2; ++pass) {
    std::vector<int> pos;
    if (pass == 1) {
      for (size_t c = 0; c < ncell; ++c) m->cell_ptr[c + 1] += m->cell_ptr[c];
      m->cell_tet.assign(m->cell_ptr[ncell], 0);
      pos.assign(m->cell_ptr.begin(), m->cell_ptr.end() - 1);
    }
    for (int64_t t = 0; t < nt; ++t) {
      cell_range(t, c0, c1);
      for (int i = c0[0]; i <= c1[0]; ++i)
        for (int j = c0[1]; j <= c1[1]; ++j)
          for (int k = c0[2]; k <= c1[2]; ++k) {
            const size_t c = ((size_t)i * dim[1] + j) * dim[2] + k;
            if (pass == 0)
              m->cell_ptr[c + 1]++;
            else
              m->cell_tet[pos[c]++] = (int)t;
          }
    }
  }
}

int point_load(Mesh* m, const double* q_xyz, const double* z, int nq, std::vector<double>& rho) {
  rho.assign(m->nv, 0.0);
  const std::vector<int>& tm = m->tets_m_h;
  const std::vector<double>& X = m->grid_xyz;
  for (int k = 0; k < nq; ++k) {
    const double* x = q_xyz + 3 * (size_t)k;
    // the cell, clamped like the tets' boxes (a point outside every box meets no tet there)
    int c[3];
    bool finite = true;
    for (int d = 0; d < 3; ++d) {
      const double f = std::floor((x[d] - m->cell_lo[d]) / m->cell_h);
      if (!std::isfinite(f)) finite = false;
      c[d] = finite ? (int)std::max(0.0, std::min((double)(m->cell_dim[d] - 1), f)) : 0;
    }
    int found = -1;
    double lam[4] = {0, 0, 0, 0};
    if (finite) {
      const size_t cell = ((size_t)c[0] * m->cell_dim[1] + c[1]) * m->cell_dim[2] + c[2];
      for (int q = m->cell_ptr[cell]; q < m->cell_ptr[cell + 1] && found < 0; ++q) {
        const int t = m->cell_tet[q];
        const int* T = &tm[4 * (size_t)t];
        // barycentric coordinates by Cramer's rule on the edge matrix E (columns x_a - x_0)
        double e[3][3], r[3];
        for (int d = 0; d < 3; ++d) {
          for (int a = 0; a < 3; ++a) e[d][a] = X[3 * (size_t)T[a + 1] + d] - X[3 * (size_t)T[0] + d];
          r[d] = x[d] - X[3 * (size_t)T[0] + d];
        }
        auto det3 = [](double a[3][3]) {
          return a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0]) +
                 a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]);
        };
        const double det = det3(e);
        double l[4];
        for (int a = 0; a < 3; ++a) {
          double ea[3][3];
          for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) ea[i][j] = j == a ? r[i] : e[i][j];
          l[a + 1] = det3(ea) / det;
        }
        l[0] = 1.0 - l[1] - l[2] - l[3];
        if (std::min(std::min(l[0], l[1]), std::min(l[2], l[3])) >= -1e-12) {
          found = t;
          for (int a = 0; a < 4; ++a) lam[a] = l[a];
        }
      }
    }
    if (found < 0) {
      set_error("charges_set: charge %d lies in no tet of Omega_m", k);
      return PBFB_ERR_INVALID;
    }
    for (int a = 0; a < 4; ++a) rho[tm[4 * (size_t)found + a]] += z[k] * lam[a];
  }
  return PBFB_OK;
}

static double ms_since(std::chrono::steady_clock::time_point t0) {
  return std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
}

int mesh_create(const double* xyz, int nv, const int* tets, int64_t nt, const int* gm, int ngm, const int* gs,
                int ngs, cudaStream_t stream, Mesh** out, const int* region) {
  auto tc = std::chrono::steady_clock::now();
  PB_TRY(validate(xyz, nv, tets, nt, gm, ngm, gs, ngs, region));
  // tets of Omega_i (all of a shell mesh) and of Omega_m, AoS, in input order
  std::vector<int> ti_h, tm_h;
  if (region) {
    for (int64_t t = 0; t < nt; ++t) {
      std::vector<int>& dst = region[t] ? ti_h : tm_h;
      dst.insert(dst.end(), tets + 4 * t, tets + 4 * t + 4);
    }
  }
  const int* ti = region ? ti_h.data() : tets;
  const int64_t nti = region ? (int64_t)ti_h.size() / 4 : nt;
  const int64_t ntm = (int64_t)tm_h.size() / 4;
  const double t_validate = ms_since(tc);
  tc = std::chrono::steady_clock::now();
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    set_error("no CUDA device");
    return PBFB_ERR_CUDA;
  }
  PB_TRY(init_quadrature());
  PB_TRY(init_dense_attributes());
  PB_TRY(init_pair_attributes());
  PB_TRY(init_pcg_attributes());
  Mesh* m = new Mesh();
  int st = PBFB_OK;
  auto fail = [&](int s) {
    delete m;
    return s;
  };
  cudaGetDevice(&m->dev);
  m->stream = stream;
  m->nv = nv;
  m->nt = nti;
  m->nt_m = ntm;
  m->full = region != nullptr;
  std::vector<double> xyz_h(xyz, xyz + 3 * (size_t)nv);
  {
    std::vector<double> soa(3 * (size_t)nv);
    for (int v = 0; v < nv; ++v)
      for (int d = 0; d < 3; ++d) soa[(size_t)d * nv + v] = xyz[3 * (size_t)v + d];
    if ((st = m->xyz.upload(soa.data(), soa.size(), stream))) return fail(st);
    for (int r = 0; r < (ntm ? 2 : 1); ++r) {
      const int* src = r == 0 ? ti : tm_h.data();
      const int64_t cnt = r == 0 ? nti : ntm;
      std::vector<int> tsoa(4 * (size_t)cnt);
      for (int64_t t = 0; t < cnt; ++t)
        for (int a = 0; a < 4; ++a) tsoa[(size_t)a * cnt + t] = src[4 * t + a];
      if ((st = (r == 0 ? m->tets : m->tets_m).upload(tsoa.data(), tsoa.size(), stream))) return fail(st);
    }
  }
  std::vector<int> gmv(gm, gm + 3 * (size_t)ngm), gsv(gs, gs + 3 * (size_t)ngs);
  {
    // the two surfaces are independent: Gamma_s on a second host thread (its own error text)
    int st_s = PBFB_OK;
    std::string err_s;
    std::thread th([&] {
      cudaSetDevice(m->dev);
      st_s = build_surface(m, &m->ss, gsv, xyz_h);
      if (st_s != PBFB_OK) err_s = last_error();
    });
    st = build_surface(m, &m->sm, gmv, xyz_h);
    th.join();
    if (st) return fail(st);
    if (st_s) {
      set_error("%s", err_s.c_str());
      return fail(st_s);
    }
  }
  Surface& sm = m->sm;
  Surface& ss = m->ss;
  m->setup_ms[0] = t_validate;
  m->setup_ms[1] = ms_since(tc);
  tc = std::chrono::steady_clock::now();
  sm.col0 = nv;
  ss.col0 = nv + sm.nv;
  m->n = nv + sm.nv + ss.nv;
  // the surfaces' device geometry and Gamma_m's corrections run while the host builds the pattern below (whose uploads
  // wait for them: 2880 triangles, 6.6 ms of GPU time beside 5.7 ms of the host's)
  if ((st = m->red2.alloc(9 * (size_t)std::max(sm.npair, ss.npair)))) return fail(st);
  if ((st = launch_surface_geometry(m, &sm))) return fail(st);
  if ((st = launch_surface_geometry(m, &ss))) return fail(st);
  if ((st = launch_pair_corrections(m, &sm, 0.0))) return fail(st);
  // ---- sparse-part pattern of the coupled operator, row by row: a FEM row has the vertices of its tets, then the
  // surface unknowns of the vertices it shares a triangle with (mass coupling; an interior Gamma_m couples nothing:
  // its lam_m rows are the identity)
  const int* tt[2] = {ti, tm_h.data()};
  const int64_t tn[2] = {nti, ntm};
  std::vector<int> vptr[2], vtet[2];  // per vertex and region: its tets' entries 4 t + a, ascending
  for (int r = 0; r < 2; ++r) bucket(tt[r], 4 * tn[r], nv, [](int64_t e) { return (int)e; }, vptr[r], vtet[r]);
  // per surface: the mass pattern's rows (vertices sharing a triangle), and the surface's vertex at a mesh vertex
  std::vector<int> mptr[2], mcol[2];
  std::vector<int> at[2] = {std::vector<int>(nv, -1), std::vector<int>(nv, -1)};
  for (int si = 0; si < 2; ++si) {
    const Surface& s = si == 0 ? sm : ss;
    mptr[si].assign(s.nv + 1, 0);
    if (si == 0 && m->full) continue;
    std::vector<int> ip, ie;
    bucket(s.tri_h.data(), 3 * (int64_t)s.nt, s.nv, [](int64_t e) { return (int)e; }, ip, ie);
    std::vector<int> row;
    for (int i = 0; i < s.nv; ++i) {
      at[si][s.vmap_h[i]] = i;
      row.clear();
      for (int q = ip[i]; q < ip[i + 1]; ++q)
        for (int b = 0; b < 3; ++b) row.push_back(s.tri_h[3 * (size_t)(ie[q] / 3) + b]);
      std::sort(row.begin(), row.end());
      row.erase(std::unique(row.begin(), row.end()), row.end());
      mcol[si].insert(mcol[si].end(), row.begin(), row.end());
      mptr[si][i + 1] = (int)mcol[si].size();
    }
  }
  // row sizes; the FEM columns, distinct (a marker per column) and sorted
  std::vector<int> cols[HOST_THREADS];
  m->s_ptr_h.assign(m->n + 1, 0);
  const HostRanges ranges(nv, 256);
  ranges.run([&](int k, int64_t v0, int64_t v1) {
    std::vector<int> mark(nv, -1);
    std::vector<int>& out = cols[k];
    for (int v = (int)v0; v < (int)v1; ++v) {
      const size_t w0 = out.size();
      for (int r = 0; r < 2; ++r)
        for (int q = vptr[r][v]; q < vptr[r][v + 1]; ++q) {
          const int* T = tt[r] + 4 * (int64_t)(vtet[r][q] / 4);
          for (int b = 0; b < 4; ++b)
            if (mark[T[b]] != v) {
              mark[T[b]] = v;
              out.push_back(T[b]);
            }
        }
      std::sort(out.begin() + w0, out.end());
      int len = (int)(out.size() - w0);
      for (int si = 0; si < 2; ++si)
        if (const int i = at[si][v]; i >= 0) len += mptr[si][i + 1] - mptr[si][i];
      m->s_ptr_h[v + 1] = len;
    }
  });
  for (int si = 0; si < 2; ++si) {
    const Surface& s = si == 0 ? sm : ss;
    for (int i = 0; i < s.nv; ++i)
      m->s_ptr_h[s.col0 + i + 1] = si == 0 && m->full ? 1 : 2 * (s.c_ptr_h[i + 1] - s.c_ptr_h[i]);
  }
  for (int i = 0; i < m->n; ++i) m->s_ptr_h[i + 1] += m->s_ptr_h[i];
  m->snnz = m->s_ptr_h[m->n];
  m->fem_nnz = m->s_ptr_h[nv];
  m->s_col_h.resize(m->snnz);
  auto slot = [&](int r, int c) -> int {
    auto b = m->s_col_h.begin() + m->s_ptr_h[r], e = m->s_col_h.begin() + m->s_ptr_h[r + 1];
    return (int)(std::lower_bound(b, e, c) - m->s_col_h.begin());
  };
  auto cslot = [](const Surface& s, int i, int j) -> int {
    auto b = s.c_col_h.begin() + s.c_ptr_h[i], e = s.c_col_h.begin() + s.c_ptr_h[i + 1];
    return (int)(std::lower_bound(b, e, j) - s.c_col_h.begin());
  };
  std::vector<int> kind(m->snnz, 0), ref(m->snnz, 0);
  DBuf<int> jm_ptr, jm_idx;  // Omega_m stiffness gather (set-up only)
  {
    // per slot: tet-local entries (k * cnt + t) of the Omega_i tets, and of the Omega_m tets; a row's lie together
    // (four for every entry of vtet), the slots past the FEM columns have none
    std::vector<int> jp[2], ji[2];
    for (int r = 0; r < (ntm ? 2 : 1); ++r) {
      jp[r].assign(m->snnz + 1, (int)(16 * tn[r]));
      ji[r].resize(16 * tn[r]);
    }
    ranges.run([&](int k, int64_t v0, int64_t v1) {
      std::vector<int> rank(nv), pos;
      const int* src = cols[k].data();
      for (int v = (int)v0; v < (int)v1; ++v) {
        int* row = m->s_col_h.data() + m->s_ptr_h[v];
        const int s0 = m->s_ptr_h[v], len = m->s_ptr_h[v + 1] - s0;
        int nf = len, mass = 0;
        for (int si = 0; si < 2; ++si)
          if (const int i = at[si][v]; i >= 0) mass += mptr[si][i + 1] - mptr[si][i];
        nf -= mass;
        for (int q = 0; q < nf; ++q) {
          row[q] = src[q];
          rank[src[q]] = q;
        }
        src += nf;
        for (int si = 0, q = nf; si < 2; ++si)
          if (const int i = at[si][v]; i >= 0) {
            const Surface& s = si == 0 ? sm : ss;
            for (int e = mptr[si][i]; e < mptr[si][i + 1]; ++e, ++q) {
              row[q] = s.col0 + mcol[si][e];
              kind[s0 + q] = 1 + si;
              ref[s0 + q] = cslot(s, i, mcol[si][e]);
            }
          }
        for (int r = 0; r < (ntm ? 2 : 1); ++r) {
          pos.assign(nf + 1, 0);
          auto entries = [&](auto f) {  // f(column's rank, tet-local entry)
            for (int q = vptr[r][v]; q < vptr[r][v + 1]; ++q) {
              const int64_t t = vtet[r][q] / 4;
              const int a = vtet[r][q] % 4;
              for (int b = 0; b < 4; ++b) f(rank[tt[r][4 * t + b]], (int)(sym10(a, b) * tn[r] + t));
            }
          };
          entries([&](int c, int) { pos[c + 1]++; });
          pos[0] = 4 * vptr[r][v];
          for (int q = 0; q < nf; ++q) {
            jp[r][s0 + q] = pos[q];
            pos[q + 1] += pos[q];
          }
          for (int q = nf; q < len; ++q) jp[r][s0 + q] = pos[nf];
          entries([&](int c, int e) { ji[r][pos[c]++] = e; });
        }
      }
    });
    for (int r = 0; r < (ntm ? 2 : 1); ++r) {
      if ((st = (r == 0 ? m->jg_ptr : jm_ptr).upload(jp[r].data(), jp[r].size(), stream))) return fail(st);
      if ((st = (r == 0 ? m->jg_idx : jm_idx).upload(ji[r].data(), ji[r].size(), stream))) return fail(st);
    }
    for (int& e : vtet[0]) e = (int)((e % 4) * nti + e / 4);
    if ((st = m->ng_ptr.upload(vptr[0].data(), vptr[0].size(), stream))) return fail(st);
    if ((st = m->ng_idx.upload(vtet[0].data(), vtet[0].size(), stream))) return fail(st);
  }
  for (int si = 0; si < 2; ++si) {
    const Surface& s = si == 0 ? sm : ss;
    for (int i = 0; i < s.nv; ++i) {
      const int s0 = m->s_ptr_h[s.col0 + i], c0 = s.c_ptr_h[i], n = s.c_ptr_h[i + 1] - c0;
      if (m->full && si == 0) {
        m->s_col_h[s0] = s.col0 + i;
        kind[s0] = 7;
        continue;
      }
      for (int q = 0; q < n; ++q) {
        const int j = s.c_col_h[c0 + q];
        m->s_col_h[s0 + q] = s.vmap_h[j];
        m->s_col_h[s0 + n + q] = s.col0 + j;
        kind[s0 + q] = si == 0 ? 3 : 5;
        kind[s0 + n + q] = si == 0 ? 4 : 6;
        ref[s0 + q] = ref[s0 + n + q] = c0 + q;
      }
    }
  }
  {
    // Robin term of the block preconditioner: u-u slots of Gamma_s vertex pairs sharing a triangle
    std::vector<int> rs, rr;
    for (int i = 0; i < ss.nv; ++i)
      for (int e = mptr[1][i]; e < mptr[1][i + 1]; ++e) {
        rs.push_back(slot(ss.vmap_h[i], ss.vmap_h[mcol[1][e]]));
        rr.push_back(cslot(ss, i, mcol[1][e]));
      }
    m->nrobin = (int)rs.size();
    if ((st = m->robin_slot.upload(rs.data(), rs.size(), stream))) return fail(st);
    if ((st = m->robin_ref.upload(rr.data(), rr.size(), stream))) return fail(st);
    double area = 0.0;
    for (int t = 0; t < ss.nt; ++t) {
      const int* T = &ss.tri_h[3 * t];
      double a[3], b[3];
      for (int d = 0; d < 3; ++d) {
        a[d] = xyz_h[3 * (size_t)ss.vmap_h[T[1]] + d] - xyz_h[3 * (size_t)ss.vmap_h[T[0]] + d];
        b[d] = xyz_h[3 * (size_t)ss.vmap_h[T[2]] + d] - xyz_h[3 * (size_t)ss.vmap_h[T[0]] + d];
      }
      double c0 = a[1] * b[2] - a[2] * b[1], c1 = a[2] * b[0] - a[0] * b[2], c2 = a[0] * b[1] - a[1] * b[0];
      area += 0.5 * std::sqrt(c0 * c0 + c1 * c1 + c2 * c2);
    }
    m->gs_radius = std::sqrt(area / (4.0 * M_PI));
  }
  if ((st = m->s_ptr.upload(m->s_ptr_h.data(), m->s_ptr_h.size(), stream))) return fail(st);
  if ((st = m->s_col.upload(m->s_col_h.data(), m->s_col_h.size(), stream))) return fail(st);
  if ((st = m->s_kind.upload(kind.data(), kind.size(), stream))) return fail(st);
  if ((st = m->s_ref.upload(ref.data(), ref.size(), stream))) return fail(st);
  if ((st = m->s_val.alloc(m->snnz))) return fail(st);
  if ((st = m->s_base.alloc(m->snnz))) return fail(st);
  if ((st = m->a1.alloc(m->snnz))) return fail(st);
  if ((st = m->vol.alloc(nti))) return fail(st);
  if ((st = m->tloc.alloc(14 * (size_t)nti))) return fail(st);
  if ((st = m->red.alloc((size_t)152 * 7 * (OMEGA_MAX + 1) + 1024))) return fail(st);
  if ((st = m->scal.alloc(8192))) return fail(st);
  if (cudaMallocHost((void**)&m->pinned, 4096 * sizeof(double)) != cudaSuccess) {
    set_error("cudaMallocHost failed");
    return fail(PBFB_ERR_OOM);
  }
  m->setup_ms[2] = ms_since(tc);
  tc = std::chrono::steady_clock::now();
  // ---- device geometry and constant operator parts
  if ((st = launch_tet_volumes(m, m->tets.p, m->nt, m->vol.p))) return fail(st);
  if ((st = launch_stiffness_local(m, m->tets.p, m->nt, m->vol.p, m->tloc.p))) return fail(st);
  if ((st = launch_gather(m, m->snnz, m->jg_ptr.p, m->jg_idx.p, m->tloc.p, nullptr, 1.0, m->a1.p))) return fail(st);
  DBuf<double> locm;
  if (m->full) {
    if ((st = m->vol_m.alloc(ntm)) || (st = m->a1m.alloc(m->snnz)) || (st = locm.alloc(10 * (size_t)ntm)))
      return fail(st);
    if ((st = launch_tet_volumes(m, m->tets_m.p, ntm, m->vol_m.p))) return fail(st);
    if ((st = launch_stiffness_local(m, m->tets_m.p, ntm, m->vol_m.p, locm.p))) return fail(st);
    if ((st = launch_gather(m, m->snnz, jm_ptr.p, jm_idx.p, locm.p, nullptr, 1.0, m->a1m.p))) return fail(st);
    m->grid_xyz.swap(xyz_h);
    build_charge_grid(m, tm_h);
    m->tets_m_h.swap(tm_h);
  }
  sm.kappa = 0.0;
  sm.built = true;
  if (cudaStreamSynchronize(stream) != cudaSuccess) {
    set_error("mesh_create: %s", cudaGetErrorString(cudaGetLastError()));
    return fail(PBFB_ERR_CUDA);
  }
  m->setup_ms[3] = ms_since(tc);
  *out = m;
  return PBFB_OK;
}

// Generalised winding number of a closed triangulated surface at points q (n of them):
// w(x) = (1/4 pi) sum_tau Omega_tau(x), the signed solid angle of each triangle from half_solid_angle.
// With the normals pointing out of the enclosed region, w = 1 inside, 0 outside and 1/2 on the
// surface (points on a triangle are reported so).
// tri9: 9 coordinates per triangle.  Host threads over the points.
void winding_numbers(const double* tri9, size_t nt, const double* q, int nq, double* w) {
  auto work = [&](int k0, int k1) {
    for (int k = k0; k < k1; ++k) {
      const double x = q[3 * k], y = q[3 * k + 1], z = q[3 * k + 2];
      double sum = 0.0;
      bool on = false;
      for (size_t t = 0; t < nt; ++t) {
        const double* P = tri9 + 9 * t;
        const double a0 = P[0] - x, a1 = P[1] - y, a2 = P[2] - z;
        const double b0 = P[3] - x, b1 = P[4] - y, b2 = P[5] - z;
        const double c0 = P[6] - x, c1 = P[7] - y, c2 = P[8] - z;
        const double la = std::sqrt(a0 * a0 + a1 * a1 + a2 * a2);
        const double lb = std::sqrt(b0 * b0 + b1 * b1 + b2 * b2);
        const double lc = std::sqrt(c0 * c0 + c1 * c1 + c2 * c2);
        sum += 2.0 * half_solid_angle(a0, a1, a2, b0, b1, b2, c0, c1, c2, la, lb, lc, &on);
      }
      w[k] = on ? 0.5 : sum / (4.0 * M_PI);
    }
  };
  const int nth = (int)std::max(1u, std::min(16u, std::thread::hardware_concurrency()));
  if (nth == 1 || nq < 2 || (double)nq * (double)nt < 2e5) {
    work(0, nq);
    return;
  }
  const int nuse = std::min(nth, nq);
  std::vector<std::thread> th;
  for (int i = 0; i < nuse; ++i)
    th.emplace_back(work, (int)((int64_t)nq * i / nuse), (int)((int64_t)nq * (i + 1) / nuse));
  for (auto& t : th) t.join();
}

// Every charge strictly inside the closed surface (the charges of the three-region model lie in
// Omega_m, Sec. 2.1): winding number above 3/4.  w (may be null) receives the winding numbers.
int check_charges_inside(const double* tri9, size_t nt, const double* q, int nq, double* w_out) {
  std::vector<double> w(nq, 0.0);
  winding_numbers(tri9, nt, q, nq, w.data());
  if (w_out) std::copy(w.begin(), w.end(), w_out);
  for (int k = 0; k < nq; ++k)
    if (!(w[k] > 0.75)) return charge_outside(k, q + 3 * (size_t)k, w[k]);
  return PBFB_OK;
}

int charge_outside(int k, const double* q, double w) {
  set_error("charge %d at (%g, %g, %g) is not strictly inside Gamma_m (winding number %.3f)", k, q[0], q[1], q[2], w);
  return PBFB_ERR_INVALID;
}

}  // namespace pbfb

// ==================================================================== C ABI (host only)

extern "C" int pbfb_check_charges(const double* xyz, int32_t n_v, const int32_t* gm_tris, int32_t n_gm,
                                  const double* q_xyz, int32_t n_q, double* winding_out) {
  pbfb::set_error("");
  if (!xyz || !gm_tris || !q_xyz || n_v < 3 || n_gm < 4 || n_q < 1) {
    pbfb::set_error("check_charges: bad argument");
    return PBFB_ERR_INVALID;
  }
  std::vector<double> tri9(9 * (size_t)n_gm);
  for (int32_t t = 0; t < n_gm; ++t)
    for (int a = 0; a < 3; ++a) {
      const int32_t v = gm_tris[3 * (size_t)t + a];
      if (v < 0 || v >= n_v) {
        pbfb::set_error("check_charges: vertex id %d out of range", v);
        return PBFB_ERR_INVALID;
      }
      for (int d = 0; d < 3; ++d) tri9[9 * (size_t)t + 3 * a + d] = xyz[3 * (size_t)v + d];
    }
  for (int32_t k = 0; k < 3 * n_q; ++k)
    if (!std::isfinite(q_xyz[k])) {
      pbfb::set_error("check_charges: non-finite position");
      return PBFB_ERR_INVALID;
    }
  return pbfb::check_charges_inside(tri9.data(), (size_t)n_gm, q_xyz, n_q, winding_out);
}
