// Graph handle: CSR adjacency, normalised weights of D^-1/2 A D^-1/2 (Eq. gcn) and the
// nested bond neighbourhoods that bound the rows an exchange of s_i, s_j can change at
// each GCN layer.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <exception>
#include <memory>
#include <utility>
#include <vector>

#include "common.cuh"

namespace gna {

namespace {

struct HostGraph {
  int n = 0, E = 0, Lmax = 0;
  std::vector<int> row_ptr, col, col_edge, edges;
  std::vector<float> wf;
  std::vector<double> wd, J, Jz, hz, cb;
  std::vector<int> ball_off, ball_size, ball_vert, row_nbr, nbr_pos, max_ball, max_span;
  std::vector<int> ball_span, row_pack, bond_ent;  // compact forms, see DevGraph
  std::vector<int16_t> nbr_pos16;
  std::vector<int> rec, bond_info, max_pairs;  // rows with neighbour pairs, see DevGraph
  std::vector<uint32_t> pairs;
  bool pack_ok = true;
};

gna_status validate(int32_t n_sites, int32_t n_edges, const int32_t* edges, const double* J,
                    int32_t max_layers, bool need_J) {
  if (n_sites < 1 || n_sites > 4096) return GNA_ERR_INVALID_ARG;
  if (n_edges < 0 || n_edges > (1 << 20)) return GNA_ERR_INVALID_ARG;
  if (max_layers < 0 || max_layers > kMaxL) return GNA_ERR_INVALID_ARG;
  if (n_edges > 0 && edges == nullptr) return GNA_ERR_INVALID_ARG;
  if (need_J && n_edges > 0 && J == nullptr) return GNA_ERR_INVALID_ARG;
  std::vector<uint64_t> seen(n_edges > 0 ? n_edges : 0);
  for (int e = 0; e < n_edges; ++e) {
    int a = edges[2 * e], b = edges[2 * e + 1];
    if (a < 0 || a >= n_sites || b < 0 || b >= n_sites || a == b) return GNA_ERR_INVALID_ARG;
    seen[e] = (uint64_t)(a < b ? a : b) << 32 | (uint32_t)(a < b ? b : a);
    if (need_J && !std::isfinite(J[e])) return GNA_ERR_INVALID_ARG;
  }
  std::sort(seen.begin(), seen.end());
  if (std::adjacent_find(seen.begin(), seen.end()) != seen.end()) return GNA_ERR_INVALID_ARG;
  return GNA_OK;
}

void build(int n, int E, const int32_t* edges, const double* J, int Lmax, HostGraph* h) {
  h->n = n;
  h->E = E;
  h->Lmax = Lmax;
  std::vector<int> deg(n, 0);
  for (int e = 0; e < E; ++e) {
    deg[edges[2 * e]]++;
    deg[edges[2 * e + 1]]++;
  }
  h->row_ptr.assign(n + 1, 0);
  for (int v = 0; v < n; ++v) h->row_ptr[v + 1] = h->row_ptr[v] + deg[v];
  h->col.assign(2 * E, 0);
  h->col_edge.assign(2 * E, 0);
  std::vector<int> fill(h->row_ptr.begin(), h->row_ptr.end() - 1);
  // neighbours in edge-list order
  for (int e = 0; e < E; ++e) {
    int a = edges[2 * e], b = edges[2 * e + 1];
    h->col_edge[fill[a]] = e;
    h->col[fill[a]++] = b;
    h->col_edge[fill[b]] = e;
    h->col[fill[b]++] = a;
  }
  h->wf.resize(2 * E);
  h->wd.resize(2 * E);
  for (int v = 0; v < n; ++v)
    for (int k = h->row_ptr[v]; k < h->row_ptr[v + 1]; ++k) {
      double w = 1.0 / std::sqrt((double)deg[v] * (double)deg[h->col[k]]);
      h->wd[k] = w;
      h->wf[k] = (float)w;
    }
  h->edges.assign(edges, edges + 2 * E);
  if (J)
    h->J.assign(J, J + E);
  else
    h->J.assign(E, 1.0);

  // Nested neighbourhoods: ball_0 = (i, j); ball_l = ball_{l-1} followed by the
  // neighbours of its newest rows, in order of discovery.
  h->ball_off.assign(E + 1, 0);
  h->ball_size.assign((size_t)E * (Lmax + 1), 0);
  h->ball_span.assign((size_t)E * (Lmax + 1), 0);
  h->bond_ent.assign(E, 0);
  h->max_ball.assign(Lmax + 1, 0);
  h->max_span.assign(Lmax + 1, 0);
  h->bond_info.assign((size_t)E * 32, 0);
  h->max_pairs.assign(Lmax + 1, 0);
  h->ball_vert.clear();
  h->row_nbr.clear();
  h->nbr_pos.clear();
  std::vector<int> pos(n, -1), order;
  for (int e = 0; e < E; ++e) {
    order.clear();
    order.push_back(edges[2 * e]);
    order.push_back(edges[2 * e + 1]);
    pos[order[0]] = 0;
    pos[order[1]] = 1;
    int* sz = &h->ball_size[(size_t)e * (Lmax + 1)];
    sz[0] = 2;
    int lo = 0;
    for (int l = 1; l <= Lmax; ++l) {
      int hi = (int)order.size();
      for (int r = lo; r < hi; ++r) {
        int v = order[r];
        for (int k = h->row_ptr[v]; k < h->row_ptr[v + 1]; ++k) {
          int u = h->col[k];
          if (pos[u] < 0) {
            pos[u] = (int)order.size();
            order.push_back(u);
          }
        }
      }
      lo = hi;
      sz[l] = (int)order.size();
    }
    // the rows' tables: sizes first, then one pass that fills them
    const int rows = (int)order.size();
    int ents = 0, npairs = 0;
    for (int v : order) {
      const int d = h->row_ptr[v + 1] - h->row_ptr[v];
      ents += d;
      npairs += (d + 1) / 2;
    }
    if (e == 0) {  // room for bonds like the first one, within reason: it may be a hub's, the others not
      const size_t bonds = std::min((size_t)E, (size_t)(1 << 20) / (ents + rows) + 1), R = bonds * rows, N2 = bonds * ents;
      for (std::vector<int>* v : {&h->ball_vert, &h->row_nbr, &h->row_pack}) v->reserve(R);
      h->nbr_pos.reserve(N2);
      h->nbr_pos16.reserve(N2);
      h->rec.reserve(bonds * ((rows + 1) / 2 * 4));
      h->pairs.reserve(bonds * ((npairs + 3) / 4 * 4));
    }
    const size_t r0 = h->ball_vert.size(), e0 = h->nbr_pos.size();
    h->ball_off[e] = (int)r0;
    h->bond_ent[e] = (int)e0;
    h->ball_vert.insert(h->ball_vert.end(), order.begin(), order.end());
    h->row_nbr.resize(r0 + rows);
    h->row_pack.resize(r0 + rows);
    h->nbr_pos.resize(e0 + ents);
    h->nbr_pos16.resize(e0 + ents);
    const size_t q0 = h->rec.size(), p0 = h->pairs.size();  // 16-byte parts, zero rows as padding
    h->rec.resize(q0 + (size_t)(rows + 1) / 2 * 4, 0);
    h->pairs.resize(p0 + (size_t)(npairs + 3) / 4 * 4, 0xFFFFFFFFu);
    int* info = &h->bond_info[(size_t)e * 32];
    info[0] = (int)(q0 / 2);
    info[1] = (int)p0;
    std::memcpy(info + 2, &h->J[e], sizeof(double));
    info[4] = edges[2 * e];
    info[5] = edges[2 * e + 1];
    int* rec = h->rec.data() + q0;
    uint32_t* pr = h->pairs.data() + p0;
    int at = 0, pat = 0, l = 0;
    for (int r = 0; r < rows; ++r) {
      const int v = order[r], k0 = h->row_ptr[v], d = h->row_ptr[v + 1] - k0;
      if (at > 0xFFFF) h->pack_ok = false;
      h->row_nbr[r0 + r] = (int)e0 + at;
      h->row_pack[r0 + r] = v | ((at & 0xFFFF) << 16);
      rec[2 * r] = v | ((d + 1) / 2) << 16;
      rec[2 * r + 1] = pat;
      for (int k = 0; k < d; ++k) {
        const int p = pos[h->col[k0 + k]];
        h->nbr_pos[e0 + at + k] = p >= 0 ? p : INT_MAX;
        h->nbr_pos16[e0 + at + k] = (int16_t)(p >= 0 ? p : 32767);
        // a position as the warp-tiled kernels stage it: 4 p + (p & 1), 0xFFFF when outside
        const uint32_t s = p < 0 ? 0xFFFFu : (uint32_t)(4 * p + (p & 1));
        if (k % 2 == 0)
          pr[pat + k / 2] = s | 0xFFFF0000u;
        else
          pr[pat + k / 2] = (pr[pat + k / 2] & 0xFFFFu) | s << 16;
      }
      at += d;
      pat += (d + 1) / 2;
      for (; l <= Lmax && sz[l] == r + 1; ++l) {
        h->max_ball[l] = std::max(h->max_ball[l], sz[l]);
        h->max_span[l] = std::max(h->max_span[l], at);
        h->ball_span[(size_t)e * (Lmax + 1) + l] = at;
        h->max_pairs[l] = std::max(h->max_pairs[l], pat);
        info[8 + l] = sz[l];
        if (l > 0) info[16 + l] = pat;
      }
    }
    for (int v : order) pos[v] = -1;
  }
  h->ball_off[E] = (int)h->ball_vert.size();
}

// The handle's arrays in one device allocation, filled by one copy: add() every array, then
// upload().  (One allocation and copy per array was two thirds of a small graph's creation.)
struct Packer {
  std::vector<unsigned char> bytes;
  std::vector<std::pair<const void**, size_t>> at;  // where each array's device pointer goes, its offset
  template <typename T>
  void add(const std::vector<T>& v, const T** dst) {
    *dst = nullptr;
    if (v.empty()) return;
    const size_t o = (bytes.size() + 255) / 256 * 256;
    bytes.resize(o + v.size() * sizeof(T));
    std::memcpy(bytes.data() + o, v.data(), v.size() * sizeof(T));
    at.emplace_back((const void**)dst, o);
  }
  gna_status upload(gna_graph* g) {
    if (bytes.empty()) return GNA_OK;
    void* p = nullptr;
    GNA_CUDA_TRY(cudaMalloc(&p, bytes.size()));
    g->allocations.push_back(p);
    GNA_CUDA_TRY(cudaMemcpy(p, bytes.data(), bytes.size(), cudaMemcpyHostToDevice));
    for (auto& a : at) *a.first = (const unsigned char*)p + a.second;
    return GNA_OK;
  }
};

}  // namespace

}  // namespace gna

namespace gna {
namespace {

// Shared by both creation entries: Jxy is the off-diagonal coupling (J of Heisenberg
// bonds), Jz / hz / cb the diagonal terms (NULL hz, cb = zero).
gna_status create_graph(int32_t n_sites, int32_t n_edges, const int32_t* edges, const double* Jz,
                        const double* Jxy, const double* hz, const double* cb, int32_t max_layers,
                        gna_graph** out) {
  if (!out) return GNA_ERR_INVALID_ARG;
  *out = nullptr;
  gna_status st = validate(n_sites, n_edges, edges, Jxy, max_layers, true);
  if (st != GNA_OK) return st;
  for (const double* a : {Jz, hz, cb}) {
    if (a == nullptr) continue;
    for (int e = 0; e < n_edges; ++e)
      if (!std::isfinite(a[e])) return GNA_ERR_INVALID_ARG;
  }
  if (n_edges > 0 && Jz == nullptr) return GNA_ERR_INVALID_ARG;
  HostGraph h;
  build(n_sites, n_edges, edges, Jxy, max_layers, &h);
  h.Jz.assign(n_edges, 0.0);
  h.hz.assign(n_edges, 0.0);
  h.cb.assign(n_edges, 0.0);
  for (int e = 0; e < n_edges; ++e) {
    h.Jz[e] = Jz[e];
    if (hz) h.hz[e] = hz[e];
    if (cb) h.cb[e] = cb[e];
  }
  std::unique_ptr<gna_graph, gna_status (*)(gna_graph*)> own(new gna_graph(), gna_graph_destroy);
  gna_graph* const g = own.get();
  cudaGetDevice(&g->device);
  g->d.n = h.n;
  g->d.E = h.E;
  g->d.Lmax = h.Lmax;
  Packer pk;
  pk.add(h.row_ptr, &g->d.row_ptr);
  pk.add(h.col, &g->d.col);
  pk.add(h.col_edge, &g->d.col_edge);
  pk.add(h.wf, &g->d.wf);
  pk.add(h.wd, &g->d.wd);
  pk.add(h.edges, &g->d.edges);
  pk.add(h.J, &g->d.J);
  pk.add(h.Jz, &g->d.Jz);
  pk.add(h.hz, &g->d.hz);
  pk.add(h.cb, &g->d.cb);
  pk.add(h.ball_off, &g->d.ball_off);
  pk.add(h.ball_size, &g->d.ball_size);
  pk.add(h.ball_vert, &g->d.ball_vert);
  pk.add(h.row_nbr, &g->d.row_nbr);
  pk.add(h.nbr_pos, &g->d.nbr_pos);
  pk.add(h.ball_span, &g->d.ball_span);
  pk.add(h.row_pack, &g->d.row_pack);
  pk.add(h.nbr_pos16, &g->d.nbr_pos16);
  pk.add(h.bond_ent, &g->d.bond_ent);
  pk.add(h.rec, &g->d.rec);
  pk.add(h.pairs, &g->d.pairs);
  pk.add(h.bond_info, &g->d.bond_info);
  st = pk.upload(g);
  if (st != GNA_OK) return st;
  g->pack_ok = h.pack_ok;
  g->h_row_ptr = h.row_ptr;
  g->h_col = h.col;
  g->h_edges = h.edges;
  g->h_ball_size = h.ball_size;
  g->h_ball_off = h.ball_off;
  g->h_J = h.J;
  g->max_ball = h.max_ball;
  g->max_span = h.max_span;
  g->max_pairs = h.max_pairs;
  g->min_deg = h.row_ptr[1] - h.row_ptr[0];
  for (int v = 0; v < h.n; ++v) {
    g->max_deg = std::max(g->max_deg, h.row_ptr[v + 1] - h.row_ptr[v]);
    g->min_deg = std::min(g->min_deg, h.row_ptr[v + 1] - h.row_ptr[v]);
  }
  *out = own.release();
  return GNA_OK;
}

// No exception leaves the C entries: the tables that the host has no memory for are refused.
template <typename Fn>
gna_status guarded(Fn fn) {
  try {
    return fn();
  } catch (const std::exception&) {
    return GNA_ERR_UNSUPPORTED;
  }
}

}  // namespace
}  // namespace gna

extern "C" gna_status gna_graph_create(int32_t n_sites, int32_t n_edges, const int32_t* edges,
                                       const double* J, int32_t max_layers, gna_graph** out) {
  return gna::guarded([&] { return gna::create_graph(n_sites, n_edges, edges, J, J, nullptr, nullptr, max_layers, out); });
}

extern "C" gna_status gna_graph_create_xxz(int32_t n_sites, int32_t n_edges, const int32_t* edges,
                                           const double* Jz, const double* Jxy, const double* hz,
                                           const double* c, int32_t max_layers, gna_graph** out) {
  if (n_edges > 0 && (Jz == nullptr || Jxy == nullptr || hz == nullptr || c == nullptr))
    return GNA_ERR_INVALID_ARG;
  return gna::guarded([&] { return gna::create_graph(n_sites, n_edges, edges, Jz, Jxy, hz, c, max_layers, out); });
}

extern "C" gna_status gna_graph_destroy(gna_graph* g) {
  if (!g) return GNA_ERR_INVALID_ARG;
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != g->device) cudaSetDevice(g->device);
  for (void* p : g->allocations) cudaFree(p);
  if (cur != g->device) cudaSetDevice(cur);
  delete g;
  return GNA_OK;
}

extern "C" gna_status gna_graph_info(const gna_graph* g, int32_t* n_sites, int32_t* n_edges,
                                     int32_t* max_layers) {
  if (!g) return GNA_ERR_INVALID_ARG;
  if (n_sites) *n_sites = g->d.n;
  if (n_edges) *n_edges = g->d.E;
  if (max_layers) *max_layers = g->d.Lmax;
  return GNA_OK;
}

extern "C" gna_status gna_ball_sizes_host(int32_t n_sites, int32_t n_edges, const int32_t* edges,
                                          int32_t n_layers, int32_t* out) {
  using namespace gna;
  if (!out && n_edges > 0) return GNA_ERR_INVALID_ARG;
  return guarded([&] {
    gna_status st = validate(n_sites, n_edges, edges, nullptr, n_layers, false);
    if (st != GNA_OK) return st;
    HostGraph h;
    build(n_sites, n_edges, edges, nullptr, n_layers, &h);
    std::memcpy(out, h.ball_size.data(), h.ball_size.size() * sizeof(int32_t));
    return (gna_status)GNA_OK;
  });
}
