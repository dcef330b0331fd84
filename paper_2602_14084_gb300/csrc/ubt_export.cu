// ubt_export.cu -- the built graph copied to the host for inspection.
//
// The library numbers vertices by reverse Node Order and sorts rows for the
// traversal (ubt_internal.cuh).  ubt_graph_export_traversal copies those arrays;
// the other exports show the graph by the caller's ids: forward lists in id order of their owners, FIXED lists by |q|
// descending (then id) and REAL ones by id, the pairs grouped by the owner
// the "pull" tuning names, and the owners split into task classes by their
// lists and streamed work.  The host rearranges copies of the device arrays.
#include <algorithm>
#include <exception>
#include <numeric>
#include <vector>

#include "ubt_internal.cuh"

namespace ubt {
namespace {

struct HostGraph {
  std::vector<uint32_t> row_ptr;  // n + 1, by id
  std::vector<uint64_t> adj;      // m, neighbours by id
  std::vector<uint32_t> eid;      // m
};

ubt_status host_graph(const ubt_graph* g, cudaStream_t s, HostGraph* h) {
  const size_t n = (size_t)g->n, m = (size_t)g->m;
  std::vector<uint32_t> vid(n), rp(n + 1), eid(m);
  std::vector<uint64_t> adj(m);
  if (n) UBT_CUDA(cudaMemcpyAsync(vid.data(), g->vid, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost, s));
  UBT_CUDA(cudaMemcpyAsync(rp.data(), g->row_ptr, sizeof(uint32_t) * (n + 1), cudaMemcpyDeviceToHost, s));
  if (m) {
    UBT_CUDA(cudaMemcpyAsync(adj.data(), g->adj, sizeof(uint64_t) * m, cudaMemcpyDeviceToHost, s));
    UBT_CUDA(cudaMemcpyAsync(eid.data(), g->eid, sizeof(uint32_t) * m, cudaMemcpyDeviceToHost, s));
  }
  UBT_CUDA(cudaStreamSynchronize(s));
  h->row_ptr.assign(n + 1, 0);
  for (size_t r = 0; r < n; r++) h->row_ptr[vid[r] + 1] = rp[r + 1] - rp[r];
  for (size_t v = 0; v < n; v++) h->row_ptr[v + 1] += h->row_ptr[v];
  h->adj.resize(m);
  h->eid.resize(m);
  const bool fixed = g->kind == UBT_GRAPH_FIXED;
  std::vector<std::pair<uint64_t, uint32_t>> row;  // sort key, position
  for (size_t r = 0; r < n; r++) {
    row.clear();
    for (uint32_t p = rp[r]; p < rp[r + 1]; p++) {
      const uint32_t w = vid[adj_col(adj[p])];
      const int64_t q = adj_q(adj[p]);
      row.emplace_back(fixed ? ((uint64_t)(32768 - (q < 0 ? -q : q)) << 32) | w : w, p);
    }
    std::sort(row.begin(), row.end());
    uint32_t at = h->row_ptr[vid[r]];
    for (const auto& x : row) {
      h->adj[at] = adj_pack((uint32_t)x.first, adj_valbits(adj[x.second]));
      h->eid[at++] = eid[x.second];
    }
  }
  return UBT_OK;
}

struct HostPairs {
  std::vector<uint32_t> ptr;    // n + 1
  std::vector<uint64_t> pairs;  // streamed vertex | CSR position << 32
};

HostPairs host_pairs(const ubt_graph* g, const HostGraph& h) {
  const size_t n = (size_t)g->n;
  auto len = [&](size_t v) { return h.row_ptr[v + 1] - h.row_ptr[v]; };
  auto owner = [&](size_t u, size_t v) { return g->pull && len(v) > len(u) ? v : u; };
  HostPairs p;
  p.ptr.assign(n + 1, 0);
  for (size_t u = 0; u < n; u++)
    for (uint32_t i = h.row_ptr[u]; i < h.row_ptr[u + 1]; i++) p.ptr[owner(u, adj_col(h.adj[i])) + 1]++;
  for (size_t v = 0; v < n; v++) p.ptr[v + 1] += p.ptr[v];
  std::vector<uint32_t> next(p.ptr.begin(), p.ptr.end() - 1);
  p.pairs.resize(h.adj.size());
  for (size_t u = 0; u < n; u++)
    for (uint32_t i = h.row_ptr[u]; i < h.row_ptr[u + 1]; i++) {
      const uint32_t v = adj_col(h.adj[i]);
      const size_t x = owner(u, v);
      p.pairs[next[x]++] = ((uint64_t)i << 32) | (x == u ? v : (uint32_t)u);
    }
  return p;
}

// owners with at least 2 list entries and a pair: giant, hub and medium ones
void host_lists(const ubt_graph* g, const HostGraph& h, const HostPairs& p, std::vector<uint32_t> (&cls)[3]) {
  std::vector<std::pair<int, uint32_t>> by_work[3];  // - log2 of the streamed work, owner
  for (size_t x = 0; x < (size_t)g->n; x++) {
    const int64_t len = h.row_ptr[x + 1] - h.row_ptr[x];
    if (len < 2 || p.ptr[x + 1] == p.ptr[x]) continue;
    int64_t work = 0;
    for (uint32_t i = p.ptr[x]; i < p.ptr[x + 1]; i++) {
      const uint32_t s = (uint32_t)p.pairs[i];
      work += h.row_ptr[s + 1] - h.row_ptr[s];
    }
    const int c = len > g->giant_threshold ? 0 : (len > g->hub_threshold || work > g->block_work) ? 1 : 2;
    int lg = 0;
    while ((work >> lg) > 1) lg++;
    by_work[c].emplace_back(-lg, (uint32_t)x);
  }
  for (int c = 0; c < 3; c++) {
    std::stable_sort(by_work[c].begin(), by_work[c].end());
    for (const auto& x : by_work[c]) cls[c].push_back(x.second);
  }
}

ubt_status export_graph(const ubt_graph* g, uint32_t* h_row_ptr, uint64_t* h_adj, uint32_t* h_eid, uint32_t* h_lists,
                        int64_t* h_list_sizes, uint32_t* h_pair_ptr, uint64_t* h_pairs, cudaStream_t s) {
  HostGraph h;
  const ubt_status st = host_graph(g, s, &h);
  if (st != UBT_OK) return st;
  if (h_row_ptr) std::copy(h.row_ptr.begin(), h.row_ptr.end(), h_row_ptr);
  if (h_adj) std::copy(h.adj.begin(), h.adj.end(), h_adj);
  if (h_eid) std::copy(h.eid.begin(), h.eid.end(), h_eid);
  if (!h_lists && !h_list_sizes && !h_pair_ptr && !h_pairs) return UBT_OK;
  const HostPairs p = host_pairs(g, h);
  if (h_pair_ptr) std::copy(p.ptr.begin(), p.ptr.end(), h_pair_ptr);
  if (h_pairs) std::copy(p.pairs.begin(), p.pairs.end(), h_pairs);
  if (h_lists || h_list_sizes) {
    std::vector<uint32_t> cls[3];
    host_lists(g, h, p, cls);
    for (int c = 0; c < 3; c++) {
      if (h_list_sizes) h_list_sizes[c] = (int64_t)cls[c].size();
      if (h_lists) h_lists = std::copy(cls[c].begin(), cls[c].end(), h_lists);
    }
    if (h_list_sizes) h_list_sizes[3] = 0;
  }
  return UBT_OK;
}

}  // namespace
}  // namespace ubt

using namespace ubt;

// nothing throws across the boundary: host memory that runs out is an invalid size here
extern "C" ubt_status ubt_graph_export(const ubt_graph* g, uint32_t* h_row_ptr, uint64_t* h_adj, uint32_t* h_eid,
                                       uint32_t* h_lists, int64_t* h_list_sizes, void* stream) {
  if (!g) return UBT_ERR_INVALID_ARG;
  try {
    return export_graph(g, h_row_ptr, h_adj, h_eid, h_lists, h_list_sizes, nullptr, nullptr, (cudaStream_t)stream);
  } catch (const std::exception&) {
    return UBT_ERR_INVALID_ARG;
  }
}

extern "C" ubt_status ubt_graph_export_pairs(const ubt_graph* g, uint32_t* h_pair_ptr, uint64_t* h_pairs,
                                             void* stream) {
  if (!g) return UBT_ERR_INVALID_ARG;
  try {
    return export_graph(g, nullptr, nullptr, nullptr, nullptr, nullptr, h_pair_ptr, h_pairs, (cudaStream_t)stream);
  } catch (const std::exception&) {
    return UBT_ERR_INVALID_ARG;
  }
}

extern "C" ubt_status ubt_graph_export_traversal(const ubt_graph* g, uint32_t* h_vid, uint32_t* h_row_ptr,
                                                 uint64_t* h_adj, uint32_t* h_eid, uint32_t* h_rowid,
                                                 uint32_t* h_pair_ptr, uint64_t* h_pairs, uint64_t* h_tasks,
                                                 int64_t* h_sizes, void* stream) {
  if (!g) return UBT_ERR_INVALID_ARG;
  if (h_rowid && !g->rowid) return UBT_ERR_UNSUPPORTED;
  cudaStream_t s = (cudaStream_t)stream;
  auto copy = [&](void* to, const void* from, size_t bytes) {
    return to && bytes ? cudaMemcpyAsync(to, from, bytes, cudaMemcpyDeviceToHost, s) : cudaSuccess;
  };
  const size_t n = (size_t)g->n, m = (size_t)g->m;
  UBT_CUDA(copy(h_vid, g->vid, 4 * n));
  UBT_CUDA(copy(h_row_ptr, g->row_ptr, 4 * (n + 1)));
  UBT_CUDA(copy(h_adj, g->adj, 8 * m));
  UBT_CUDA(copy(h_eid, g->eid, 4 * m));
  UBT_CUDA(copy(h_rowid, g->rowid, 4 * m));
  UBT_CUDA(copy(h_pair_ptr, g->pair_ptr, 4 * (n + 1)));
  UBT_CUDA(copy(h_pairs, g->pairs, 8 * m));
  for (int c = 0; c < kTaskClasses; c++) {
    UBT_CUDA(copy(h_tasks, g->lists[c], 8 * (size_t)g->n_tasks[c]));
    if (h_tasks) h_tasks += g->n_tasks[c];
    if (h_sizes) h_sizes[c] = g->n_tasks[c];
  }
  if (h_sizes) h_sizes[kTaskClasses] = g->merge_first;
  UBT_CUDA(cudaStreamSynchronize(s));
  return UBT_OK;
}
