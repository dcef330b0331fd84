// ubt_build.cu -- building the graph the exact algorithms traverse.
//
//   validate   ids < n, no self-loops, probabilities in range       (Def. 1)
//   degree     undirected degree of every vertex
//   number     every vertex by its position in reverse Node Order (degree, then
//              id, Sec. 4; the graphs of a batch apart): a radix sort by degree
//   CSR        forward lists N>(u) as offsets + packed (neighbour, value)
//   sort       every list ascending by neighbour (duplicates are equal neighbours)
//   pairs      every forward edge u -> v is a pair owned by v, whose list
//              becomes the table while the part of u's list after v is
//              streamed through it; pairs grouped by owner
//   work lists owners (>= 1 list entry, >= 1 pair) split by list length and
//              streamed work into block tasks and warp tasks, each ordered by
//              decreasing work
//
// Why the later vertex owns: Alg. 1 streams N>(v) through a table of N>(u) for
// u -> v.  The triangles of the pair lie in N>(u) n N>(v); streaming the part of
// N>(u) after v through a table of N>(v) finds the same ones and probes 0.62x
// the entries that streaming the shorter whole list does (R-MAT scale 20: 1.97e9
// -> 1.22e9, Chung-Lu of 1e6 vertices: 3.16e8 -> 1.95e8), and choosing the better
// direction per pair would remove only another 0.5 %.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "ubt_internal.cuh"

namespace ubt {

namespace {

constexpr int kSortHugeBlocks = 16;  // blocks sorting lists longer than that

// error word: lowest (edge index << 8 | code) wins, so the report is deterministic
__device__ inline void report(unsigned long long* err, uint64_t index, int code) {
  atomicMin(err, (unsigned long long)((index << 8) | (uint64_t)code));
}

__global__ void k_vertex_graph(const int64_t* __restrict__ voff, int64_t ng, int64_t n, uint32_t* vgraph) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = ng;  // find g with voff[g] <= v < voff[g+1]
    while (hi - lo > 1) {
      int64_t mid = (lo + hi) / 2;
      if (voff[mid] <= v) lo = mid; else hi = mid;
    }
    vgraph[v] = (uint32_t)lo;
  }
}

// Adds 1 to ctr[key] for every lane with `on`, with one atomic per run of
// equal keys in consecutive lanes (edge lists sorted by source put a
// vertex's edges together, and one counter then takes every lane's add);
// returns the lane's slot: the counter's old value plus its rank in the run.
// All 32 lanes call it.
__device__ __forceinline__ uint32_t add_by_runs(uint32_t* ctr, uint32_t key, bool on) {
  const uint32_t lane = lane_id();
  const unsigned act = __ballot_sync(kFull, on);
  const uint32_t prev = __shfl_up_sync(kFull, key, 1);
  const bool head = on && !(lane > 0 && ((act >> (lane - 1)) & 1u) && prev == key);
  const unsigned heads = __ballot_sync(kFull, head);
  const unsigned upto = (2u << lane) - 1u;          // lanes 0..lane (all bits for lane 31)
  const unsigned after = (heads | ~act) & ~upto;     // where runs end, after this lane
  const uint32_t next = after ? (uint32_t)__ffs(after) - 1u : 32u;
  uint32_t old = 0;
  if (head) old = atomicAdd(&ctr[key], next - lane);
  const unsigned mine = heads & upto;
  const uint32_t my_head = mine ? 31u - (uint32_t)__clz(mine) : lane;
  return __shfl_sync(kFull, old, my_head) + (lane - my_head);
}

// Grid-stride loops over the edges in which every warp takes 32 consecutive
// edges per step, so that warp-wide runs (add_by_runs) see neighbours.
#define UBT_FOR_EDGE_WARPS(base, m)                                                                     \
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < (m);               \
       base += (int64_t)gridDim.x * blockDim.x)

__global__ void k_validate_degree(int64_t n, int64_t m, const uint32_t* __restrict__ src,
                                  const uint32_t* __restrict__ dst, const uint32_t* __restrict__ k,
                                  const float* __restrict__ p, const uint32_t* __restrict__ vgraph,
                                  uint32_t* __restrict__ deg, unsigned long long* err) {
  const uint32_t lane = lane_id();
  UBT_FOR_EDGE_WARPS(base, m) {
    const int64_t i = base + lane;
    bool ok = i < m;
    const uint32_t a = ok ? src[i] : 0u, b = ok ? dst[i] : 0u;
    if (ok && ((int64_t)a >= n || (int64_t)b >= n)) { report(err, i, -UBT_ERR_VERTEX_OOB); ok = false; }
    if (ok && a == b) { report(err, i, -UBT_ERR_SELF_LOOP); ok = false; }
    if (ok) {
      if (k) {
        if (k[i] > 65536u) report(err, i, -UBT_ERR_PROB_OOB);
      } else {
        const float x = p[i];
        if (!(x >= 0.0f && x <= 1.0f)) report(err, i, -UBT_ERR_PROB_OOB);
      }
      if (vgraph && vgraph[a] != vgraph[b]) { report(err, i, -UBT_ERR_INVALID_ARG); ok = false; }
    }
    add_by_runs(deg, a, ok);
    if (ok) atomicAdd(&deg[b], 1u);
  }
}

// out: [0] the largest degree, [1] the vertices of degree > kMergeDegree
constexpr uint32_t kMergeDegree = 32;
__global__ void k_degree_stats(int64_t n, const uint32_t* __restrict__ deg, unsigned long long* out) {
  uint32_t best = 0, large = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    best = max(best, deg[v]);
    large += deg[v] > kMergeDegree ? 1u : 0u;
  }
  best = __reduce_max_sync(kFull, best);
  large = __reduce_add_sync(kFull, large);
  if (lane_id() == 0) {
    atomicMax(&out[0], (unsigned long long)best);
    if (large) atomicAdd(&out[1], (unsigned long long)large);
  }
}

// ---------------------------------------------------------------- vertex numbers
//
// Reverse Node Order is a stable sort of the ids n - 1 .. 0 by degree
// descending (and, for a batch, by graph first: the least significant key is
// sorted first, 8 bits a pass).  A pass counts the digits of every tile, scans
// the counts digit by digit, and writes every id to its place; a warp takes
// 512 consecutive items, so ranks within a warp and the warps' order keep the
// sort stable.  Bound by the launches (four a pass) up to a few million vertices.
constexpr int kRankThreads = 256;
constexpr int kRankItems = 16;
constexpr int64_t kRankTile = kRankThreads * kRankItems;

struct RankKey {
  const uint32_t* key;  // by id
  int shift;
  uint32_t flip;        // 255: descending
};
__device__ __forceinline__ uint32_t rank_digit(const RankKey& k, uint32_t id) {
  return ((k.key[id] >> k.shift) & 255u) ^ k.flip;
}
__device__ __forceinline__ uint32_t rank_item(const uint32_t* in, int64_t i, int64_t n) {
  return in ? in[i] : (uint32_t)(n - 1 - i);
}

// hist[digit * tiles + tile]
__global__ void __launch_bounds__(kRankThreads)
k_rank_count(int64_t n, const uint32_t* __restrict__ in, RankKey k, uint32_t* __restrict__ hist) {
  __shared__ uint32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  for (int j = 0; j < kRankItems; j++) {
    const int64_t i = blockIdx.x * kRankTile + j * kRankThreads + threadIdx.x;
    if (i < n) atomicAdd(&cnt[rank_digit(k, rank_item(in, i, n))], 1u);
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
}

// off: the scanned counts.  out[place] = id and, in the last pass, rank[id] = place.
__global__ void __launch_bounds__(kRankThreads)
k_rank_scatter(int64_t n, const uint32_t* __restrict__ in, RankKey k, const uint32_t* __restrict__ off,
               uint32_t* __restrict__ out, uint32_t* __restrict__ rank) {
  constexpr int kWarps = kRankThreads / 32;
  __shared__ uint32_t cnt[kWarps][256];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kWarps * 256; i += kRankThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  uint32_t id[kRankItems], at[kRankItems];  // at: digit << 16 | rank among the warp's items of that digit
#pragma unroll
  for (int j = 0; j < kRankItems; j++) {
    const int64_t i = blockIdx.x * kRankTile + wid * (32 * kRankItems) + j * 32 + lane;
    const bool on = i < n;
    id[j] = on ? rank_item(in, i, n) : 0u;
    const uint32_t d = on ? rank_digit(k, id[j]) : 256u;
    const unsigned peers = __match_any_sync(kFull, d);
    const uint32_t before = on ? cnt[wid][d] : 0u;
    at[j] = (d << 16) | (before + __popc(peers & lanemask_lt()));
    __syncwarp();
    if (on && lane == __ffs(peers) - 1) cnt[wid][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  uint32_t run = off[(size_t)threadIdx.x * gridDim.x + blockIdx.x];
  for (int w = 0; w < kWarps; w++) {
    const uint32_t c = cnt[w][threadIdx.x];
    cnt[w][threadIdx.x] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRankItems; j++) {
    const uint32_t d = at[j] >> 16;
    if (d > 255u) continue;
    const uint32_t place = cnt[wid][d] + (at[j] & 0xFFFFu);
    out[place] = id[j];
    if (rank) rank[id[j]] = place;
  }
}

// by the vertex numbers: the graph of every vertex, and the first number of every graph
__global__ void k_rank_graphs(int64_t n, const uint32_t* __restrict__ vid, const uint32_t* __restrict__ by_id,
                              uint32_t* __restrict__ by_rank, const int64_t* __restrict__ voff, int64_t ng,
                              uint32_t* __restrict__ gstart) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ng; g += (int64_t)gridDim.x * blockDim.x)
    gstart[g] = (uint32_t)voff[g];
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    by_rank[r] = by_id[vid[r]];
}

// an edge belongs to the row of its earlier endpoint in Node Order: the larger number
__global__ void k_out_degree(int64_t m, const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                             const uint32_t* __restrict__ rank, uint32_t* __restrict__ outdeg) {
  const uint32_t lane = lane_id();
  UBT_FOR_EDGE_WARPS(base, m) {
    const int64_t i = base + lane;
    const bool on = i < m;
    add_by_runs(outdeg, on ? max(rank[src[i]], rank[dst[i]]) : 0u, on);
  }
}

__global__ void k_scatter(int64_t m, const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                          const uint32_t* __restrict__ k, const float* __restrict__ p,
                          const uint32_t* __restrict__ rank, uint32_t* __restrict__ next,
                          uint64_t* __restrict__ adj, uint32_t* __restrict__ eid,
                          const uint32_t* __restrict__ key_in, uint32_t* __restrict__ key_out) {
  const uint32_t lane = lane_id();
  UBT_FOR_EDGE_WARPS(base, m) {
    const int64_t i = base + lane;
    const bool on = i < m;
    const uint32_t a = on ? rank[src[i]] : 0u, b = on ? rank[dst[i]] : 0u;
    const uint32_t row = max(a, b), hi = min(a, b);
    const uint32_t pos = add_by_runs(next, row, on);  // next[row] starts at the row's offset
    if (!on) continue;
    uint32_t val;
    if (k) {
      val = (uint32_t)(int32_t)(32768 - (int32_t)k[i]);     // q = 32768 - k
    } else {
      val = real_valbits(p[i]);
    }
    adj[pos] = adj_pack(hi, val);
    eid[pos] = (uint32_t)i;
    if (key_out) key_out[pos] = key_in[i];
  }
}

// sort keys: by neighbour (forward rows); by (32768 - |q|, id) (undirected rows)
__device__ inline uint64_t key_by_col(uint64_t e) { return (uint64_t)adj_col(e); }
__device__ inline uint64_t key_by_absq(uint64_t e) {
  const int32_t q = adj_q(e);
  const uint32_t aq = (uint32_t)(q < 0 ? -q : q);
  return ((uint64_t)(32768u - aq) << 32) | adj_col(e);
}

// How a row is sorted: forward rows by neighbour (a duplicate edge shows as two
// equal neighbouring keys); undirected rows by (|q| descending, id), unchecked
// (the forward rows of the same edges were checked first).
enum : int { kSortById = 0, kSortByAbsq = 2 };

// Lists of <= 32 entries: one warp per list, bitonic network over the lanes.
// Bitonic sort of the words held by each aligned group of W lanes (W = 8, 16 or
// 32), ascending within every group.
template <int W>
__device__ __forceinline__ void group_bitonic(uint64_t& key, int lane) {
  const int li = lane & (W - 1);
#pragma unroll
  for (int kk = 2; kk <= W; kk <<= 1) {
#pragma unroll
    for (int j = kk >> 1; j > 0; j >>= 1) {
      const uint64_t ok = __shfl_xor_sync(kFull, key, j);
      const bool up = (li & kk) == 0;
      const bool lower = (li & j) == 0;
      key = (lower == up) == (ok < key) ? ok : key;
    }
  }
}

// Sorts the rows of one group of W lanes (row rs..rs+len, len <= W; groups
// without a row pass row = false everywhere), as `mode` says.  The network
// moves one word per comparator, the sort key << 5 | the entry's lane (the
// words are distinct), and the entries follow once at the end.
template <int W>
__device__ __forceinline__ void sort_group_row(uint64_t* adj, uint32_t* eid, uint32_t* ekey, uint32_t rs, uint32_t len,
                                               bool row, int mode, unsigned long long* err, int lane) {
  const int li = lane & (W - 1);
  const bool in = row && (uint32_t)li < len;
  const uint64_t e = in ? adj[rs + li] : 0ull;
  const uint32_t id = in ? eid[rs + li] : 0u;
  const uint32_t ky = (in && ekey) ? ekey[rs + li] : 0u;
  uint64_t key = in ? ((mode == kSortById ? key_by_col(e) : key_by_absq(e)) << 5) | (uint64_t)lane
                    : (~0ull << 5) | (uint64_t)lane;
  group_bitonic<W>(key, lane);
  if (mode == kSortById) {
    const uint64_t prev = __shfl_up_sync(kFull, key >> 5, 1);
    if (in && li > 0 && prev == key >> 5) report(err, rs + li, -UBT_ERR_DUPLICATE_EDGE);
  }
  const int from = (int)(key & 31u);
  const uint64_t se = __shfl_sync(kFull, e, from);
  const uint32_t sid = __shfl_sync(kFull, id, from);
  const uint32_t sky = ekey ? __shfl_sync(kFull, ky, from) : 0u;
  if (in) {
    adj[rs + li] = se;
    eid[rs + li] = sid;
    if (ekey) ekey[rs + li] = sky;
  }
}

// Rows of 2..32 entries: a warp takes 4 consecutive rows; the rows of at most
// 8 entries are sorted together, one per 8-lane group, then those of at most
// 16 two at a time and the others one after another by the whole warp.
__global__ void k_sort_short_rows(int64_t n, const uint32_t* __restrict__ row_ptr, uint64_t* adj, uint32_t* eid,
                                  uint32_t* ekey, int mode, unsigned long long* err) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t u0 = 4 * (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)); u0 < n; u0 += 4 * warps) {
    const int64_t u = u0 + (lane >> 3);
    uint32_t rs = 0, len = 0;
    if (u < n) {
      rs = row_ptr[u];
      len = row_ptr[u + 1] - rs;
    }
    if (__any_sync(kFull, len >= 2 && len <= 8))
      sort_group_row<8>(adj, eid, ekey, rs, len, len >= 2 && len <= 8, mode, err, lane);
    unsigned mid = __ballot_sync(kFull, (lane & 7) == 0 && len > 8 && len <= 16);
    while (mid) {
      const int g0 = __ffs(mid) - 1;
      mid &= mid - 1;
      const int g1 = mid ? __ffs(mid) - 1 : g0;
      const bool two = mid != 0;
      mid &= mid - 1;
      const int g = lane < 16 ? g0 : g1;
      const uint32_t rsg = __shfl_sync(kFull, rs, g), leng = __shfl_sync(kFull, len, g);
      sort_group_row<16>(adj, eid, ekey, rsg, leng, lane < 16 || two, mode, err, lane);
    }
    unsigned big = __ballot_sync(kFull, (lane & 7) == 0 && len > 16 && len <= 32);
    while (big) {
      const int g = __ffs(big) - 1;
      big &= big - 1;
      const uint32_t rsg = __shfl_sync(kFull, rs, g), leng = __shfl_sync(kFull, len, g);
      sort_group_row<32>(adj, eid, ekey, rsg, leng, true, mode, err, lane);
    }
  }
}

// Rows of 33..512 entries: one warp per row, R = 4, 8 or 16 words per lane
// (entry r * 32 + lane in register r).  A word is the sort key << 12 | the
// entry's position in the row; the words are distinct, so a bitonic network
// over registers and lanes moves one word per comparator, and the entries are
// gathered by position once at the end.
template <int R>
__device__ __forceinline__ void warp_bitonic(unsigned long long (&k)[R], int lane) {
#pragma unroll
  for (int kk = 2; kk <= 32 * R; kk <<= 1) {
#pragma unroll
    for (int j = kk >> 1; j > 0; j >>= 1) {
      if (j >= 32) {  // partner in another register of the same lane
        const int rj = j >> 5;
#pragma unroll
        for (int r = 0; r < R; r++) {
          if ((r & rj) == 0) {
            const unsigned long long a = k[r], b = k[r | rj];
            const bool asc = (((r << 5) | lane) & kk) == 0;
            k[r] = (a < b) == asc ? a : b;
            k[r | rj] = (a < b) == asc ? b : a;
          }
        }
      } else {        // partner in another lane, same register
#pragma unroll
        for (int r = 0; r < R; r++) {
          const unsigned long long o = __shfl_xor_sync(kFull, k[r], j);
          const bool up = (((r << 5) | lane) & kk) == 0;
          const bool take_min = ((lane & j) == 0) == up;
          k[r] = take_min ? (o < k[r] ? o : k[r]) : (o > k[r] ? o : k[r]);
        }
      }
    }
  }
}

template <int R>
__device__ __forceinline__ void sort_row_warp(uint64_t* adj, uint32_t* eid, uint32_t* ekey, uint32_t rs, uint32_t len,
                                              int mode, unsigned long long* err, int lane) {
  unsigned long long k[R];
  if (mode == kSortById) {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t i = (uint32_t)(r * 32 + lane);
      k[r] = i < len ? (key_by_col(adj[rs + i]) << 12) | i : ~0ull;
    }
    warp_bitonic<R>(k, lane);
#pragma unroll
    for (int r = 0; r < R; r++) {  // duplicates: equal neighbours at adjacent sorted positions
      const unsigned long long up1 = __shfl_up_sync(kFull, k[r], 1);
      const unsigned long long last = __shfl_sync(kFull, k[r > 0 ? r - 1 : 0], 31);
      const unsigned long long prev = lane > 0 ? up1 : last;
      const uint32_t i = (uint32_t)(r * 32 + lane);
      if (i < len && i > 0 && (prev >> 12) == (k[r] >> 12)) report(err, rs + i, -UBT_ERR_DUPLICATE_EDGE);
    }
  } else {
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint32_t i = (uint32_t)(r * 32 + lane);
      k[r] = i < len ? (key_by_absq(adj[rs + i]) << 12) | i : ~0ull;
    }
    warp_bitonic<R>(k, lane);
  }
  // gather by position, one array at a time: every lane reads its entries'
  // sources before any lane of the warp overwrites that array
  uint32_t pw[(R + 1) / 2];  // two 12-bit positions per register
#pragma unroll
  for (int r = 0; r < R; r += 2)
    pw[r / 2] = (uint32_t)(k[r] & 0xFFFu) | (r + 1 < R ? (uint32_t)(k[r + 1] & 0xFFFu) << 16 : 0u);
#define UBT_POS(r) ((r) & 1 ? pw[(r) / 2] >> 16 : pw[(r) / 2] & 0xFFFFu)
#pragma unroll
  for (int r = 0; r < R; r++)
    if ((uint32_t)(r * 32 + lane) < len) k[r] = adj[rs + UBT_POS(r)];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < R; r++)
    if ((uint32_t)(r * 32 + lane) < len) adj[rs + r * 32 + lane] = k[r];
  uint32_t v[R];
#pragma unroll
  for (int r = 0; r < R; r++)
    if ((uint32_t)(r * 32 + lane) < len) v[r] = eid[rs + UBT_POS(r)];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < R; r++)
    if ((uint32_t)(r * 32 + lane) < len) eid[rs + r * 32 + lane] = v[r];
  if (ekey) {
#pragma unroll
    for (int r = 0; r < R; r++)
      if ((uint32_t)(r * 32 + lane) < len) v[r] = ekey[rs + UBT_POS(r)];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; r++)
      if ((uint32_t)(r * 32 + lane) < len) ekey[rs + r * 32 + lane] = v[r];
  }
#undef UBT_POS
}

// One launch per R takes the rows of the list with 16 R < len <= 32 R (R = 4:
// every row up to 128 entries) and leaves the others to the other launches.
template <int R>
__global__ void k_sort_mid_rows(const uint32_t* __restrict__ rows, uint32_t nrows, const uint32_t* __restrict__ row_ptr,
                                uint64_t* adj, uint32_t* eid, uint32_t* ekey, int mode, unsigned long long* err) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t r0 = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); r0 < nrows; r0 += warps) {
    const uint32_t u = rows[r0];
    const uint32_t rs = row_ptr[u], len = row_ptr[u + 1] - rs;
    if (len > 32u * R || (R > 4 && len <= 16u * R)) continue;
    sort_row_warp<R>(adj, eid, ekey, rs, len, mode, err, lane);
  }
}

// the warp sorts of every row of the list (lengths 33..warp_max)
template <int R>
ubt_status launch_mid_sort(const uint32_t* rows, uint32_t nrows, const uint32_t* row_ptr, uint64_t* adj, uint32_t* eid,
                           uint32_t* ekey, int mode, unsigned long long* err, int g, int thr, cudaStream_t s) {
  k_sort_mid_rows<R><<<g, thr, 0, s>>>(rows, nrows, row_ptr, adj, eid, ekey, mode, err);
  return UBT_OK;
}

ubt_status launch_mid_sorts(const uint32_t* rows, uint32_t nrows, const uint32_t* row_ptr, uint64_t* adj,
                            uint32_t* eid, uint32_t* ekey, int mode, unsigned long long* err, uint32_t warp_max,
                            int sms, int thr, cudaStream_t s) {
  const int g = (int)std::min<unsigned long long>((nrows + 7) / 8, (unsigned long long)sms * 32);
  ubt_status st = launch_mid_sort<4>(rows, nrows, row_ptr, adj, eid, ekey, mode, err, g, thr, s);
  if (st == UBT_OK && warp_max >= 256) st = launch_mid_sort<8>(rows, nrows, row_ptr, adj, eid, ekey, mode, err, g, thr, s);
  if (st == UBT_OK && warp_max >= 512)
    st = launch_mid_sort<16>(rows, nrows, row_ptr, adj, eid, ekey, mode, err, g, thr, s);
  return st;
}

// Lists longer than the "warp_sort_max" tuning (256) and at most
// "sort_smem_max" (4096): one block per list sorts 64-bit words (sort key <<
// 12 | position in the list) in shared memory; the keys are distinct by
// construction, so the network only moves one word per comparator, and the
// entries are gathered by position once at the end.
constexpr int kPackedSortThreads = 512;
constexpr int kPackedPerThread = 8;                  // 4096 entries / 512 threads
constexpr uint32_t kPackedMax = kPackedSortThreads * kPackedPerThread;

// ascending bitonic network over pk[0..cap), cap a power of two
__device__ __forceinline__ void bitonic_packed(unsigned long long* pk, uint32_t cap) {
  for (uint32_t kk = 2; kk <= cap; kk <<= 1) {
    for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
      for (uint32_t t = threadIdx.x; t < (cap >> 1); t += blockDim.x) {
        const uint32_t i = ((t & ~(j - 1)) << 1) | (t & (j - 1));  // the comparator's lower index
        const uint32_t ixj = i | j;
        const unsigned long long a = pk[i], b = pk[ixj];
        const unsigned long long lo = a < b ? a : b, hi = a < b ? b : a;
        const bool asc = (i & kk) == 0;
        pk[i] = asc ? lo : hi;
        pk[ixj] = asc ? hi : lo;
      }
      __syncthreads();
    }
  }
}

// One block sorts the entries [rs, rs + len) of a row, len <= kPackedPerThread
// x its threads; pk holds the power of two >= len words.
__device__ __forceinline__ void sort_packed(uint64_t* adj, uint32_t* eid, uint32_t* ekey, uint32_t rs, uint32_t len,
                                            int mode, unsigned long long* err, unsigned long long* pk) {
  uint32_t cap = 64;
  while (cap < len) cap <<= 1;
  if (mode == kSortById) {
    for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x)
      pk[i] = i < len ? (key_by_col(adj[rs + i]) << 12) | i : ~0ull;
    __syncthreads();
    bitonic_packed(pk, cap);
    for (uint32_t i = threadIdx.x + 1; i < len; i += blockDim.x)
      if ((pk[i] >> 12) == (pk[i - 1] >> 12)) report(err, rs + i, -UBT_ERR_DUPLICATE_EDGE);
  } else {
    for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x)
      pk[i] = i < len ? (key_by_absq(adj[rs + i]) << 12) | i : ~0ull;
    __syncthreads();
    bitonic_packed(pk, cap);
  }
  // gather every entry's sources before any thread overwrites the list
  uint64_t e[kPackedPerThread];
  uint32_t d[kPackedPerThread], y[kPackedPerThread];
#pragma unroll
  for (int c = 0; c < kPackedPerThread; c++) {
    const uint32_t i = threadIdx.x + c * blockDim.x;
    if (i < len) {
      const uint32_t w = (uint32_t)(pk[i] & 0xFFFu);
      e[c] = adj[rs + w];
      d[c] = eid[rs + w];
      y[c] = ekey ? ekey[rs + w] : 0u;
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < kPackedPerThread; c++) {
    const uint32_t i = threadIdx.x + c * blockDim.x;
    if (i < len) {
      adj[rs + i] = e[c];
      eid[rs + i] = d[c];
      if (ekey) ekey[rs + i] = y[c];
    }
  }
  __syncthreads();
}

// One launch per class takes the rows of the list with lo < len <= hi, with
// hi / 2 threads (at most 512): every thread has a comparator at every stage.
__global__ void __launch_bounds__(kPackedSortThreads)
k_sort_long_rows_packed(const uint32_t* __restrict__ rows, uint32_t nrows, const uint32_t* __restrict__ row_ptr,
                        uint64_t* adj, uint32_t* eid, uint32_t* ekey, int mode, unsigned long long* err,
                        uint32_t lo, uint32_t hi) {
  extern __shared__ __align__(16) unsigned long long pk[];  // hi words
  for (uint32_t r = blockIdx.x; r < nrows; r += gridDim.x) {
    const uint32_t u = rows[r];
    const uint32_t rs = row_ptr[u], len = row_ptr[u + 1] - rs;
    if (len <= lo || len > hi) continue;
    if (len > kPackedMax || len > kPackedPerThread * blockDim.x) {  // the launches never give such a row here
      if (threadIdx.x == 0) report(err, rs, -UBT_ERR_INVALID_ARG);
      continue;
    }
    sort_packed(adj, eid, ekey, rs, len, mode, err, pk);
  }
}

// the block sorts of every row of the list (lengths warp_max + 1 .. smem_max),
// by class: (128, 256] with 128 threads, (256, 512] with 256, longer with 512
ubt_status launch_block_sorts(const uint32_t* rows, uint32_t nrows, const uint32_t* row_ptr, uint64_t* adj, uint32_t* eid,
                        uint32_t* ekey, int mode, unsigned long long* err, uint32_t warp_max, uint32_t smem_max,
                        int sms, cudaStream_t s) {
  const uint32_t bounds[4] = {128, 256, 512, kPackedMax};
  for (int c = 0; c < 3; c++) {
    const uint32_t lo = bounds[c], hi = c == 2 ? std::max(smem_max, 512u) : bounds[c + 1];
    if (hi <= warp_max || lo >= smem_max) continue;
    const int threads = (int)std::min<uint32_t>(hi / 2, kPackedSortThreads);
    const size_t smem = (size_t)hi * 8;
    UBT_CUDA(cudaFuncSetAttribute(k_sort_long_rows_packed, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int per_sm = std::max(1, std::min(2048 / threads, (int)(200 * 1024 / smem)));
    const int g = (int)std::min<unsigned long long>(nrows, (unsigned long long)sms * per_sm);
    k_sort_long_rows_packed<<<g, threads, smem, s>>>(rows, nrows, row_ptr, adj, eid, ekey, mode, err, lo, hi);
  }
  return UBT_OK;
}

// Longer lists: one block per list, bitonic network in a per-block global
// slice (lists longer than the "sort_smem_max" tuning).  A list longer than a
// slice names a vertex twice: each of its vertices has at least its length as
// degree, so distinct ones are at most sqrt(2m).
__global__ void k_sort_long_rows(const uint32_t* __restrict__ rows, uint32_t nrows, const uint32_t* __restrict__ row_ptr,
                                 uint64_t* adj, uint32_t* eid, uint32_t* ekey, unsigned long long* err,
                                 char* gtmp, int64_t gtmp_cap) {
  for (uint32_t r = blockIdx.x; r < nrows; r += gridDim.x) {
    const uint32_t u = rows[r];
    const uint32_t rs = row_ptr[u], re = row_ptr[u + 1];
    const uint32_t len = re - rs;
    if ((int64_t)len > gtmp_cap) {
      if (threadIdx.x == 0) report(err, rs, -UBT_ERR_DUPLICATE_EDGE);
      continue;
    }
    uint32_t cap = 64;
    while (cap < len) cap <<= 1;
    char* base = gtmp + (size_t)blockIdx.x * (size_t)gtmp_cap * 24;
    uint64_t* key = (uint64_t*)base;
    uint64_t* ev = key + cap;
    uint32_t* iv = (uint32_t*)(ev + cap);
    uint32_t* yv = iv + cap;
    for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x) {
      if (i < len) {
        ev[i] = adj[rs + i];
        iv[i] = eid[rs + i];
        yv[i] = ekey ? ekey[rs + i] : 0u;
        key[i] = key_by_col(ev[i]);
      } else {
        key[i] = ~0ull; ev[i] = ~0ull; iv[i] = 0; yv[i] = 0;
      }
    }
    __syncthreads();
    for (uint32_t kk = 2; kk <= cap; kk <<= 1) {
      for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
        for (uint32_t i = threadIdx.x; i < cap; i += blockDim.x) {
          const uint32_t ixj = i ^ j;
          if (ixj > i) {
            const bool asc = (i & kk) == 0;
            const uint64_t a = key[i], b = key[ixj];
            if ((a > b) == asc && a != b) {
              key[i] = b; key[ixj] = a;
              uint64_t te = ev[i]; ev[i] = ev[ixj]; ev[ixj] = te;
              uint32_t ti = iv[i]; iv[i] = iv[ixj]; iv[ixj] = ti;
              uint32_t ty = yv[i]; yv[i] = yv[ixj]; yv[ixj] = ty;
            }
          }
        }
        __syncthreads();
      }
    }
    for (uint32_t i = threadIdx.x + 1; i < len; i += blockDim.x)
      if (key[i] == key[i - 1]) report(err, rs + i, -UBT_ERR_DUPLICATE_EDGE);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < len; i += blockDim.x) {
      adj[rs + i] = ev[i];
      eid[rs + i] = iv[i];
      if (ekey) ekey[rs + i] = yv[i];
    }
    __syncthreads();
  }
}

// Rows longer than 32: counts[2] of 33..128, or up to warp_max and at most
// smem_max (warp sort, listed from the end of `mid`), counts[0] of the others
// up to smem_max (block sort in shared memory, from the start of `mid`),
// counts[1] longer (block sort in global memory, `huge`).
__global__ void k_collect_long(int64_t n, const uint32_t* __restrict__ row_ptr, uint32_t smem_max, uint32_t warp_max,
                               uint32_t* mid, uint32_t* huge, unsigned long long* counts) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t len = row_ptr[u + 1] - row_ptr[u];
    if (len <= 32) continue;
    if (len <= 128 || (len <= warp_max && len <= smem_max))
      mid[n - 1 - (int64_t)atomicAdd(&counts[2], 1ull)] = (uint32_t)u;
    else if (len <= smem_max) mid[atomicAdd(&counts[0], 1ull)] = (uint32_t)u;
    else huge[atomicAdd(&counts[1], 1ull)] = (uint32_t)u;
  }
}

// rowid[p] = the row that holds CSR position p, and the forward entries that
// name a vertex: its degree less its own list (one thread per row)
__global__ void k_row_ids(int64_t n, const uint32_t* __restrict__ row_ptr, const uint32_t* __restrict__ deg,
                          const uint32_t* __restrict__ vid, uint32_t* __restrict__ rowid, uint32_t* __restrict__ indeg) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = row_ptr[u], e = row_ptr[u + 1];
    indeg[u] = deg[vid[u]] - (e - b);
    for (uint32_t p = b; p < e; p++) rowid[p] = (uint32_t)u;
  }
}

// Pair words grouped by owner.  next[v] holds the next free position of owner
// v's pairs in its low half (it starts at pair_ptr[v]) and the streamed work
// so far in its high half, in units of kWorkUnit entries (rounded up per pair), so one
// 64-bit atomic places a pair and adds its work.  absq (FIXED, or null): a
// histogram of |q| >> 9 over one warp's edges in eight.  streamed: the sum of
// the streamed lengths.
//
// Every list starts with the first vertices, so their counters would take a
// returning atomic from most rows, one after another in L2: a block ranks the
// pairs of the first kHotOwners vertices among its kFillTile entries in shared
// memory and reserves one range per vertex (Chung-Lu of 1e6 vertices: 656 -> 185 us).
// Counts and work are 32-bit words there: a returning 64-bit shared-memory add
// goes round a loop once per lane of the same address, and where one vertex is
// in every row (a star of 2e6 leaves) that was the kernel (329 us, now 25).
// What remains is bound by the atomics' and the pair words' random sectors.
constexpr uint32_t kWorkUnit = 8;
constexpr int kFillThreads = 256, kFillItems = 16;
constexpr int64_t kFillTile = kFillThreads * kFillItems;
constexpr uint32_t kHotOwners = 1024;
__global__ void __launch_bounds__(kFillThreads)
k_pair_fill(int64_t m, const uint32_t* __restrict__ row_ptr, const uint64_t* __restrict__ adj,
            const uint32_t* __restrict__ rowid, unsigned long long* __restrict__ next, uint64_t* __restrict__ pairs,
            unsigned long long* __restrict__ absq, unsigned long long* __restrict__ streamed) {
  __shared__ uint32_t s_q[65];
  __shared__ uint32_t s_hot[kHotOwners], s_work[kHotOwners];  // count, then the reserved base; work
  for (int i = threadIdx.x; i < 65; i += kFillThreads) s_q[i] = 0;
  unsigned long long sum = 0;
  for (int64_t base = blockIdx.x * kFillTile; base < m; base += (int64_t)gridDim.x * kFillTile) {
    for (uint32_t i = threadIdx.x; i < kHotOwners; i += kFillThreads) s_hot[i] = s_work[i] = 0;
    __syncthreads();
    uint32_t v[kFillItems], at[kFillItems];
    unsigned long long word[kFillItems];
#pragma unroll
    for (int j = 0; j < kFillItems; j++) {
      const int64_t i = base + j * kFillThreads + threadIdx.x;
      v[j] = kEmpty;
      if (i >= m) continue;
      const uint64_t e = adj[i];
      v[j] = adj_col(e);
      const uint32_t start = row_ptr[rowid[i]], len = (uint32_t)i - start;
      uint32_t aq = 0;
      if (absq) {
        const int32_t q = adj_q(e);
        aq = (uint32_t)(q < 0 ? -q : q);
        if (((i >> 5) & 7) == 0) atomicAdd(&s_q[aq >> 9], 1u);
      }
      word[j] = pair_pack(start, len, aq >> 1);
      sum += len;
      const uint32_t units = (len + kWorkUnit - 1) / kWorkUnit;
      if (v[j] < kHotOwners) {
        at[j] = atomicAdd(&s_hot[v[j]], 1u);
        if (units) atomicAdd(&s_work[v[j]], units);
      } else {
        at[j] = (uint32_t)atomicAdd(&next[v[j]], ((unsigned long long)units << 32) | 1ull);
      }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < kHotOwners; i += kFillThreads) {
      const uint32_t c = s_hot[i];
      if (c) s_hot[i] = (uint32_t)atomicAdd(&next[i], ((unsigned long long)s_work[i] << 32) | c);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kFillItems; j++)
      if (v[j] != kEmpty) pairs[v[j] < kHotOwners ? s_hot[v[j]] + at[j] : at[j]] = word[j];
    __syncthreads();
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
  if (lane_id() == 0 && sum) atomicAdd(streamed, sum);
  if (absq) {
    __syncthreads();
    for (int i = threadIdx.x; i < 65; i += kFillThreads)
      if (s_q[i]) atomicAdd(&absq[i], (unsigned long long)s_q[i]);
  }
}

constexpr uint8_t kNoTask = 0xFF;
constexpr int kLgMax = 47;   // work buckets 2^0 .. 2^47 (undirected owners)
constexpr int kLgTask = 40;  // and of the traversal's owners: lg * kTaskClasses + class < 255
constexpr int kTaskBuckets = kTaskClasses * (kLgTask + 1);
static_assert(kTaskBuckets <= kNoTask, "a bucket is one byte");

// Per owner x (one thread): its streamed work (from k_pair_fill), the log2
// bucket and class; bucket[x] = lg * kTaskClasses + cls, or kNoTask (no list entries or
// no pairs: no triangle can be found there).  Per-block counts in shared
// memory, one global atomic per block and bucket.  An owner of more than
// kHeavyPairs pairs is a block task whatever its work (whose 32 bits could
// wrap there).
// A table is a bitmap where the vertices it can hold -- the ones before x in
// its graph's range -- are at most block_bits (block tasks) or warp_bits (warp
// tasks), else a hash table.
// stats: [0] oriented wedges sum_v in(v) |N>(v)| (Alg. 1's probes), [1] longest
//        list, [2] streamed entries (set by k_pair_fill), [3] longest list of
//        a kHubHash task, [4] of a kHubBits task, [5] largest range of one,
//        [6] first pair of a vertex from merge_from on, [7] owners whose tasks
//        are block tasks,
//        [kStatBuckets + bucket] bucket sizes
constexpr uint32_t kHeavyPairs = 1u << 16;
constexpr int kStatBuckets = 8;
// A pair's own loads count as this many streamed entries.
constexpr unsigned long long kPairWork = 16;
// An owner whose work exceeds part_work is several block tasks, each with its
// own copy of the table and a share of the pairs, so that no owner's work is
// the length of the query.  With part_work >= the whole work / kMaxParts at
// most kMaxParts tasks are added.
constexpr unsigned long long kPartWork = 1 << 17, kMaxParts = 1 << 15;
__device__ __forceinline__ unsigned long long whole_work(unsigned long long streamed, int64_t m) {
  return streamed + (kWorkUnit + kPairWork) * (unsigned long long)m;  // an upper bound of the owners' sum
}
__device__ __forceinline__ unsigned long long owner_work(unsigned long long next, uint32_t np) {
  return np ? (next >> 32) * kWorkUnit + kPairWork * np : 0ull;
}
__device__ __forceinline__ uint32_t owner_parts(unsigned long long work, unsigned long long whole) {
  const unsigned long long part = max(min(kPartWork, max(4096ull, whole / 2048)), whole / kMaxParts + 1);
  return (uint32_t)min(work / part + 1, kMaxParts);
}
__global__ void k_row_stats(int64_t n, int64_t m, const uint32_t* __restrict__ row_ptr, const uint32_t* __restrict__ pair_ptr,
                            const unsigned long long* __restrict__ work, const uint32_t* __restrict__ vgraph,
                            const uint32_t* __restrict__ gstart, uint32_t hub_thr, uint32_t giant_thr,
                            unsigned long long block_work, uint32_t block_bits, uint32_t warp_bits, int64_t merge_from,
                            uint8_t* __restrict__ bucket, unsigned long long* stats) {
  __shared__ uint32_t s_cnt[kTaskBuckets];
  __shared__ unsigned long long s_wedges;
  __shared__ uint32_t s_max, s_hash, s_len, s_bits, s_hubs;
  for (int i = threadIdx.x; i < kTaskBuckets; i += blockDim.x) s_cnt[i] = 0;
  if (threadIdx.x == 0) { s_wedges = 0; s_max = 0; s_hash = 0; s_len = 0; s_bits = 0; s_hubs = 0; }
  __syncthreads();
  const unsigned long long whole = whole_work(stats[2], m);
  // the default limit on small graphs: smaller, so that one warp's work is not the whole query's length
  if (block_work == kBlockWork) block_work = min(block_work, max(2048ull, whole / 4096));
  unsigned long long wedges = 0;
  uint32_t mx = 0, hash = 0, blen = 0, bits = 0, hubs = 0;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t len = row_ptr[x + 1] - row_ptr[x];
    const uint32_t np = pair_ptr[x + 1] - pair_ptr[x];
    const unsigned long long w = owner_work(work[x], np);
    uint8_t b = kNoTask;
    wedges += (unsigned long long)np * len;
    if (x == merge_from) stats[6] = pair_ptr[x];
    if (len > 0 && np > 0 && x < merge_from) {
      const uint32_t range = (uint32_t)x - (gstart ? gstart[vgraph[x]] : 0u);
      const bool block = len > hub_thr || w > block_work || np > kHeavyPairs;
      const int cls = len > giant_thr ? kGiant
                      : block ? (range <= block_bits && len <= kBitsLen ? kHubBits : kHubHash) : (range <= warp_bits ? kMedBits : kMedHash);
      int lg = w ? 63 - __clzll(w) : 0;
      lg = lg > kLgTask ? kLgTask : lg;
      b = (uint8_t)(lg * kTaskClasses + cls);
      atomicAdd(&s_cnt[b], cls <= kHubBits ? owner_parts(w, whole) : 1u);
      hubs += cls <= kHubBits ? 1u : 0u;
      if (cls == kHubHash) hash = max(hash, len);
      if (cls == kHubBits) {
        blen = max(blen, len);
        bits = max(bits, range);
      }
    }
    bucket[x] = b;
    mx = max(mx, len);
  }
  atomicAdd(&s_wedges, wedges);
  atomicMax(&s_max, mx);
  atomicMax(&s_hash, hash);
  atomicMax(&s_len, blen);
  atomicMax(&s_bits, bits);
  if (hubs) atomicAdd(&s_hubs, hubs);
  __syncthreads();
  for (int i = threadIdx.x; i < kTaskBuckets; i += blockDim.x)
    if (s_cnt[i]) atomicAdd(&stats[kStatBuckets + i], (unsigned long long)s_cnt[i]);
  if (threadIdx.x == 0) {
    atomicAdd(&stats[0], s_wedges);
    atomicMax(&stats[1], (unsigned long long)s_max);
    atomicMax(&stats[3], (unsigned long long)s_hash);
    atomicMax(&stats[4], (unsigned long long)s_len);
    atomicMax(&stats[5], (unsigned long long)s_bits);
    if (s_hubs) atomicAdd(&stats[7], (unsigned long long)s_hubs);
  }
}

// Task lists, by class and in a class by falling bucket: every block ranks its
// owners' tasks per bucket in shared memory and reserves one range per bucket
// with a single global atomic.  Where a bucket starts follows from the bucket
// sizes, summed up by each block: a copy of them to the host and the starts
// back, with a wait between, was 15 us of every build.  cursor: zero before.
__global__ void k_fill_lists(int64_t n, int64_t m, const unsigned long long* __restrict__ work,
                             const uint32_t* __restrict__ pair_ptr, const uint8_t* __restrict__ bucket,
                             const unsigned long long* __restrict__ stats, unsigned long long* cursor,
                             uint64_t* __restrict__ lists) {
  __shared__ uint32_t s_cnt[kTaskBuckets];
  __shared__ unsigned long long s_base[kTaskBuckets];
  __shared__ uint32_t s_first[kTaskBuckets], s_all[kTaskClasses], s_class[kTaskClasses];
  const unsigned long long whole = whole_work(stats[2], m);
  for (int i = threadIdx.x; i < kTaskBuckets; i += blockDim.x) s_first[i] = (uint32_t)stats[kStatBuckets + i];
  __syncthreads();
  if (threadIdx.x < kTaskClasses) {  // a class's buckets, the largest work first
    uint32_t run = 0;
    for (int b = kLgTask * kTaskClasses + threadIdx.x; b >= 0; b -= kTaskClasses) {
      const uint32_t size = s_first[b];
      s_first[b] = run;
      run += size;
    }
    s_all[threadIdx.x] = run;
  }
  __syncthreads();
  if (threadIdx.x < kTaskClasses) {
    uint32_t run = 0;
    for (int c = 0; c < (int)threadIdx.x; c++) run += s_all[c];
    s_class[threadIdx.x] = run;
  }
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    for (int i = threadIdx.x; i < kTaskBuckets; i += blockDim.x) s_cnt[i] = 0;
    __syncthreads();
    const int64_t x = base + threadIdx.x;
    const uint8_t b = x < n ? bucket[x] : kNoTask;
    uint32_t rank = 0, parts = 1;
    if (b != kNoTask) {
      if (b % kTaskClasses <= kHubBits) parts = owner_parts(owner_work(work[x], pair_ptr[x + 1] - pair_ptr[x]), whole);
      rank = atomicAdd(&s_cnt[b], parts);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kTaskBuckets; i += blockDim.x)
      if (s_cnt[i]) s_base[i] = s_class[i % kTaskClasses] + s_first[i] + atomicAdd(&cursor[i], (unsigned long long)s_cnt[i]);
    __syncthreads();
    if (b != kNoTask)
      for (uint32_t i = 0; i < parts; i++)
        lists[s_base[b] + rank + i] = (uint32_t)x | ((uint64_t)i << 32) | ((uint64_t)(parts - 1) << 48);
    __syncthreads();
  }
}

// ---------------------------------------------------------------- undirected AEO adjacency

// both directions of every edge, in row order of arrival (sorted below), and
// the row of every position, so that the passes over the entries below take
// one thread an entry: a warp per row left the row of a hub -- tens of thousands
// of entries -- to one warp, which was the length of the pass (Chung-Lu of 1e6
// vertices, four passes: 2.96 ms, now 0.6)
__global__ void k_uscatter(int64_t m, const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                           const uint32_t* __restrict__ k, const uint32_t* __restrict__ uptr,
                           uint32_t* __restrict__ ufill, uint64_t* __restrict__ uadj, uint32_t* __restrict__ ueid,
                           uint32_t* __restrict__ urow) {
  const uint32_t lane = lane_id();
  UBT_FOR_EDGE_WARPS(base, m) {
    const int64_t i = base + lane;
    const bool on = i < m;
    const uint32_t a = on ? src[i] : 0u, b = on ? dst[i] : 0u;
    const uint32_t sa = add_by_runs(ufill, a, on);
    if (!on) continue;
    const uint32_t val = (uint32_t)(int32_t)(32768 - (int32_t)k[i]);
    const uint32_t pa = uptr[a] + sa;
    const uint32_t pb = uptr[b] + atomicAdd(&ufill[b], 1u);
    uadj[pa] = adj_pack(b, val);
    ueid[pa] = (uint32_t)i;
    urow[pa] = a;
    uadj[pb] = adj_pack(a, val);
    ueid[pb] = (uint32_t)i;
    urow[pb] = b;
  }
}

// Rows longer than the shared-memory sort limit: their runs of `chunk` entries
// are sorted one block each, then merged pairwise between two buffers, every
// entry finding its place by a binary search in the other run.  One block per
// row and a bitonic network in global memory took as long as the longest row
// (Chung-Lu of 1e6 vertices, rows up to 50,000: 2.46 ms, now 0.42).
__global__ void __launch_bounds__(kPackedSortThreads)
k_sort_chunks(const uint32_t* __restrict__ rows, uint32_t nrows, const uint32_t* __restrict__ row_ptr, uint64_t* adj,
              uint32_t* eid, unsigned long long* err, uint32_t chunk) {
  extern __shared__ __align__(16) unsigned long long pk[];  // chunk words
  for (uint32_t r = blockIdx.x; r < nrows; r += gridDim.x) {
    const uint32_t rs = row_ptr[rows[r]], len = row_ptr[rows[r] + 1] - rs;
    for (uint64_t c = (uint64_t)blockIdx.y * chunk; c < len; c += (uint64_t)gridDim.y * chunk)
      sort_packed(adj, eid, nullptr, rs + (uint32_t)c, min(chunk, len - (uint32_t)c), kSortByAbsq, err, pk);
  }
}
__global__ void k_merge_runs(const uint32_t* __restrict__ rows, uint32_t nrows, const uint32_t* __restrict__ row_ptr,
                             const uint64_t* __restrict__ adj, const uint32_t* __restrict__ eid,
                             uint64_t* __restrict__ adj_out, uint32_t* __restrict__ eid_out, uint64_t width) {
  for (uint32_t r = blockIdx.x; r < nrows; r += gridDim.x) {
    const uint32_t rs = row_ptr[rows[r]], len = row_ptr[rows[r] + 1] - rs;
    for (uint64_t i = (uint64_t)blockIdx.y * blockDim.x + threadIdx.x; i < len; i += (uint64_t)gridDim.y * blockDim.x) {
      const uint64_t run = i / width, base = run * width, other = (run ^ 1) * width;
      const uint64_t e = adj[rs + i], key = key_by_absq(e);
      uint64_t lo = min((uint64_t)len, other), hi = min((uint64_t)len, other + width);
      while (lo < hi) {  // entries of the other run before this one (keys are distinct)
        const uint64_t mid = (lo + hi) >> 1;
        if (key_by_absq(adj[rs + mid]) < key) lo = mid + 1; else hi = mid;
      }
      const uint64_t at = rs + (other < base ? lo + (i - base) : i + (lo - min((uint64_t)len, other)));
      adj_out[at] = e;
      eid_out[at] = eid[rs + i];
    }
  }
}
// adj_tmp, eid_tmp: as long as the rows; max_len: an upper bound of their lengths
ubt_status sort_huge_rows(const uint32_t* rows, uint32_t nrows, const uint32_t* row_ptr, uint64_t* adj, uint32_t* eid,
                          uint64_t* adj_tmp, uint32_t* eid_tmp, unsigned long long* err, uint32_t chunk,
                          uint64_t max_len, int sms, cudaStream_t s) {
  const unsigned gx = std::min<uint32_t>(nrows, 65535u);
  const unsigned gy = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((max_len + chunk - 1) / chunk, 4 * sms / gx + 1));
  const size_t smem = (size_t)chunk * 8;
  k_sort_chunks<<<dim3(gx, gy), kPackedSortThreads, smem, s>>>(rows, nrows, row_ptr, adj, eid, err, chunk);
  uint64_t* src = adj;
  uint32_t* srce = eid;
  uint64_t* dst = adj_tmp;
  uint32_t* dste = eid_tmp;
  const unsigned my = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((max_len + 255) / 256, 32 * sms / gx + 1));
  // a last round whose runs have no other run copies the rows back where needed
  for (uint64_t width = chunk; width < max_len || src != adj; width *= 2) {
    k_merge_runs<<<dim3(gx, my), 256, 0, s>>>(rows, nrows, row_ptr, src, srce, dst, dste, width);
    std::swap(src, dst);
    std::swap(srce, dste);
  }
  UBT_CUDA(cudaGetLastError());
  return UBT_OK;
}

// epos[2e + side] = position of edge e in the row of its smaller (side 0) or
// larger (side 1) endpoint; umir[p] = the position of p's edge in the other row
__global__ void k_uepos(int64_t m2, const uint32_t* __restrict__ urow, const uint64_t* __restrict__ uadj,
                        const uint32_t* __restrict__ ueid, uint32_t* __restrict__ epos) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < m2; p += (int64_t)gridDim.x * blockDim.x)
    epos[2 * (size_t)ueid[p] + (urow[p] > adj_col(uadj[p]) ? 1 : 0)] = (uint32_t)p;
}
__global__ void k_umirror(int64_t m, const uint32_t* __restrict__ epos, uint32_t* __restrict__ umir) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t p0 = epos[2 * e], p1 = epos[2 * e + 1];
    umir[p0] = p1;
    umir[p1] = p0;
  }
}

// Edge index: every input edge once.  The table has at least four times as
// many slots as edges, so every insert finds a free slot; the loop bound is a
// self-check.
__global__ void k_edge_index(int64_t m, const uint32_t* __restrict__ src, const uint32_t* __restrict__ dst,
                             const uint32_t* __restrict__ k, uint4* __restrict__ eslots, uint64_t slots, int shift,
                             uint32_t* __restrict__ filter, unsigned long long* err) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = edge_index_key(src[i], dst[i]);
    atomicOr(&filter[edge_index_home(key, shift + kEdgeFilterLog)], edge_filter_bits(key));
    uint64_t h = edge_index_home(key, shift);
    uint64_t it = 0;
    for (; it < slots; it++) {
      unsigned long long* slot_key = reinterpret_cast<unsigned long long*>(&eslots[h]);
      if (atomicCAS(slot_key, (unsigned long long)kEdgeIndexEmpty, (unsigned long long)key) == kEdgeIndexEmpty) {
        eslots[h].z = (uint32_t)(int32_t)(32768 - (int32_t)k[i]);
        break;
      }
      h = (h + 1) & (slots - 1);
    }
    if (it == slots) report(err, i, -UBT_ERR_INVALID_ARG);
  }
}

// AEO traversal: edge x-y is handled by x, the endpoint with the longer list
// (ties: the larger id), which holds the hash table; y's list is streamed.
__device__ inline bool aeo_owns(uint32_t x, uint32_t y, uint32_t dx, uint32_t dy) {
  return dx > dy || (dx == dy && x > y);
}
// The pairs keep the order of the rows -- an owner's strongest edges first -- so
// that the edges a warp takes together pass or fail the cutoffs together: placed
// by atomics, in the order that warps came, they cost k_aeo up to a fifth
// (Chung-Lu of 1e6 vertices, t = 0.8: 9.3-10.0 ms, in order 8.5).  own[c]: which of the
// entries [32 c, 32 c + 32) belong to their row's vertex, cnt[c] how many; the
// scan of cnt then places every pair and every owner's first one.
// work[x]: the entries that x's edges stream.
__global__ void k_apair_own(int64_t m2, const uint32_t* __restrict__ uptr, const uint64_t* __restrict__ uadj,
                            const uint32_t* __restrict__ urow, uint32_t* __restrict__ own_bits,
                            uint32_t* __restrict__ cnt, unsigned long long* __restrict__ work) {
  const uint32_t lane = lane_id();
  UBT_FOR_EDGE_WARPS(base, m2) {
    const int64_t p = base + lane;
    uint32_t x = kEmpty, dy = 0;
    bool own = false;
    if (p < m2) {
      x = urow[p];
      const uint32_t y = adj_col(uadj[p]);
      dy = uptr[y + 1] - uptr[y];
      own = aeo_owns(x, y, uptr[x + 1] - uptr[x], dy);
    }
    const unsigned bits = __ballot_sync(kFull, own);
    if (lane == 0) {
      own_bits[base >> 5] = bits;
      cnt[base >> 5] = __popc(bits);
    }
    // the entries of a row are neighbours: one add per row that the warp holds
    const unsigned row = __match_any_sync(kFull, x);
    unsigned long long sum = own ? dy : 0ull;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long o = __shfl_up_sync(kFull, sum, d);
      if (lane >= (uint32_t)d && ((row >> (lane - d)) & 1u)) sum += o;
    }
    if ((int)lane == 31 - __clz((int)row) && sum) atomicAdd(&work[x], sum);
  }
}
// pairs before entry p (m2: all)
__device__ __forceinline__ uint32_t apairs_before(uint32_t p, const uint32_t* __restrict__ own_bits,
                                                  const uint32_t* __restrict__ before) {
  const uint32_t in = p & 31u;
  return before[p >> 5] + (in ? __popc(own_bits[p >> 5] & ((1u << in) - 1u)) : 0u);
}
__global__ void k_apair_ptr(int64_t n, const uint32_t* __restrict__ uptr, const uint32_t* __restrict__ own_bits,
                            const uint32_t* __restrict__ before, uint32_t* __restrict__ apair_ptr) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= n; x += (int64_t)gridDim.x * blockDim.x)
    apair_ptr[x] = apairs_before(uptr[x], own_bits, before);
}
// pair words by owner: streamed endpoint | position of the edge in x's row << 32
__global__ void k_apair_fill(int64_t m2, const uint64_t* __restrict__ uadj, const uint32_t* __restrict__ own_bits,
                             const uint32_t* __restrict__ before, uint64_t* __restrict__ apairs) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < m2; p += (int64_t)gridDim.x * blockDim.x)
    if ((own_bits[p >> 5] >> (p & 31)) & 1u)
      apairs[apairs_before((uint32_t)p, own_bits, before)] = ((uint64_t)p << 32) | adj_col(uadj[p]);
}
// owners by decreasing log2 of their streamed work, those with rows longer
// than kAeoWarpRow (whole-block tasks) first: bucket = lg * 2 + (1 if block)
constexpr uint32_t kAeoWarpRow = 128;
__global__ void k_afill_lists(int64_t n, const uint32_t* __restrict__ uptr, const uint32_t* __restrict__ apair_ptr,
                              const unsigned long long* __restrict__ work, unsigned long long* cursor,
                              uint32_t* __restrict__ lists, int count_only) {
  constexpr int kB = 2 * (kLgMax + 1);
  __shared__ uint32_t s_cnt[kB];
  __shared__ unsigned long long s_base[kB];
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    for (int i = threadIdx.x; i < kB; i += blockDim.x) s_cnt[i] = 0;
    __syncthreads();
    const int64_t x = base + threadIdx.x;
    const bool on = x < n && apair_ptr[x + 1] != apair_ptr[x];
    int b = 0;
    uint32_t rank = 0;
    if (on) {
      const unsigned long long w = work[x];
      b = (w ? 63 - __clzll(w) : 0) * 2 + (uptr[x + 1] - uptr[x] > kAeoWarpRow ? 1 : 0);
      rank = atomicAdd(&s_cnt[b], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kB; i += blockDim.x)
      if (s_cnt[i]) s_base[i] = atomicAdd(&cursor[i], (unsigned long long)s_cnt[i]);
    __syncthreads();
    if (on && !count_only) lists[s_base[b] + rank] = (uint32_t)x;
    __syncthreads();
  }
}

struct BuildLayout {
  // persistent
  Scratch* scratch;
  uint32_t* vid;
  uint32_t* row_ptr;
  uint64_t* adj;
  uint32_t* eid;
  uint32_t* rowid;
  uint32_t* ekey;
  uint32_t* keep;        // pruned queries (FIXED graphs)
  uint32_t* keep_tmp;
  uint32_t* pair_ptr;
  uint64_t* pairs;
  uint64_t* lists;       // tasks by class
  uint32_t* vgraph;
  uint32_t* gstart;
  uint32_t* uptr;        // undirected AEO adjacency (optional)
  uint64_t* uadj;
  uint32_t* ueid;
  uint32_t* umir;
  uint32_t* uepos;
  uint32_t* apair_ptr;
  uint64_t* apairs;
  uint32_t* alist;
  unsigned long long* awork;
  unsigned long long* lqueue;  // long vertex samples of a local-count call (with the undirected rows)
  uint32_t* efilter;           // filter of the edge index, in the build temporaries' place
  uint4* eslots;               // edge index (optional)
  int64_t eh_slots;
  unsigned long long* gacc;
  unsigned long long* bacc;
  uint32_t* gtab;
  // build temporaries
  uint32_t* deg;
  uint32_t* fill;
  uint32_t* rank;              // number of every id
  uint32_t* rank_tmp;          // ids between passes
  uint32_t* rank_hist;
  uint32_t* vgraph_id;         // batch: graph of every id
  uint32_t* scan_tmp;
  uint32_t* mid_rows;
  uint32_t* huge_rows;
  uint8_t* bucket;
  unsigned long long* work;    // next pair position and streamed work per owner
  unsigned long long* stats;   // kStats counters, as many cursors, 4 counters, 65 |q| classes
  char* sort_tmp;
  size_t total;
};
constexpr int kStats = kStatBuckets + kTaskBuckets;
constexpr int kLengths = 2 * kStats, kClasses = kLengths + 4, kBuildWords = kClasses + 65;
static_assert(kStats >= 2 * (kLgMax + 1), "the undirected owners' cursors share the array");

int64_t list_bound(int64_t n, int64_t m) {
  // a forward list under Node Order holds at most sqrt(2m) entries
  int64_t b = (int64_t)sqrt(2.0 * (double)m) + 2;
  return std::min<int64_t>(b, std::max<int64_t>(n, 1));
}

int64_t pow2_at_least(int64_t x) {
  int64_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

BuildLayout layout(void* ws, size_t cap, int64_t n, int64_t m, int32_t kind, const ubt_graph_opts* opts,
                   int sm_count) {
  Carver c(ws, cap);
  BuildLayout L;
  const bool has_key = opts && opts->d_edge_key;
  const bool batch = opts && opts->d_vertex_offsets;
  const int64_t ng = batch ? opts->n_graphs : 1;
  const int64_t n1 = std::max<int64_t>(n, 1);
  L.scratch = c.take<Scratch>(1);
  L.vid = c.take<uint32_t>(n1);
  L.row_ptr = c.take<uint32_t>(n + 1);
  L.adj = c.take<uint64_t>(std::max<int64_t>(m, 1));
  L.eid = c.take<uint32_t>(std::max<int64_t>(m, 1));
  L.rowid = kind == UBT_GRAPH_FIXED ? c.take<uint32_t>(std::max<int64_t>(m, 1)) : nullptr;
  L.keep = kind == UBT_GRAPH_FIXED ? c.take<uint32_t>(m + 2) : nullptr;
  L.keep_tmp = kind == UBT_GRAPH_FIXED ? c.take<uint32_t>(scan_tmp_words(m)) : nullptr;
  L.ekey = has_key ? c.take<uint32_t>(std::max<int64_t>(m, 1)) : nullptr;
  L.pair_ptr = c.take<uint32_t>(n + 1);
  L.pairs = c.take<uint64_t>(std::max<int64_t>(m, 1));
  L.lists = c.take<uint64_t>(n1 + kMaxParts);
  L.vgraph = batch ? c.take<uint32_t>(n1) : nullptr;
  L.gstart = batch ? c.take<uint32_t>(ng) : nullptr;
  const bool und = opts && (opts->flags & UBT_OPT_UNDIRECTED);
  L.uptr = und ? c.take<uint32_t>(n + 1) : nullptr;
  L.uadj = und ? c.take<uint64_t>(std::max<int64_t>(2 * m, 1)) : nullptr;
  L.ueid = und ? c.take<uint32_t>(std::max<int64_t>(2 * m, 1)) : nullptr;
  // one piece: the long rows' sort uses both as its second buffer of entries
  L.uepos = und ? c.take<uint32_t>(std::max<int64_t>(4 * m, 2)) : nullptr;
  L.umir = und ? L.uepos + 2 * m : nullptr;
  L.apair_ptr = und ? c.take<uint32_t>(n + 1) : nullptr;
  L.apairs = und ? c.take<uint64_t>(std::max<int64_t>(m, 1)) : nullptr;
  L.alist = und ? c.take<uint32_t>(n1) : nullptr;
  L.awork = und ? c.take<unsigned long long>(n1) : nullptr;
  L.lqueue = und ? c.take<unsigned long long>(kLongHead + kLongQueue) : nullptr;
  const bool eidx = und && (opts->flags & UBT_OPT_EDGE_INDEX);
  L.eh_slots = eidx ? pow2_at_least(std::max<int64_t>(4 * m, 64)) : 0;
  L.eslots = eidx ? c.take<uint4>(L.eh_slots) : nullptr;
  L.gacc = c.take<unsigned long long>(std::max<int64_t>(m, 1));
  // only enumeration (FIXED graphs) reads the row ids of a built graph; the
  // build of a REAL one keeps them in the accumulators
  if (!L.rowid) L.rowid = (uint32_t*)L.gacc;
  // per graph: T, sum_lo, sum_hi (expected counts) of a batch
  L.bacc = c.take<unsigned long long>(3 * std::max<int64_t>(ng, 1));
  const int64_t gslots = gtab_slots_for(m);
  L.gtab = gslots ? c.take<uint32_t>((size_t)gslots * 3 * (size_t)sm_count) : nullptr;
  L.stats = c.take<unsigned long long>(kBuildWords);
  const size_t temporaries = c.off;
  L.deg = c.take<uint32_t>(n + 1);
  L.fill = c.take<uint32_t>(n + 1);
  L.rank = c.take<uint32_t>(n1);
  L.rank_tmp = c.take<uint32_t>(n1);
  const int64_t rank_hist = 256 * ((n + kRankTile - 1) / kRankTile);
  L.rank_hist = c.take<uint32_t>(rank_hist + 1);
  L.vgraph_id = batch ? c.take<uint32_t>(n1) : nullptr;
  L.scan_tmp = c.take<uint32_t>(scan_tmp_words(std::max(std::max(n, ng), rank_hist)) + 2);
  L.mid_rows = c.take<uint32_t>(n1);
  L.huge_rows = c.take<uint32_t>(n1);
  L.bucket = c.take<uint8_t>(n1);
  L.work = c.take<unsigned long long>(n1);
  const int64_t lb = list_bound(n, m);
  L.sort_tmp = lb > tuning().sort_smem_max
                   ? c.take<char>((size_t)kSortHugeBlocks * (size_t)pow2_at_least(lb) * 24) : nullptr;
  // the filter takes the temporaries' place: the index is the last thing built
  L.efilter = nullptr;
  if (eidx) {
    const size_t end = c.off;
    c.off = temporaries;
    L.efilter = c.take<uint32_t>((size_t)(L.eh_slots >> kEdgeFilterLog));
    c.off = std::max(c.off, end);
  }
  L.total = c.off + 256;
  return L;
}

// L.vid and L.rank from the degrees (and, for a batch, L.vgraph_id)
ubt_status rank_vertices(const BuildLayout& L, int64_t n, unsigned long long max_deg, int64_t n_graphs, cudaStream_t s) {
  RankKey pass[8];
  int np = 0;
  for (int sh = 0; sh == 0 || (max_deg >> sh) != 0; sh += 8) pass[np++] = RankKey{L.deg, sh, 255u};
  if (L.vgraph_id)
    for (int sh = 0; sh < 32 && ((uint64_t)(n_graphs - 1) >> sh) != 0; sh += 8)
      pass[np++] = RankKey{L.vgraph_id, sh, 0u};
  const unsigned tiles = (unsigned)((n + kRankTile - 1) / kRankTile);
  const uint32_t* in = nullptr;  // the ids n - 1 .. 0
  for (int i = 0; i < np; i++) {
    uint32_t* out = (np - 1 - i) % 2 == 0 ? L.vid : L.rank_tmp;  // the last pass ends in vid
    k_rank_count<<<tiles, kRankThreads, 0, s>>>(n, in, pass[i], L.rank_hist);
    UBT_CUDA(exclusive_scan_u32(L.rank_hist, L.rank_hist, 256 * (int64_t)tiles, L.scan_tmp, s));
    k_rank_scatter<<<tiles, kRankThreads, 0, s>>>(n, in, pass[i], L.rank_hist, out, i == np - 1 ? L.rank : nullptr);
    in = out;
  }
  UBT_CUDA(cudaGetLastError());
  return UBT_OK;
}

int device_sm_count(int* dev) {
  int d = 0, sms = 0;
  cudaGetDevice(&d);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
  if (dev) *dev = d;
  return sms > 0 ? sms : 1;
}

ubt_status status_from_err(unsigned long long e) {
  if (e == ~0ull) return UBT_OK;
  return -(ubt_status)(e & 0xFF);
}

}  // namespace

int64_t gtab_slots_for(int64_t m) {
  // a list's table holds 4x its entries (power of two); lists whose table
  // exceeds the shared-memory limit get one in global memory, sized for the
  // longest possible list
  const int64_t need = pow2_at_least(4 * list_bound(INT64_MAX / 4, m));
  return need > tuning().smem_table_max ? need : 0;
}

}  // namespace ubt

using namespace ubt;

extern "C" ubt_status ubt_graph_workspace_size(int64_t n, int64_t m, int32_t flags, const ubt_graph_opts* opts,
                                               size_t* h_bytes) {
  if (!h_bytes || n < 0 || m < 0 || n >= 0xFFFFFFFFll || m >= 0xFFFFFFFFll) return UBT_ERR_INVALID_ARG;
  if (flags != UBT_GRAPH_FIXED && flags != UBT_GRAPH_REAL) return UBT_ERR_INVALID_ARG;
  if (opts && opts->d_vertex_offsets && opts->n_graphs < 1) return UBT_ERR_INVALID_ARG;
  BuildLayout L = layout(nullptr, 0, n, m, flags, opts, device_sm_count(nullptr));
  *h_bytes = L.total;
  return UBT_OK;
}

extern "C" ubt_status ubt_create_graph(int64_t n, int64_t m, const uint32_t* d_src, const uint32_t* d_dst,
                                       const uint32_t* d_k, const float* d_p, int32_t flags,
                                       const ubt_graph_opts* opts, void* d_workspace, size_t ws_bytes,
                                       void* stream, ubt_graph** h_out) {
  UBT_RANGE("ubt_create_graph");
  if (!h_out) return UBT_ERR_INVALID_ARG;
  *h_out = nullptr;
  if (n < 0 || m < 0 || n >= 0xFFFFFFFFll || m >= 0xFFFFFFFFll) return UBT_ERR_INVALID_ARG;
  if (flags == UBT_GRAPH_FIXED) {
    if ((m > 0 && !d_k) || d_p) return UBT_ERR_INVALID_ARG;
  } else if (flags == UBT_GRAPH_REAL) {
    if ((m > 0 && !d_p) || d_k) return UBT_ERR_INVALID_ARG;
  } else {
    return UBT_ERR_INVALID_ARG;
  }
  if (m > 0 && (!d_src || !d_dst)) return UBT_ERR_INVALID_ARG;
  const bool und = opts && (opts->flags & UBT_OPT_UNDIRECTED);
  if (opts && (opts->flags & ~(int64_t)(UBT_OPT_UNDIRECTED | UBT_OPT_EDGE_INDEX))) return UBT_ERR_INVALID_ARG;
  if (opts && (opts->flags & UBT_OPT_EDGE_INDEX) && !und) return UBT_ERR_INVALID_ARG;
  if (und && flags != UBT_GRAPH_FIXED) return UBT_ERR_UNSUPPORTED;
  if (!d_workspace || ((uintptr_t)d_workspace & 255)) return UBT_ERR_INVALID_ARG;
  const bool batch = opts && opts->d_vertex_offsets;
  if (batch && opts->n_graphs < 1) return UBT_ERR_INVALID_ARG;
  const int64_t ng = batch ? opts->n_graphs : 1;
  int dev = 0;
  const int sms = device_sm_count(&dev);
  BuildLayout L = layout(d_workspace, ws_bytes, n, m, flags, opts, sms);
  if (ws_bytes < L.total) return UBT_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t s = (cudaStream_t)stream;
  const Tuning& T = tuning();
  const int64_t hub_thr = std::max<int64_t>(2, T.hub_threshold);
  const int64_t giant_thr = std::max<int64_t>(hub_thr, T.smem_table_max / 4);
  const int pull = T.pull ? 1 : 0;
  const int64_t block_work = std::max<int64_t>(1, T.block_work);

  UBT_CUDA(cudaMemsetAsync(L.scratch, 0, sizeof(Scratch), s));
  UBT_CUDA(cudaMemsetAsync(L.deg, 0, (size_t)((char*)(L.fill + n + 1) - (char*)L.deg), s));  // deg and fill
  UBT_CUDA(cudaMemsetAsync(L.stats, 0, sizeof(unsigned long long) * kBuildWords, s));
  // what the host reads lies together, as a copy to the host is 15 us: bucket
  // statistics, list cursors, row lengths (first the largest degree), the
  // first error, |q| classes
  unsigned long long* const lcount = L.stats + kLengths;
  unsigned long long* const derr = lcount + 3;
  UBT_CUDA(cudaMemsetAsync(derr, 0xFF, sizeof(unsigned long long), s));
  const int thr = 256;
  const int grid_e = (int)std::min<int64_t>(std::max<int64_t>((m + thr - 1) / thr, 1), (int64_t)sms * 32);
  const int grid_v = (int)std::min<int64_t>(std::max<int64_t>((n + thr - 1) / thr, 1), (int64_t)sms * 32);
  const int grid_w = (int)std::min<int64_t>(std::max<int64_t>((n + 7) / 8, 1), (int64_t)sms * 32);

  if (batch) {
    k_vertex_graph<<<grid_v, thr, 0, s>>>(opts->d_vertex_offsets, opts->n_graphs, n, L.vgraph_id);
  }
  // 1. validate + degree
  NvtxPhases phase;
  phase.next("build: validate and degree");
  if (m > 0)
    k_validate_degree<<<grid_e, thr, 0, s>>>(n, m, d_src, d_dst, d_k, d_p, L.vgraph_id, L.deg, derr);
  if (n > 0) k_degree_stats<<<grid_v, thr, 0, s>>>(n, L.deg, lcount);
  unsigned long long deg_stats[4] = {0, 0, 0, 0};
  UBT_CUDA(cudaMemcpyAsync(deg_stats, lcount, sizeof(deg_stats), cudaMemcpyDeviceToHost, s));
  UBT_CUDA(cudaStreamSynchronize(s));
  ubt_status st = status_from_err(deg_stats[3]);
  if (st != UBT_OK) return st;
  // 2. orientation + CSR offsets
  phase.next("build: orient, scatter, sort");
  if (n > 0) {
    UBT_CUDA(cudaMemsetAsync(lcount, 0, 3 * sizeof(unsigned long long), s));
    st = rank_vertices(L, n, deg_stats[0], ng, s);
    if (st != UBT_OK) return st;
    if (batch) k_rank_graphs<<<grid_v, thr, 0, s>>>(n, L.vid, L.vgraph_id, L.vgraph, opts->d_vertex_offsets, ng, L.gstart);
  }
  if (m > 0) k_out_degree<<<grid_e, thr, 0, s>>>(m, d_src, d_dst, L.rank, L.fill);
  UBT_CUDA(exclusive_scan_u32(L.fill, L.row_ptr, n, L.scan_tmp, s, L.fill));
  if (m > 0)
    k_scatter<<<grid_e, thr, 0, s>>>(m, d_src, d_dst, d_k, d_p, L.rank, L.fill, L.adj, L.eid,
                                     opts ? opts->d_edge_key : nullptr, L.ekey);
  // 3. sort every forward list
  const int fixed = flags == UBT_GRAPH_FIXED;
  const int mode = kSortById;
  if (n > 0) {
    k_sort_short_rows<<<grid_w, thr, 0, s>>>(n, L.row_ptr, L.adj, L.eid, L.ekey, mode, derr);
    const uint32_t sort_smem = (uint32_t)tuning().sort_smem_max;
    const uint32_t warp_max = (uint32_t)tuning().warp_sort_max;
    k_collect_long<<<grid_v, thr, 0, s>>>(n, L.row_ptr, sort_smem, warp_max, L.mid_rows, L.huge_rows, lcount);
    unsigned long long lc[3] = {0, 0, 0};
    UBT_CUDA(cudaMemcpyAsync(lc, lcount, sizeof(lc), cudaMemcpyDeviceToHost, s));
    UBT_CUDA(cudaStreamSynchronize(s));
    if (lc[2]) {
      st = launch_mid_sorts(L.mid_rows + (n - (int64_t)lc[2]), (uint32_t)lc[2], L.row_ptr, L.adj, L.eid, L.ekey, mode,
                            derr, warp_max, sms, thr, s);
      if (st != UBT_OK) return st;
    }
    if (lc[0]) {
      st = launch_block_sorts(L.mid_rows, (uint32_t)lc[0], L.row_ptr, L.adj, L.eid, L.ekey, mode, derr,
                              warp_max, sort_smem, sms, s);
      if (st != UBT_OK) return st;
    }
    if (lc[1]) {
      const int64_t cap = L.sort_tmp ? pow2_at_least(list_bound(n, m)) : 0;
      const int g = (int)std::min<unsigned long long>(lc[1], (unsigned long long)kSortHugeBlocks);
      k_sort_long_rows<<<g, 1024, 0, s>>>(L.huge_rows, (uint32_t)lc[1], L.row_ptr, L.adj, L.eid, L.ekey,
                                          derr, L.sort_tmp, cap);
    }
    UBT_CUDA(cudaGetLastError());
  }
  // 4. pairs grouped by owner.  (Rows with a duplicate are known by now, but
  // not here: the host looks once, at the end.  Nothing below reads more of
  // such rows than their lengths.)
  phase.next("build: pairs and work lists");
  unsigned long long* absq = fixed ? L.stats + kClasses : nullptr;
  if (n == 0) UBT_CUDA(cudaMemsetAsync(L.pair_ptr, 0, sizeof(uint32_t), s));
  if (n > 0) {
    k_row_ids<<<grid_v, thr, 0, s>>>(n, L.row_ptr, L.deg, L.vid, L.rowid, L.fill);
    UBT_CUDA(exclusive_scan_u32(L.fill, L.pair_ptr, n, L.scan_tmp, s, nullptr, L.work));
    const int grid_f = (int)std::min<int64_t>((m + kFillTile - 1) / kFillTile, (int64_t)sms * 8);
    if (m > 0) k_pair_fill<<<grid_f, kFillThreads, 0, s>>>(m, L.row_ptr, L.adj, L.rowid, L.work, L.pairs, absq, &L.stats[2]);
    UBT_CUDA(cudaGetLastError());
  }
  // 5. work lists: the owners of every task class by decreasing work bucket
  unsigned long long stats[kBuildWords];
  // vertices of degree <= kMergeDegree are the last ones (of a batch, every
  // graph's last ones: its pairs all go to tables)
  const int64_t merge_from = batch ? n : (int64_t)deg_stats[1];
  if (n > 0) {
    k_row_stats<<<grid_v, thr, 0, s>>>(n, m, L.row_ptr, L.pair_ptr, L.work, L.vgraph, L.gstart, (uint32_t)hub_thr,
                                      (uint32_t)giant_thr, (unsigned long long)block_work, (uint32_t)T.block_bits,
                                      (uint32_t)T.warp_bits, merge_from, L.bucket, L.stats);
    k_fill_lists<<<grid_v, thr, 0, s>>>(n, m, L.work, L.pair_ptr, L.bucket, L.stats, L.stats + kStats, L.lists);
    UBT_CUDA(cudaGetLastError());
  }
  UBT_CUDA(cudaMemcpyAsync(stats, L.stats, sizeof(stats), cudaMemcpyDeviceToHost, s));
  UBT_CUDA(cudaStreamSynchronize(s));
  st = status_from_err(stats[kLengths + 3]);
  if (st != UBT_OK) return st;
  int64_t count_cls[kTaskClasses] = {}, first_cls[kTaskClasses] = {};
  for (int b = 0; b < kTaskBuckets; b++) count_cls[b % kTaskClasses] += (int64_t)stats[kStatBuckets + b];
  for (int c = 1; c < kTaskClasses; c++) first_cls[c] = first_cls[c - 1] + count_cls[c - 1];
  // 6. undirected adjacency in Absolute Edge Order, its mirror positions and
  //    the AEO pair partition (optional)
  int64_t n_aowners = 0, n_ablock = 0, max_udeg = 0;
  if (und && n > 0) {
    phase.next("build: undirected rows in Absolute Edge Order");
    uint32_t* urow = (uint32_t*)L.gacc;  // the row of every entry, in the (not yet used) accumulators
    const int64_t m2 = 2 * m;
    const int grid_2 = (int)std::min<int64_t>(std::max<int64_t>((m2 + thr - 1) / thr, 1), (int64_t)sms * 32);
    UBT_CUDA(exclusive_scan_u32(L.deg, L.uptr, n, L.scan_tmp, s));
    UBT_CUDA(cudaMemsetAsync(L.fill, 0, sizeof(uint32_t) * (n + 1), s));
    if (m > 0) k_uscatter<<<grid_e, thr, 0, s>>>(m, d_src, d_dst, d_k, L.uptr, L.fill, L.uadj, L.ueid, urow);
    k_sort_short_rows<<<grid_w, thr, 0, s>>>(n, L.uptr, L.uadj, L.ueid, nullptr, kSortByAbsq, derr);
    const uint32_t sort_smem = (uint32_t)tuning().sort_smem_max;
    UBT_CUDA(cudaMemsetAsync(lcount, 0, 3 * sizeof(unsigned long long), s));
    const uint32_t warp_max = (uint32_t)tuning().warp_sort_max;
    k_collect_long<<<grid_v, thr, 0, s>>>(n, L.uptr, sort_smem, warp_max, L.mid_rows, L.huge_rows, lcount);
    unsigned long long lc[3] = {0, 0, 0};
    UBT_CUDA(cudaMemcpyAsync(lc, lcount, sizeof(lc), cudaMemcpyDeviceToHost, s));
    UBT_CUDA(cudaStreamSynchronize(s));
    if (lc[2]) {
      st = launch_mid_sorts(L.mid_rows + (n - (int64_t)lc[2]), (uint32_t)lc[2], L.uptr, L.uadj, L.ueid, nullptr,
                            kSortByAbsq, derr, warp_max, sms, thr, s);
      if (st != UBT_OK) return st;
    }
    if (lc[0]) {
      st = launch_block_sorts(L.mid_rows, (uint32_t)lc[0], L.uptr, L.uadj, L.ueid, nullptr, kSortByAbsq,
                              derr, warp_max, sort_smem, sms, s);
      if (st != UBT_OK) return st;
    }
    if (lc[1]) {
      st = sort_huge_rows(L.huge_rows, (uint32_t)lc[1], L.uptr, L.uadj, L.ueid, (uint64_t*)L.uepos,
                          (uint32_t*)L.apairs, derr, sort_smem, deg_stats[0], sms, s);
      if (st != UBT_OK) return st;
    }
    if (m > 0) {
      k_uepos<<<grid_2, thr, 0, s>>>(m2, urow, L.uadj, L.ueid, L.uepos);
      k_umirror<<<grid_e, thr, 0, s>>>(m, L.uepos, L.umir);
    }
    // which entries are pairs, and how many before each 32 of them, in the (not
    // yet used) words of the kept counts: 2 ceil(2m / 32) + 1 <= m + 2
    const int64_t chunks = (m2 + 31) / 32;
    uint32_t* const own_bits = L.keep;
    uint32_t* const before = L.keep + chunks;
    UBT_CUDA(cudaMemsetAsync(L.awork, 0, sizeof(unsigned long long) * n, s));
    if (m > 0) k_apair_own<<<grid_2, thr, 0, s>>>(m2, L.uptr, L.uadj, urow, own_bits, before, L.awork);
    UBT_CUDA(exclusive_scan_u32(before, before, chunks, L.keep_tmp, s));
    k_apair_ptr<<<grid_v, thr, 0, s>>>(n, L.uptr, own_bits, before, L.apair_ptr);
    if (m > 0) k_apair_fill<<<grid_2, thr, 0, s>>>(m2, L.uadj, own_bits, before, L.apairs);
    unsigned long long* acur = L.stats;  // 2 (kLgMax + 1) cursors
    constexpr int kAB = 2 * (kLgMax + 1);
    UBT_CUDA(cudaMemsetAsync(acur, 0, sizeof(unsigned long long) * kAB, s));
    k_afill_lists<<<grid_v, thr, 0, s>>>(n, L.uptr, L.apair_ptr, L.awork, acur, L.alist, 1);
    unsigned long long acount[kAB];
    UBT_CUDA(cudaMemcpyAsync(acount, acur, sizeof(acount), cudaMemcpyDeviceToHost, s));
    UBT_CUDA(cudaStreamSynchronize(s));
    unsigned long long run = 0;
    for (int cls = 1; cls >= 0; cls--) {  // block tasks, then warp tasks
      for (int lg = kLgMax; lg >= 0; lg--) {
        const unsigned long long c = acount[lg * 2 + cls];
        acount[lg * 2 + cls] = run;
        run += c;
      }
      if (cls == 1) n_ablock = (int64_t)run;
    }
    n_aowners = (int64_t)run;
    UBT_CUDA(cudaMemcpyAsync(acur, acount, sizeof(acount), cudaMemcpyHostToDevice, s));
    k_afill_lists<<<grid_v, thr, 0, s>>>(n, L.uptr, L.apair_ptr, L.awork, acur, L.alist, 0);
    if (L.eslots) {  // last: the filter lies where the build's temporaries were
      UBT_CUDA(cudaMemsetAsync(L.eslots, 0xFF, sizeof(uint4) * (size_t)L.eh_slots, s));
      UBT_CUDA(cudaMemsetAsync(L.efilter, 0, sizeof(uint32_t) * (size_t)(L.eh_slots >> kEdgeFilterLog), s));
      int lg = 0;
      while ((1ll << lg) < L.eh_slots) lg++;
      if (m > 0)
        k_edge_index<<<grid_e, thr, 0, s>>>(m, d_src, d_dst, d_k, L.eslots, (uint64_t)L.eh_slots, 64 - lg, L.efilter,
                                            derr);
    }
    unsigned long long err = 0;
    UBT_CUDA(cudaMemcpyAsync(&err, derr, sizeof(err), cudaMemcpyDeviceToHost, s));
    UBT_CUDA(cudaGetLastError());
    UBT_CUDA(cudaStreamSynchronize(s));
    max_udeg = (int64_t)deg_stats[0];
    st = status_from_err(err);
    if (st != UBT_OK) return st;
  }

  ubt_graph* g = new (std::nothrow) ubt_graph();
  if (!g) return UBT_ERR_INVALID_ARG;
  g->n = n;
  g->m = m;
  g->kind = flags;
  g->n_graphs = ng;
  g->vid = L.vid;
  g->row_ptr = L.row_ptr;
  g->adj = L.adj;
  g->eid = L.eid;
  g->rowid = flags == UBT_GRAPH_FIXED ? L.rowid : nullptr;
  g->keep = L.keep;
  g->keep_tmp = L.keep_tmp;
  for (int b = 64; b >= 0; b--) g->kept[b] = g->kept[b + 1] + (double)stats[kClasses + b];
  for (int b = 64; b >= 0; b--) g->kept[b] = g->kept[0] > 0 ? g->kept[b] / g->kept[0] : 1.0;
  g->ekey = L.ekey ? L.ekey : L.eid;
  g->pair_ptr = L.pair_ptr;
  g->pairs = L.pairs;
  for (int c = 0; c < kTaskClasses; c++) {
    g->lists[c] = L.lists + first_cls[c];
    g->n_tasks[c] = count_cls[c];
  }
  g->vgraph = L.vgraph;
  g->gstart = L.gstart;
  g->uptr = L.uptr;
  g->uadj = L.uadj;
  g->ueid = L.ueid;
  g->umir = L.umir;
  g->uepos = L.uepos;
  g->apair_ptr = L.apair_ptr;
  g->apairs = L.apairs;
  g->alist = L.alist;
  g->n_aowners = n_aowners;
  g->n_ablock = n_ablock;
  g->max_udeg = max_udeg;
  g->lqueue = L.lqueue;
  g->eslots = L.eslots;
  g->efilter = L.efilter;
  g->eh_slots = L.eh_slots;
  {
    int lg = 0;
    while ((1ll << lg) < L.eh_slots) lg++;
    g->eh_shift = 64 - lg;
  }
  g->gacc = L.gacc;
  g->bacc = L.bacc;
  g->gtab = L.gtab;
  g->gtab_slots = gtab_slots_for(m);
  g->gtab_blocks = L.gtab ? sms : 0;
  g->scratch = L.scratch;
  g->wedges = (int64_t)stats[0];
  g->max_out = (int64_t)stats[1];
  g->probes = (int64_t)stats[2];
  g->max_hash_len = (int64_t)stats[3];
  g->max_bits_len = (int64_t)stats[4];
  g->max_bits = (int64_t)stats[5];
  g->warp_bits = T.warp_bits;
  g->merge_first = merge_from < n ? (int64_t)stats[6] : m;
  g->hub_vertices = (int64_t)stats[7];
  g->hub_threshold = hub_thr;
  g->giant_threshold = giant_thr;
  g->block_work = block_work;
  g->pull = pull;
  g->device = dev;
  g->sm_count = sms;
  *h_out = g;
  return UBT_OK;
}

extern "C" ubt_status ubt_destroy_graph(ubt_graph* g) {
  if (!g) return UBT_ERR_INVALID_ARG;
  delete g;
  return UBT_OK;
}

extern "C" ubt_status ubt_graph_get_info(const ubt_graph* g, ubt_graph_info* h_info) {
  if (!g || !h_info) return UBT_ERR_INVALID_ARG;
  h_info->n = g->n;
  h_info->m = g->m;
  h_info->max_out_degree = g->max_out;
  h_info->hub_vertices = g->hub_vertices;
  h_info->wedges = g->wedges;
  h_info->kind = g->kind;
  h_info->probes = g->probes;
  return UBT_OK;
}

namespace ubt {
namespace {

// New edge values of a REAL graph: CSR position pos holds input edge eid[pos],
// so its value becomes s(p[eid[pos]]); the rows stay sorted (by vertex number).
// A p outside [0, 1] (or NaN) leaves the entry as it was and records the
// first such input index in the self-check word (code 6).
__global__ void k_set_edge_values(int64_t m, const float* __restrict__ p, const uint32_t* __restrict__ eid,
                                  uint64_t* __restrict__ adj, unsigned long long* guard) {
  for (int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; pos < m; pos += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t e = eid[pos];
    const float x = p[e];
    if (!(x >= 0.0f && x <= 1.0f)) {
      atomicCAS(guard, 0ull, (6ull << 56) | (unsigned long long)e);
      continue;
    }
    adj[pos] = adj_pack(adj_col(adj[pos]), real_valbits(x));
  }
}

}  // namespace
}  // namespace ubt

extern "C" ubt_status ubt_set_edge_values(ubt_graph* g, const float* d_p, void* stream) {
  UBT_RANGE("ubt_set_edge_values");
  if (!g || (!d_p && g->m > 0)) return UBT_ERR_INVALID_ARG;
  if (g->kind != UBT_GRAPH_REAL) return UBT_ERR_UNSUPPORTED;
  if (g->m == 0) return UBT_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int grid = (int)std::min<int64_t>((g->m + 255) / 256, (int64_t)g->sm_count * 8);
  k_set_edge_values<<<grid, 256, 0, s>>>(g->m, d_p, g->eid, g->adj, &g->scratch->guard);
  UBT_CUDA(cudaGetLastError());
  return UBT_OK;
}
