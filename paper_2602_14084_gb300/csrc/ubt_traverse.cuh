// ubt_traverse.cuh -- the triangle traversal every query runs.
//
// Forward edge iteration under Node Order (Alg. 1, Sec. 4): triangle {u,v,w}
// with u < v < w in Node Order is found exactly once, from its pair (u, v),
// as w in N>(u) n N>(v).  Every forward edge is one pair.  Alg. 1 streams
// N>(v) through a table of N>(u); here the later vertex v owns the pair (the
// "owner" x): the table holds N>(v), and of N>(u) only the part after v is
// streamed -- the entries of row u before v's position, as the rows are
// sorted latest vertex first (ubt_internal.cuh).
//
// GPU layout of that loop (two persistent kernels, three kinds of task):
//   * N>(x) becomes a table in shared memory that answers "is w in N>(x), and
//     with which edge value and CSR position":
//       bitmap  one bit per vertex before x in its graph's range, and where a
//               word's first entry is in the list: membership is one 4-byte
//               shared load, a hit's entry is found by counting bits (its CSR
//               position too) and its value loaded from the list's values.
//               The touched words are cleared after the task, so a table costs
//               what its list is long, not its range.
//       hash    neighbour -> edge value, CSR position in 4-slot buckets read
//               with one 16-byte load, at most 1/4 full: for owners whose range
//               is too large for a bitmap (low-degree vertices of large graphs)
//     A shared-memory load serves 32 random 4-byte words in 3-4 cycles and 32
//     random 16-byte buckets in about 10, which bound the hash form.
//   * The pairs of x are handed to one warp 32 at a time.  The lists N>(s)
//     are streamed with coalesced 8-byte loads: long lists one after another
//     by the whole warp, short lists concatenated ("flattened") so that every
//     lane has an entry (a "list" is the streamed part of a row).  Each entry w is probed in x's table; a hit is a
//     triangle and goes to the visitor with the three edge values and CSR
//     positions.
//   * Task classes, by owner:
//       giant   list longer than the shared-memory hash table: whole block, hash
//               table in a per-block slice of global memory
//       hub     long list or heavy streamed work: whole block, warps take
//               `unit` pairs at a time (bitmap or hash table)
//       medium  the rest: one warp, its own table (bitmap or hash)
//   * Owners of degree at most 32, the last in the numbering, have no table:
//     their pairs, consecutive in the pair array, are merged, one pair a lane
//     (both lists hold at most 32 entries).  They are most of the owners -- 2.1
//     of 2.5 million tasks, but 20 % of the pairs, of a Chung-Lu graph of 4e6
//     vertices -- and a warp task costs some 700 instructions before its first
//     probe.
//   * Probability pruning (FIXED graphs, level L > 0): an edge with |q_e| 2^30
//     < L is in no triangle with |P| >= L (Lemma 2: the other two factors are
//     at most 2^15).  Where a level removes enough (prune_pays), the query
//     first writes the kept entries of all rows in order (keep_entries) and
//     the traversal runs on those: `adj` holds the kept entries and keep[pos]
//     says how many lie before the unpruned position pos.  A pair that fails
//     is skipped from its pair word alone.  Otherwise nothing is pruned; the
//     visitors classify every product exactly either way.
//
// Hits go through a queue: a warp appends the triangles that its lanes find --
// the table slot, the two other edges' values, positions -- to a queue in
// shared memory and takes them 32 at a time, so that the table lookup of the
// value, the product and what the query does with it run on full warps
// instead of the third of the lanes that hits on average (a miss costs only
// the membership test and its part of the append).
//
// Visitors implement: smem_bytes(params, threads) (shared memory they need) /
// block_init / task_begin / task_end / block_end; item (what is queued of a
// triangle; with kMore the streamed edge's position too) and take (called by
// all 32 lanes of a warp, converged, with up to 32 queued triangles, `on` in
// the lanes that have one).  A visitor sees a triangle as
// (x, s, w): the pair edge x-s, the table edge x-w and the streamed edge s-w;
// s is given as an (unpruned) CSR position in its row, whose rowid it is.  A
// visitor may also define probed(n): after each batch of at most 32 pairs the
// whole warp calls it with n >= the number of entries the batch probed (the
// same n in every lane).
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "ubt_internal.cuh"


namespace ubt {

struct TravArgs {
  const uint32_t* row_ptr;
  const uint64_t* adj;
  const uint32_t* pair_ptr;    // pairs of owner x: [pair_ptr[x], pair_ptr[x + 1])
  const uint64_t* pairs;       // pair words (ubt_internal.cuh)
  const uint32_t* keep;        // pruned: kept entries before every position (adj holds the kept ones); else null
  const uint64_t* lists[kTaskClasses];  // owner | part << 32 | (parts - 1) << 48
  uint32_t n_tasks[kTaskClasses];
  const uint32_t* vgraph;      // batch: graph of every vertex and first vertex of every graph (else null)
  const uint32_t* gstart;
  uint32_t merge_first;     // pairs [merge_first, m) are merged
  uint32_t n, m;            // vertices, edges (bounds of the self-checks)
  Scratch* sc;              // task counters (zeroed before launch)
  uint32_t* gtab;           // giant tables: gtab_blocks x gtab_slots x 3 words
  uint32_t gtab_slots;      // power of two
  uint32_t gtab_blocks;
  uint32_t hub_slots;       // shared-memory hash table of a hub (power of two)
  uint32_t warp_slots;      // per-warp hash table (power of two)
  uint32_t hub_bits, hub_len;    // bitmap table of a hub: range and list
  uint32_t warp_bits, warp_len;  // and of a medium task
  uint32_t unit;            // pairs per warp step in block tasks
  uint32_t batch;           // warp tasks taken per grab
  uint32_t long_min;        // streamed lists at least this long take the whole-warp path
  uint32_t long_tail;       // 1: a long list's last < 64 entries join the concatenated short lists
  uint32_t qmin2;           // pairs with |q| >> 1 below this are skipped (0: none)
};

__device__ __forceinline__ uint32_t hash_slot(uint32_t w, int shift) { return (w * 0x9E3779B1u) >> shift; }

// visitors with a probed(n) member are told how many entries each batch probed
template <class V, class = void>
struct HasProbed : std::false_type {};
template <class V>
struct HasProbed<V, std::void_t<decltype(std::declval<V&>().probed(0u))>> : std::true_type {};

// visitors with a finish() member write their answer in the traversal's last block
template <class V, class = void>
struct HasFinish : std::false_type {};
template <class V>
struct HasFinish<V, std::void_t<decltype(std::declval<V&>().finish())>> : std::true_type {};

// the fewest threads of the main kernel's blocks a visitor wants (kMinThreads)
template <class V, class = void>
struct MinThreads {
  static constexpr int value = 64;
};
template <class V>
struct MinThreads<V, std::void_t<decltype(V::kMinThreads)>> {
  static constexpr int value = V::kMinThreads;
};

// Self-checks record the first violated invariant in Scratch::guard and skip
// the offending access: 1 probe limit (find), 2 probe limit (insert),
// 3 neighbour id >= n, 4 list offsets out of order or past m, 5 table larger
// than its region.
enum : unsigned long long { kGuardFind = 1, kGuardInsert = 2, kGuardVertex = 3, kGuardList = 4, kGuardTable = 5 };
static __device__ __noinline__ void guard_fail(Scratch* sc, unsigned long long code, unsigned long long info) {
  atomicCAS(&sc->guard, 0ull, (code << 56) | (info & ((1ull << 56) - 1)));
}

__device__ __forceinline__ int64_t qabs(uint32_t valbits) {
  const int32_t q = (int32_t)valbits;
  return q < 0 ? -(int64_t)q : (int64_t)q;
}

// first index in [0, len) of a |q|-descending list whose |q| * c < L (len if none)
__device__ __forceinline__ uint32_t prune_prefix(const uint64_t* __restrict__ row, uint32_t len, int64_t c, int64_t L) {
  if (len == 0) return 0;
  if (qabs(adj_valbits(row[len - 1])) * c >= L) return len;
  if (qabs(adj_valbits(row[0])) * c < L) return 0;
  uint32_t lo = 0, hi = len - 1;  // row[lo] passes, row[hi] fails
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (qabs(adj_valbits(row[mid])) * c >= L) lo = mid; else hi = mid;
  }
  return hi;
}

// Hash table: key = neighbour id, val = edge value bits, pos = CSR position,
// in buckets of 4 slots (one 16-byte load reads a bucket's keys); at most 1/4
// of the slots are used, so nearly every lookup ends in its home bucket.
struct Table {
  uint32_t* key;
  uint32_t* val;
  uint32_t* pos;
  uint32_t bmask;  // buckets - 1
  int shift;
};

__device__ __forceinline__ Table make_table(uint32_t* base, uint32_t cap, uint32_t slots) {
  Table t;
  t.key = base;
  t.val = base + cap;
  t.pos = base + 2 * cap;
  const uint32_t nb = slots >> 2;
  t.bmask = nb - 1;
  t.shift = 32 - (31 - __clz((int)nb));
  return t;
}

// slots for a list: a power of two >= 4x its entries (min 32, i.e. 8 buckets)
__device__ __forceinline__ uint32_t slots_for(uint32_t entries) {
  uint32_t s = 32;
  while (s < 4 * entries) s <<= 1;
  return s;
}

// A bucket with a free slot ends every probe sequence, and there are more
// buckets than entries, so both loops end within bmask + 1 buckets; the limit
// is a self-check.  Slots of a bucket are taken in order (first free slot).
template <bool kPos = true>
__device__ __forceinline__ void table_insert(const Table& t, uint32_t w, uint32_t val, uint32_t pos, Scratch* sc) {
  uint32_t b = hash_slot(w, t.shift);
  for (uint32_t it = 0; it <= t.bmask; it++) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if (atomicCAS(&t.key[4 * b + i], kEmpty, w) == kEmpty) {
        t.val[4 * b + i] = val;
        if (kPos) t.pos[4 * b + i] = pos;
        return;
      }
    }
    b = (b + 1) & t.bmask;
  }
  guard_fail(sc, kGuardInsert, w);
}

// Find w in the table (kPos: also return the entry's CSR position).
//
// Inserts take the first free slot of a bucket and nothing is ever removed,
// so a bucket's used slots are a prefix and a bucket has room iff its last
// slot is empty; a key missing from a bucket with room is absent.  With at
// most 1/4 of the slots used, nearly every lookup reads one bucket and takes
// no branch.
template <bool kPos>
__device__ __forceinline__ bool table_find(const Table& t, uint32_t w, uint32_t& val, uint32_t& pos, Scratch* sc) {
  uint32_t b = hash_slot(w, t.shift);
  const uint4 k = reinterpret_cast<const uint4*>(t.key)[b];
  const bool m0 = k.x == w, m1 = k.y == w, m2 = k.z == w, m3 = k.w == w;
  bool hit = m0 | m1 | m2 | m3;
  uint32_t s = 4 * b + (m0 ? 0u : (m1 ? 1u : (m2 ? 2u : 3u)));
  if (!hit && k.w != kEmpty) {  // the home bucket is full: continue in the next ones
    bool ended = false;
    for (uint32_t it = 1; it <= t.bmask; it++) {
      b = (b + 1) & t.bmask;
      const uint4 kk = reinterpret_cast<const uint4*>(t.key)[b];
      const bool n0 = kk.x == w, n1 = kk.y == w, n2 = kk.z == w, n3 = kk.w == w;
      if (n0 | n1 | n2 | n3) {
        hit = true;
        s = 4 * b + (n0 ? 0u : (n1 ? 1u : (n2 ? 2u : 3u)));
        ended = true;
        break;
      }
      if (kk.w == kEmpty) {
        ended = true;
        break;
      }
    }
    if (!ended) guard_fail(sc, kGuardFind, w);
  }
  if (hit) {
    val = t.val[s];
    if (kPos) pos = t.pos[s];
  }
  return hit;
}

// Words of table memory per slot: visitors that need no CSR position keep
// only keys and values (8 bytes a slot), which lets more warp tables share
// an SM's shared memory.
template <bool kPos>
struct TableWords {
  static constexpr uint32_t kWords = kPos ? 3u : 2u;
};
// 32-bit words of shared memory a table of `slots` slots takes for visitor V
template <class V>
__host__ __device__ constexpr uint32_t table_words(uint32_t slots) {
  return slots * TableWords<V::kPos>::kWords;
}

// The slot of w for the 32 converged lanes of a warp (every lane calls it; a
// lane without an entry passes any key and ignores the result): the search
// past a full home bucket -- rare, at most 1/4 of the slots are used -- is
// entered by the whole warp only when some lane needs it, so that the common
// case runs without a divergent branch.
template <class T>
__device__ __forceinline__ bool table_slot_warp(const T& t, uint32_t w, uint32_t& slot, Scratch* sc) {
  uint32_t b = hash_slot(w, t.shift);
  const uint4 k = reinterpret_cast<const uint4*>(t.key)[b];
  const bool m0 = k.x == w, m1 = k.y == w, m2 = k.z == w, m3 = k.w == w;
  bool hit = m0 | m1 | m2 | m3;
  slot = 4 * b + (m0 ? 0u : (m1 ? 1u : (m2 ? 2u : 3u)));
  const bool more = !hit && k.w != kEmpty;
  if (__any_sync(kFull, more)) {
    if (more) {  // the home bucket is full: continue in the next ones
      bool ended = false;
      for (uint32_t it = 1; it <= t.bmask; it++) {
        b = (b + 1) & t.bmask;
        const uint4 kk = reinterpret_cast<const uint4*>(t.key)[b];
        const bool n0 = kk.x == w, n1 = kk.y == w, n2 = kk.z == w, n3 = kk.w == w;
        if (n0 | n1 | n2 | n3) {
          hit = true;
          slot = 4 * b + (n0 ? 0u : (n1 ? 1u : (n2 ? 2u : 3u)));
          ended = true;
          break;
        }
        if (kk.w == kEmpty) {
          ended = true;
          break;
        }
      }
      if (!ended) guard_fail(sc, kGuardFind, w);
    }
  }
  return hit;
}

// Per-lane description of one pair handed to probe_pairs: owner x (its list
// is the table), position and value of the pair edge, an unpruned position of
// the streamed row, and the streamed entries [vs, vs + dv) of adj.
struct Pair {
  uint32_t x, s, pe, qe, vs, dv;
};

// ------------------------------------------------------------ tables

// Bitmap of the list N>(x): a bit for every entry w, pre[word] = the list index
// of the word's first entry, val[i] the edge value of entry i.  Words are
// numbered by w >> 5 from the graph's first one, `w0`; the lookups use 32-bit
// shared-memory addresses of the (possibly unbacked) word 0, which saves the
// subtraction per probe.
struct BitTable {
  uint32_t* bits;   // all zero between tasks
  uint16_t* pre;
  uint32_t* val;
  uint32_t w0;      // first word of the graph's range
  uint32_t lo;      // first vertex of the graph's range
  uint32_t rs;      // CSR position of the list
  uint32_t abits, apre;  // shared addresses of words 0
};
#ifdef __CUDACC__
// the table for a graph that starts at vertex `first`
__device__ __forceinline__ void bit_table_graph(BitTable& t, uint32_t first) {
  t.lo = first;
  t.w0 = first >> 5;
  t.abits = (uint32_t)__cvta_generic_to_shared(t.bits) - 4u * t.w0;
  t.apre = (uint32_t)__cvta_generic_to_shared(t.pre) - 2u * t.w0;
}
__device__ __forceinline__ uint32_t lds32(uint32_t at) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t at) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(at) : "memory");
  return v;
}
#endif
__host__ __device__ inline uint32_t bit_words(uint32_t range) { return (range + 31) / 32 + 1; }  // any alignment of the first vertex
__host__ __device__ inline size_t bit_table_bytes(uint32_t range, uint32_t len) {
  const size_t w = bit_words(range);
  return (w * 4 + (w * 2 + 3) / 4 * 4 + (size_t)len * 4 + 15) / 16 * 16;
}
__device__ __forceinline__ BitTable bit_table_at(char* base, uint32_t range, uint32_t len) {
  const uint32_t w = bit_words(range);
  BitTable t;
  t.bits = (uint32_t*)base;
  t.val = t.bits + w;
  t.pre = (uint16_t*)(t.val + len);
  t.rs = 0;
  bit_table_graph(t, 0);
  return t;
}
// entries i0, i0 + step, ... of the list into the table / out of it again
__device__ __forceinline__ void bit_table_load(const BitTable& t, const uint64_t* __restrict__ adj, uint32_t len,
                                               uint32_t i0, uint32_t step) {
  for (uint32_t i = i0; i < len; i += step) {
    const uint64_t e = adj[t.rs + i];
    const uint32_t b = adj_col(e), w = (b >> 5) - t.w0;
    atomicOr(&t.bits[w], 1u << (b & 31));
    t.val[i] = adj_valbits(e);
    if (i == 0 || (adj_col(adj[t.rs + i - 1]) >> 5) - t.w0 != w) t.pre[w] = (uint16_t)i;
  }
}
__device__ __forceinline__ void bit_table_clear(const BitTable& t, const uint64_t* __restrict__ adj, uint32_t len,
                                                uint32_t i0, uint32_t step) {
  for (uint32_t i = i0; i < len; i += step) t.bits[(adj_col(adj[t.rs + i]) >> 5) - t.w0] = 0;
}

// Membership of U entries and, for a queued hit, its table entry: the edge
// value, CSR position and vertex.
__device__ __forceinline__ uint32_t none(const BitTable& t) { return t.lo; }  // a vertex that may be probed
template <int U>
__device__ __forceinline__ void find(const BitTable& t, const uint64_t (&e)[U], const bool (&act)[U], bool (&hit)[U],
                                     uint32_t (&slot)[U], Scratch*) {
  uint32_t word[U];
#pragma unroll
  for (int i = 0; i < U; i++) {
    slot[i] = adj_col(e[i]);
    word[i] = lds32(t.abits + 4u * (slot[i] >> 5));
  }
#pragma unroll
  for (int i = 0; i < U; i++) hit[i] = act[i] && ((word[i] >> (slot[i] & 31)) & 1u);
}
template <bool kPos>
__device__ __forceinline__ void entry(const BitTable& t, uint32_t slot, uint32_t& val, uint32_t& pos, uint32_t& w) {
  const uint32_t wi = slot >> 5;
  const uint32_t at = lds16(t.apre + 2u * wi) + __popc(lds32(t.abits + 4u * wi) & ((1u << (slot & 31)) - 1u));
  val = t.val[at];
  pos = t.rs + at;
  w = slot;
}
// A warp task's hash table: keys in 4-slot buckets and every key's list index;
// values come from the list itself, in L1 (6 bytes a slot instead of 8, or 12
// with CSR positions: the warp tables' shared memory is taken from L1, which
// the streamed rows need; Chung-Lu of 4e6 vertices, forward + backward: 7.4 -> 6.5 ms).
struct ListTable {
  uint32_t* key;
  uint16_t* at;
  const uint64_t* list;
  uint32_t rs;     // CSR position of the list
  uint32_t bmask;  // buckets - 1
  int shift;
};
__host__ __device__ inline size_t list_table_bytes(uint32_t slots) { return (size_t)slots * 6; }
__device__ __forceinline__ ListTable list_table_at(uint32_t* base, uint32_t slots, const uint64_t* adj, uint32_t rs) {
  ListTable t;
  t.key = base;
  t.at = (uint16_t*)(base + slots);
  t.list = adj + rs;
  t.rs = rs;
  const uint32_t nb = slots >> 2;
  t.bmask = nb - 1;
  t.shift = 32 - (31 - __clz((int)nb));
  return t;
}
__device__ __forceinline__ void list_table_insert(const ListTable& t, uint32_t i, Scratch* sc) {
  const uint32_t w = adj_col(t.list[i]);
  uint32_t b = hash_slot(w, t.shift);
  for (uint32_t it = 0; it <= t.bmask; it++) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (atomicCAS(&t.key[4 * b + k], kEmpty, w) == kEmpty) {
        t.at[4 * b + k] = (uint16_t)i;
        return;
      }
    }
    b = (b + 1) & t.bmask;
  }
  guard_fail(sc, kGuardInsert, w);
}
template <bool kPos>
__device__ __forceinline__ void entry(const ListTable& t, uint32_t slot, uint32_t& val, uint32_t& pos, uint32_t& w) {
  const uint32_t i = t.at[slot];
  val = adj_valbits(t.list[i]);
  pos = t.rs + i;
  w = t.key[slot];
}
__device__ __forceinline__ uint32_t none(const ListTable&) { return 0; }
template <int U>
__device__ __forceinline__ void find(const ListTable& t, const uint64_t (&e)[U], const bool (&act)[U], bool (&hit)[U],
                                     uint32_t (&slot)[U], Scratch* sc) {
#pragma unroll
  for (int i = 0; i < U; i++) {
    const bool found = table_slot_warp(t, adj_col(e[i]), slot[i], sc);
    hit[i] = act[i] && found;
  }
}
__device__ __forceinline__ uint32_t none(const Table&) { return 0; }
template <int U>
__device__ __forceinline__ void find(const Table& t, const uint64_t (&e)[U], const bool (&act)[U], bool (&hit)[U],
                                     uint32_t (&slot)[U], Scratch* sc) {
#pragma unroll
  for (int i = 0; i < U; i++) {
    const bool found = table_slot_warp(t, adj_col(e[i]), slot[i], sc);
    hit[i] = act[i] && found;
  }
}
template <bool kPos>
__device__ __forceinline__ void entry(const Table& t, uint32_t slot, uint32_t& val, uint32_t& pos, uint32_t& w) {
  val = t.val[slot];
  pos = kPos ? t.pos[slot] : 0u;
  w = t.key[slot];
}

// ------------------------------------------------------------ the queue of hits

// A warp's queue of items (V::Item, 8 or 16 bytes, the table slot in x) and, if
// V::kMore, one more word each.  Fewer than 32 are queued between steps; a
// step adds at most 32 V::kU.  Appending is a predicated store per entry, with
// no branch: most of the traversal's instructions are here.
template <class V>
struct Queue {
  static constexpr int kCap = 32 + 32 * V::kU;
  static constexpr uint32_t kItem = (uint32_t)sizeof(typename V::Item);
  static constexpr int kBytes = kCap * (int)(kItem + (V::kMore ? 4 : 0));
  typename V::Item* q;
  uint32_t* more;
  uint32_t base, end;  // shared addresses of the first item and past the last
  __device__ explicit Queue(char* mem)
      : q((typename V::Item*)mem), more((uint32_t*)(mem + kCap * kItem)),
        base((uint32_t)__cvta_generic_to_shared(mem)), end(base) {}
  __device__ __forceinline__ void append(bool hit, const typename V::Item& it, uint32_t extra, uint32_t lt) {
    const unsigned m = __ballot_sync(kFull, hit);
    const uint32_t at = end + kItem * __popc(m & lt);
    if constexpr (kItem == 8)
      asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.v2.u32 [%1], {%2, %3}; }" ::"r"((uint32_t)hit),
                   "r"(at), "r"(it.x), "r"(it.y) : "memory");
    else
      asm volatile("{ .reg .pred p; setp.ne.u32 p, %0, 0; @p st.shared.v4.u32 [%1], {%2, %3, %4, %5}; }" ::"r"(
                       (uint32_t)hit),
                   "r"(at), "r"(it.x), "r"(it.y), "r"(it.z), "r"(it.w) : "memory");
    if constexpr (V::kMore)
      if (hit) more[(at - base) / kItem] = extra;
    end += kItem * __popc(m);
  }
  // the last `cnt` <= 32 queued triangles to the visitor (kWhole: cnt is 32)
  template <bool kWhole, class T>
  __device__ __forceinline__ void take(const T& t, V& vis, uint32_t x, uint32_t cnt) {
    const uint32_t lane = lane_id();
    end -= kItem * cnt;
    const uint32_t first = (end - base) / kItem + lane;
    const bool on = kWhole || lane < cnt;
    typename V::Item it = {};
    uint32_t extra = 0, val = 0, pos = 0, w = 0;
    if (on) {
      it = q[first];
      if constexpr (V::kMore) extra = more[first];
      entry<V::kPos>(t, it.x, val, pos, w);
    }
    __syncwarp();
    vis.take(on, cnt, it, extra, x, val, pos, w);
  }
  template <class T>
  __device__ __forceinline__ void take_full(const T& t, V& vis, uint32_t x) {
    if (end - base >= 32 * kItem) {
      __syncwarp();
      do take<true>(t, vis, x, 32); while (end - base >= 32 * kItem);
    }
  }
  template <class T>
  __device__ __forceinline__ void take_all(const T& t, V& vis, uint32_t x) {
    __syncwarp();
    if (end != base) take<false>(t, vis, x, (end - base) / kItem);
  }
};

// U entries of streamed lists per lane (act: this lane has one; a lane
// without one passes an entry naming vertex none()): probed, the hits queued.
// q, pe: value and CSR position of the pair edge, s: the row's position, pos:
// of the entry.
template <class V, class T, int U>
__device__ __forceinline__ void probe(const T& t, V& vis, Queue<V>& queue, const uint64_t (&e)[U], const bool (&act)[U],
                                      uint32_t x, const uint32_t (&s)[U], const uint32_t (&q)[U],
                                      const uint32_t (&pe)[U], const uint32_t (&pos)[U], Scratch* sc) {
  static_assert(U <= V::kU, "the queue has room for kU entries a lane");
  bool hit[U];
  uint32_t slot[U];
  find<U>(t, e, act, hit, slot, sc);
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int i = 0; i < U; i++)
    queue.append(hit[i], V::item(slot[i], q[i], adj_valbits(e[i]), s[i], pe[i], pos[i]), pos[i], lt);
  queue.take_full(t, vis, x);
}

// The whole warp probes 32 U entries of one long list, U per lane, all loads
// issued before the probes: `row` and `pos` are the lane's first entry and its
// position, `left` the entries from lane 0's on.  kAll: all 32 U exist.
template <class V, class T, int U, bool kAll>
__device__ __forceinline__ void long_steps(const uint64_t* __restrict__ row, uint32_t pos0, uint32_t left, Scratch* sc,
                                           V& vis, Queue<V>& queue, const T& t, int lane, uint32_t x, uint32_t sj,
                                           uint32_t qj, uint32_t pj) {
  uint64_t e[U];
  bool act[U];
  uint32_t s[U], q[U], pe[U], pos[U];
#pragma unroll
  for (int i = 0; i < U; i++) {
    act[i] = kAll || 32 * i + lane < left;
    e[i] = act[i] ? row[32 * i] : (uint64_t)none(t);
    pos[i] = pos0 + 32 * i;
    s[i] = sj;
    q[i] = qj;
    pe[i] = pj;
  }
  probe<V, T, U>(t, vis, queue, e, act, x, s, q, pe, pos, sc);
}

// One warp probes the lists of up to 32 pairs (one per lane; empty ones have dv = 0).
template <class V, class T>
__device__ __forceinline__ void probe_pairs(const TravArgs& a, V& vis, Queue<V>& queue, const T& t, const Pair& pr) {
  const int lane = (int)lane_id();
  const uint64_t* __restrict__ adj = a.adj;
  Scratch* const sc = a.sc;
  uint32_t vs = pr.vs, dv = pr.dv;
  // long lists: one at a time, the whole warp streams it, V::kU entries per lane
  const uint32_t kLong = a.long_min;
  const bool tail_short = a.long_tail != 0;
  const bool was_long = dv >= kLong;
  unsigned longm = __ballot_sync(kFull, was_long);
  uint32_t probed = 0;  // entries of the long lists (the same in every lane)
  while (longm) {
    const int j = __ffs(longm) - 1;
    longm &= longm - 1;
    const uint32_t sj = __shfl_sync(kFull, pr.s, j);
    const uint32_t vsj = __shfl_sync(kFull, vs, j);
    const uint32_t dvj = __shfl_sync(kFull, dv, j);
    if constexpr (HasProbed<V>::value) probed += dvj;
    const uint32_t qj = __shfl_sync(kFull, pr.qe, j);
    const uint32_t pj = __shfl_sync(kFull, pr.pe, j);
    uint32_t left = dvj, pos = vsj + lane;
    const uint64_t* __restrict__ row = adj + vsj + lane;
    constexpr int kU = V::kU;
    while (left >= 32 * kU) {
      long_steps<V, T, kU, true>(row, pos, left, sc, vis, queue, t, lane, pr.x, sj, qj, pj);
      row += 32 * kU;
      pos += 32 * kU;
      left -= 32 * kU;
    }
    if (tail_short) {
      // full half-chunk, then the rest (< 64 entries) is streamed with the short lists
      if (kU > 2 && left >= 64) {
        long_steps<V, T, 2, true>(row, pos, left, sc, vis, queue, t, lane, pr.x, sj, qj, pj);
        left -= 64;
      }
      if (lane == j) {
        vs += dvj - left;
        dv = left;
      }
    } else {
      for (; left; left -= min(left, 64u)) {
        long_steps<V, T, 2, false>(row, pos, left, sc, vis, queue, t, lane, pr.x, sj, qj, pj);
        row += 64;
        pos += 64;
      }
    }
  }
  // short lists: concatenated so that every lane probes one entry per half-step
  const uint32_t ds = (was_long && !tail_short) ? 0u : dv;
  uint32_t incl = ds;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += y;
  }
  const uint32_t total = __shfl_sync(kFull, incl, 31);
  const uint32_t base_pos = vs - (incl - ds);  // position of entry f of the concatenation: base_pos + f
  for (uint32_t base = 0; base < total; base += 64) {
    uint64_t e[2];
    bool act[2];
    uint32_t sv[2], q[2], pe[2], pos[2];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      const uint32_t f = base + 32 * i + lane;
      act[i] = f < total;
      // owner: number of lanes whose inclusive end is <= f
      int j = 0;
#pragma unroll
      for (int b = 16; b > 0; b >>= 1) {
        const uint32_t tj = __shfl_sync(kFull, incl, j + b - 1);
        if (tj <= f) j += b;
      }
      j = j > 31 ? 31 : j;
      pos[i] = __shfl_sync(kFull, base_pos, j) + f;
      e[i] = act[i] ? adj[pos[i]] : (uint64_t)none(t);
      sv[i] = __shfl_sync(kFull, pr.s, j);
      q[i] = __shfl_sync(kFull, pr.qe, j);
      pe[i] = __shfl_sync(kFull, pr.pe, j);
    }
    probe<V, T, 2>(t, vis, queue, e, act, pr.x, sv, q, pe, pos, sc);
  }
  // a long list's tail streamed with the short lists is counted twice: an upper bound
  if constexpr (HasProbed<V>::value) vis.probed(probed + total);
}

// This lane's pair among the pairs [ps, ps + cnt) of owner x (kEmpty: of any
// owner).  The pair edge's entry is the one right after its streamed entries.
__device__ __forceinline__ Pair owner_pair(const TravArgs& a, uint32_t x, uint32_t ps, uint32_t cnt) {
  const int lane = (int)lane_id();
  Pair pr;
  pr.x = x;
  pr.qe = 0;
  const uint64_t d = (uint32_t)lane < cnt ? a.pairs[ps + lane] : 0ull;
  bool ok = (uint32_t)lane < cnt && pair_absq2(d) >= a.qmin2;
  pr.vs = pair_start(d);
  pr.dv = pair_len(d);
  pr.s = pr.pe = pr.vs + pr.dv;
  if (ok && (pr.pe >= a.m || pr.pe < pr.vs)) {
    guard_fail(a.sc, kGuardList, x);
    ok = false;
  }
  if (ok && a.keep) {
    pr.vs = a.keep[pr.vs];
    const uint32_t pe = a.keep[pr.pe];
    ok = a.keep[pr.pe + 1] > pe;  // the pair edge is kept
    pr.dv = pe - pr.vs;
    pr.pe = pe;
  }
  if (!ok) pr.dv = 0;
  if (pr.dv) {
    const uint64_t e = a.adj[pr.pe];
    pr.qe = adj_valbits(e);
    if (x == kEmpty) pr.x = adj_col(e);
    if (adj_col(e) != pr.x) {
      guard_fail(a.sc, kGuardVertex, x);
      pr.dv = 0;
    }
  }
  return pr;
}

// Owner x's list: entries [rs, rs + len) of adj; false if the offsets are out of order.
__device__ __forceinline__ bool owner_list(const TravArgs& a, uint32_t x, uint32_t& rs, uint32_t& len) {
  rs = a.row_ptr[x];
  uint32_t re = a.row_ptr[x + 1];
  if (re < rs || re > a.m) return false;
  if (a.keep) {
    rs = a.keep[rs];
    re = a.keep[re];
    if (re < rs || re > a.m) return false;
  }
  len = re - rs;
  return true;
}

// Pair range of owner x, checked against the pair array's bounds.
__device__ __forceinline__ bool pair_range(const TravArgs& a, uint32_t x, uint32_t& ps, uint32_t& np) {
  ps = a.pair_ptr[x];
  const uint32_t pe = a.pair_ptr[x + 1];
  if (pe < ps || pe > a.m) return false;
  np = pe - ps;
  return true;
}

// ------------------------------------------------------------ tasks

// The pairs [ps, ps + np) of owner x by a whole block whose table is loaded:
// warps take pairs `unit` at a time, fewer as the pairs run out, so that they
// reach the closing barrier at about the same time.
template <class V, class T>
__device__ __forceinline__ void block_pairs(const TravArgs& a, V& vis, Queue<V>& queue, const T& t, uint32_t x,
                                            uint32_t ps, uint32_t np, uint32_t* s_misc) {
  const int lane = threadIdx.x & 31;
  const uint32_t nw = blockDim.x >> 5;
  vis.task_begin(x);
  while (true) {
    uint32_t c = 0, cnt = 0;
    if (lane == 0) {
      const uint32_t seen = *(volatile uint32_t*)&s_misc[1];
      const uint32_t rem = seen < np ? np - seen : 0u;
      const uint32_t want = min(a.unit, max(8u, rem / (2 * nw)));
      c = atomicAdd(&s_misc[1], want);
      cnt = c < np ? min(want, np - c) : 0u;
    }
    c = __shfl_sync(kFull, c, 0);
    cnt = __shfl_sync(kFull, cnt, 0);
    if (cnt == 0) break;
    probe_pairs<V, T>(a, vis, queue, t, owner_pair(a, x, ps + c, cnt));
  }
  queue.take_all(t, vis, x);
  vis.task_end(x);
}

// Owner x's list and pairs; false: nothing to do (or a failed self-check).
__device__ __forceinline__ bool owner_task(const TravArgs& a, uint32_t x, uint32_t& rs, uint32_t& len, uint32_t& ps,
                                           uint32_t& np, bool report) {
  if (x >= a.n) {
    if (report) guard_fail(a.sc, kGuardVertex, x);
    return false;
  }
  if (!owner_list(a, x, rs, len) || !pair_range(a, x, ps, np)) {
    if (report) guard_fail(a.sc, kGuardList, x);
    return false;
  }
  return len > 0 && np > 0;
}
// A block task's share of its owner's pairs: part / parts of them.
__device__ __forceinline__ void task_part(uint64_t task, uint32_t& ps, uint32_t& np) {
  const uint32_t part = (uint32_t)(task >> 32) & 0xFFFFu, parts = (uint32_t)(task >> 48) + 1u;
  const uint32_t p0 = (uint32_t)((uint64_t)np * part / parts), p1 = (uint32_t)((uint64_t)np * (part + 1) / parts);
  ps += p0;
  np = p1 - p0;
}
// first vertex of x's graph
__device__ __forceinline__ uint32_t graph_start(const TravArgs& a, uint32_t x) {
  return a.gstart ? a.gstart[a.vgraph[x]] : 0u;
}

// A whole block handles (a part of) owner x with a hash table in `tab`: shared
// memory (hub) or a global slice (giant).
template <class V>
__device__ __forceinline__ void block_task_hash(const TravArgs& a, V& vis, Queue<V>& queue, uint64_t task,
                                                uint32_t* tab, uint32_t cap, uint32_t* s_misc) {
  const int tid = threadIdx.x;
  const uint32_t x = (uint32_t)task;
  uint32_t rs = 0, len = 0, ps = 0, np = 0;
  if (!owner_task(a, x, rs, len, ps, np, tid == 0)) return;
  task_part(task, ps, np);
  const uint32_t slots = slots_for(len);
  if (slots > cap) {
    if (tid == 0) guard_fail(a.sc, kGuardTable, x);
    return;
  }
  const Table t = make_table(tab, cap, slots);
  for (uint32_t i = tid; i < slots; i += blockDim.x) t.key[i] = kEmpty;
  if (tid == 0) s_misc[1] = 0;
  __syncthreads();
  for (uint32_t i = tid; i < len; i += blockDim.x) {
    const uint64_t e = a.adj[rs + i];
    table_insert<V::kPos>(t, adj_col(e), adj_valbits(e), rs + i, a.sc);
  }
  __syncthreads();
  block_pairs<V, Table>(a, vis, queue, t, x, ps, np, s_misc);
  __syncthreads();
}

// The same with a bitmap table.
template <class V>
__device__ __forceinline__ void block_task_bits(const TravArgs& a, V& vis, Queue<V>& queue, uint64_t task, BitTable t,
                                                uint32_t* s_misc) {
  const int tid = threadIdx.x;
  const uint32_t x = (uint32_t)task;
  uint32_t len = 0, ps = 0, np = 0;
  if (!owner_task(a, x, t.rs, len, ps, np, tid == 0)) return;
  task_part(task, ps, np);
  bit_table_graph(t, graph_start(a, x));
  if (x - t.lo > a.hub_bits || len > a.hub_len) {
    if (tid == 0) guard_fail(a.sc, kGuardTable, x);
    return;
  }
  if (tid == 0) s_misc[1] = 0;
  bit_table_load(t, a.adj, len, tid, blockDim.x);
  __syncthreads();
  block_pairs<V, BitTable>(a, vis, queue, t, x, ps, np, s_misc);
  __syncthreads();
  bit_table_clear(t, a.adj, len, tid, blockDim.x);  // the next task's first barrier orders it
}

// One warp handles owner x with its own table.
template <class V>
__device__ __forceinline__ void warp_task_hash(const TravArgs& a, V& vis, Queue<V>& queue, uint32_t x, uint32_t* tab) {
  const int lane = (int)lane_id();
  uint32_t rs = 0, len = 0, ps = 0, np = 0;
  if (!owner_task(a, x, rs, len, ps, np, lane == 0)) return;
  const uint32_t slots = slots_for(len);
  if (slots > a.warp_slots) {
    if (lane == 0) guard_fail(a.sc, kGuardTable, x);
    return;
  }
  const ListTable t = list_table_at(tab, slots, a.adj, rs);
  for (uint32_t i = lane; i < slots; i += 32) t.key[i] = kEmpty;
  __syncwarp();
  for (uint32_t i = lane; i < len; i += 32) list_table_insert(t, i, a.sc);
  __syncwarp();
  vis.task_begin(x);
  for (uint32_t cs = 0; cs < np; cs += 32)
    probe_pairs<V, ListTable>(a, vis, queue, t, owner_pair(a, x, ps + cs, min(32u, np - cs)));
  queue.take_all(t, vis, x);
  vis.task_end(x);
  __syncwarp();
}
template <class V>
__device__ __forceinline__ void warp_task_bits(const TravArgs& a, V& vis, Queue<V>& queue, uint32_t x, BitTable t) {
  const int lane = (int)lane_id();
  uint32_t len = 0, ps = 0, np = 0;
  if (!owner_task(a, x, t.rs, len, ps, np, lane == 0)) return;
  bit_table_graph(t, graph_start(a, x));
  if (x - t.lo > a.warp_bits || len > a.warp_len) {
    if (lane == 0) guard_fail(a.sc, kGuardTable, x);
    return;
  }
  bit_table_load(t, a.adj, len, lane, 32);
  __syncwarp();
  vis.task_begin(x);
  for (uint32_t cs = 0; cs < np; cs += 32)
    probe_pairs<V, BitTable>(a, vis, queue, t, owner_pair(a, x, ps + cs, min(32u, np - cs)));
  queue.take_all(t, vis, x);
  vis.task_end(x);
  __syncwarp();
  bit_table_clear(t, a.adj, len, lane, 32);
  __syncwarp();
}

// Pairs merged lane by lane: the "slot" of a hit is the position of x-w in
// x's list.
struct MergeTable {
  const uint64_t* adj;
};
template <bool kPos>
__device__ __forceinline__ void entry(const MergeTable& t, uint32_t slot, uint32_t& val, uint32_t& pos, uint32_t& w) {
  const uint64_t e = t.adj[slot];
  val = adj_valbits(e);
  pos = slot;
  w = adj_col(e);
}
constexpr uint32_t kMergeGrab = 256;  // pairs a warp takes at a time, at most
template <class V>
__device__ __forceinline__ void merge_tasks(const TravArgs& a, V& vis, Queue<V>& queue) {
  const uint32_t lane = lane_id(), lt = lanemask_lt(), npairs = a.m - a.merge_first;
  const MergeTable t{a.adj};
  const uint64_t* __restrict__ adj = a.adj;
  // few pairs: spread over all warps, 32 each, or a graph of 20,000 edges is 78
  // warps' work (count of three thresholds 137 us a call, 104 spread)
  const uint32_t grab = min(kMergeGrab, npairs / (gridDim.x * (blockDim.x >> 5)) / 32 * 32 + 32);
  while (true) {
    unsigned long long t0 = 0;
    if (lane == 0) t0 = atomicAdd(&a.sc->task[7], (unsigned long long)grab);
    t0 = __shfl_sync(kFull, t0, 0);
    if (t0 >= npairs) break;
    for (uint32_t p0 = (uint32_t)t0; p0 < min((unsigned long long)npairs, t0 + grab); p0 += 32) {
      const Pair pr = owner_pair(a, kEmpty, a.merge_first + p0, min(32u, npairs - p0));
      uint32_t dv = pr.dv, rs = 0, len = 0, i = 0, j = 0;
      if (dv && (pr.x >= a.n || !owner_list(a, pr.x, rs, len))) {
        guard_fail(a.sc, kGuardList, pr.x);
        len = 0;
      }
      uint64_t ea = dv ? adj[pr.vs] : 0ull, eb = len ? adj[rs] : 0ull;
      uint32_t steps = 0;  // at most the entries of both lists, which the queue's appends bound
      while (__any_sync(kFull, i < dv && j < len)) {
        const bool act = i < dv && j < len;
        const uint32_t ca = adj_col(ea), cb = adj_col(eb);
        const bool hit = act && ca == cb;
        if (__any_sync(kFull, hit)) {
          queue.append(hit, V::item(rs + j, pr.qe, adj_valbits(ea), pr.s, pr.pe, pr.vs + i), pr.vs + i, lt);
          queue.take_full(t, vis, pr.x);
        }
        if (act && ca <= cb && ++i < dv) ea = adj[pr.vs + i];
        if (act && cb <= ca && ++j < len) eb = adj[rs + j];
        steps++;
      }
      if constexpr (HasProbed<V>::value) vis.probed(32 * steps);
    }
  }
  queue.take_all(t, vis, kEmpty);
}

// The traversal runs as up to two persistent kernels: the rare block tasks
// with hash tables, and everything else -- the block tasks with bitmaps, then
// the warp tasks -- in one, so that a block that finds no more block tasks goes
// on to warp tasks instead of idling until the last one ends.
enum : int { kHashKernel = 0, kMainKernel = 1 };

__host__ __device__ inline size_t warp_table_bytes(const TravArgs& a) {
  const size_t h = a.n_tasks[kMedHash] ? list_table_bytes(a.warp_slots) : 0;
  const size_t b = a.n_tasks[kMedBits] ? bit_table_bytes(a.warp_bits, a.warp_len) : 0;
  return h > b ? h : b;
}
// Shared memory of a block's tables.
template <class V>
inline size_t traverse_table_bytes(const TravArgs& a, int kernel, int threads) {
  if (kernel == kHashKernel) return a.n_tasks[kHubHash] ? (size_t)table_words<V>(a.hub_slots) * 4 : 0;
  const size_t hub = a.n_tasks[kHubBits] ? bit_table_bytes(a.hub_bits, a.hub_len) : 0;
  return std::max(hub, (size_t)(threads / 32) * warp_table_bytes(a));
}
template <class V>
__host__ __device__ inline size_t visitor_bytes(const typename V::P& p, int threads) {
  return (size_t)((V::smem_bytes(p, threads) + 15) / 16) * 16 + (size_t)(threads / 32) * Queue<V>::kBytes;
}

// The next block task of a class (the same in every thread); n_tasks if none.
__device__ __forceinline__ uint32_t next_block_task(const TravArgs& a, int cls, uint32_t* s_misc) {
  if (threadIdx.x == 0) s_misc[2] = (uint32_t)atomicAdd(&a.sc->task[cls], 1ull);
  __syncthreads();
  const uint32_t task = s_misc[2];
  __syncthreads();
  return task;
}

// Warp tasks [0, n) of a class, the first eighth (the heaviest) one at a time,
// the others `batch` at a time, from two counters.
template <class F>
__device__ __forceinline__ void warp_tasks(const TravArgs& a, int cls, F&& run) {
  const uint32_t n = a.n_tasks[cls], first = n / 8;
  for (int light = 0; light < 2; light++) {
    const uint32_t step = light ? a.batch : 1u, end = light ? n : first;
    unsigned long long* ctr = &a.sc->task[cls == kMedBits ? (light ? 6 : 4) : (light ? 5 : 3)];
    while (true) {
      unsigned long long t0 = 0;
      if (lane_id() == 0) t0 = atomicAdd(ctr, (unsigned long long)step);
      t0 = __shfl_sync(kFull, t0, 0) + (light ? first : 0u);
      if (t0 >= end) break;
      const uint32_t t1 = (uint32_t)min((unsigned long long)end, t0 + step);
      for (uint32_t t = (uint32_t)t0; t < t1; t++) run((uint32_t)a.lists[cls][t]);
    }
  }
}

template <class V, int kKernel>
__device__ void traverse(const TravArgs& a, V& vis, char* queues, char* tables) {
  __shared__ uint32_t s_misc[4];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  Queue<V> queue(queues + (size_t)wid * Queue<V>::kBytes);
  if constexpr (kKernel == kHashKernel) {
    while (blockIdx.x < a.gtab_blocks) {
      const uint32_t task = next_block_task(a, kGiant, s_misc);
      if (task >= a.n_tasks[kGiant]) break;
      block_task_hash(a, vis, queue, a.lists[kGiant][task], a.gtab + (size_t)blockIdx.x * a.gtab_slots * 3,
                      a.gtab_slots, s_misc);
    }
    while (true) {
      const uint32_t task = next_block_task(a, kHubHash, s_misc);
      if (task >= a.n_tasks[kHubHash]) break;
      block_task_hash(a, vis, queue, a.lists[kHubHash][task], (uint32_t*)tables, a.hub_slots, s_misc);
    }
  } else {
    if (a.n_tasks[kHubBits]) {
      const BitTable bt = bit_table_at(tables, a.hub_bits, a.hub_len);
      for (uint32_t i = tid; i < bit_words(a.hub_bits); i += blockDim.x) bt.bits[i] = 0;
      while (true) {
        const uint32_t task = next_block_task(a, kHubBits, s_misc);
        if (task >= a.n_tasks[kHubBits]) break;
        block_task_bits(a, vis, queue, a.lists[kHubBits][task], bt, s_misc);
      }
    }
    char* mine = tables + (size_t)wid * warp_table_bytes(a);
    if (a.n_tasks[kMedBits]) {
      const BitTable bt = bit_table_at(mine, a.warp_bits, a.warp_len);
      for (uint32_t i = lane; i < bit_words(a.warp_bits); i += 32) bt.bits[i] = 0;
      __syncwarp();
      warp_tasks(a, kMedBits, [&](uint32_t x) { warp_task_bits(a, vis, queue, x, bt); });
      __syncwarp();
    }
    if (a.n_tasks[kMedHash])
      warp_tasks(a, kMedHash, [&](uint32_t x) { warp_task_hash(a, vis, queue, x, (uint32_t*)mine); });
    if (a.merge_first < a.m) merge_tasks(a, vis, queue);
  }
  __syncthreads();
  vis.block_end();
  // the last block of the main kernel turns the accumulators into the answer
  if constexpr (kKernel == kMainKernel && HasFinish<V>::value) {
    __threadfence();
    __syncthreads();
    if (tid == 0) s_misc[3] = atomicAdd(&a.sc->done, 1ull) + 1 == gridDim.x ? 1u : 0u;
    __syncthreads();
    if (s_misc[3]) {
      __threadfence();
      vis.finish();
    }
  }
}

namespace {

// Launch bounds per kernel: at most kThreads threads a block; a visitor's
// register cap (V::kRegCap) sets how many blocks must fit on one SM (65536
// registers).
template <class V, int kKernel>
struct Bounds {
  static constexpr int kThreads = kKernel == kHashKernel ? 512 : 256;
  static constexpr int kMinBlocks = 65536 / (kThreads * V::kRegCap) > 0 ? 65536 / (kThreads * V::kRegCap) : 1;
};

template <class V, int kKernel>
__global__ void __launch_bounds__(Bounds<V, kKernel>::kThreads, Bounds<V, kKernel>::kMinBlocks)
    k_traverse(TravArgs a, typename V::P p) {
  extern __shared__ __align__(16) char smem[];
  V vis(p, smem);
  vis.block_init();
  __syncthreads();
  char* queues = smem + ((V::smem_bytes(p, (int)blockDim.x) + 15) / 16) * 16;
  traverse<V, kKernel>(a, vis, queues, smem + visitor_bytes<V>(p, (int)blockDim.x));
}

// Warps of a kernel that fit on an SM: by registers (65536) and shared memory
// (227 KB, 1 KB of it per block taken by the system).
template <class V, int kKernel>
int resident_warps(const TravArgs& a, const typename V::P& p, int threads) {
  const size_t smem = visitor_bytes<V>(p, threads) + traverse_table_bytes<V>(a, kKernel, threads) + 1024;
  const int blocks = (int)std::min<size_t>((227 * 1024 + 1024) / smem, 65536 / (size_t)(threads * V::kRegCap));
  return blocks * threads / 32;
}

template <class V, int kKernel>
ubt_status launch_kernel(const ubt_graph* g, const TravArgs& a, const typename V::P& p, cudaStream_t s) {
  const Tuning& T = tuning();
  int threads = (int)(kKernel == kHashKernel ? T.block_threads : T.warp_threads);
  threads = (int)std::min<int64_t>(Bounds<V, kKernel>::kThreads, std::max<int64_t>(MinThreads<V>::value, threads / 32 * 32));
  // Larger blocks share the block tasks' table among more warps; smaller ones
  // lose less at its barriers.  Twice the threads where the table's size would
  // otherwise leave fewer than 7/8 of the warps they make room for (R-MAT scale
  // 22, tables of 26 KB: 19.8 -> 17.0 ms with 256 threads; Chung-Lu of 1e6
  // vertices, tables of 4 KB: 1.15 ms with 128, 1.21 with 256).
  if (kKernel == kMainKernel && 2 * threads <= Bounds<V, kKernel>::kThreads &&
      8 * resident_warps<V, kKernel>(a, p, threads) < 7 * resident_warps<V, kKernel>(a, p, 2 * threads))
    threads *= 2;
  // Smaller blocks where that many warps' tables do not fit at all (a large
  // hub_threshold with a visitor that prefers large blocks).
  size_t smem = 0;
  int per_sm = 0;
  for (;; threads -= 32) {
    smem = visitor_bytes<V>(p, threads) + traverse_table_bytes<V>(a, kKernel, threads);
    const cudaError_t e = resident_blocks((const void*)k_traverse<V, kKernel>, g->device, threads, smem, &per_sm);
    if (e == cudaSuccess && per_sm > 0) break;
    if (threads > 64 && (e == cudaSuccess || e == cudaErrorInvalidValue)) continue;
    UBT_CUDA(e);
    return UBT_ERR_INVALID_ARG;
  }
  per_sm = (int)std::min<int64_t>(per_sm, std::max<int64_t>(1, T.blocks_per_sm));
  int64_t blocks = (int64_t)g->sm_count * per_sm;
  if (kKernel == kMainKernel) {  // no more blocks than there is work for: each sets up its visitor's tables
    const int64_t warps = a.n_tasks[kMedHash] + a.n_tasks[kMedBits] + (a.m - a.merge_first + 31) / 32;
    blocks = std::min(blocks, std::max<int64_t>(1, a.n_tasks[kHubBits] + (warps + threads / 32 - 1) / (threads / 32)));
  }
  k_traverse<V, kKernel><<<(int)blocks, threads, smem, s>>>(a, p);
  UBT_CUDA(cudaGetLastError());
  return UBT_OK;
}

// One traversal: the task counters in a.sc are cleared, then the kernels that
// have tasks run one after the other on `s` (the main one always where the
// visitor's answer is written by its last block).
template <class V>
ubt_status launch_traversal(const ubt_graph* g, const TravArgs& a, const typename V::P& p, cudaStream_t s) {
  UBT_RANGE("traversal launch");
  UBT_CUDA(cudaMemsetAsync(a.sc->task, 0, HasFinish<V>::value ? kScratchCounts : kScratchQuery, s));
  ubt_status st = UBT_OK;
  if (a.n_tasks[kGiant] + a.n_tasks[kHubHash]) st = launch_kernel<V, kHashKernel>(g, a, p, s);
  if (st == UBT_OK && (HasFinish<V>::value || a.n_tasks[kHubBits] + a.n_tasks[kMedHash] + a.n_tasks[kMedBits] +
                                                  (a.m - a.merge_first)))
    st = launch_kernel<V, kMainKernel>(g, a, p, s);
  return st;
}

}  // namespace

}  // namespace ubt
