// ubt_worlds.cu -- Monte-Carlo sign worlds and batched per-graph queries.
//
// Sign worlds (not in the paper): world 64 w + j draws every edge sign with
// P(+) = k / 65536.  A triangle is balanced in a world iff it has an odd
// number of positive edges (Def. 3, Sec. 3), i.e. iff the XOR of its three
// sign bits is 1.  64 worlds share one 64-bit word per edge ("bit-sliced").
//
// Draws: Philox4x64-10 (Salmon, Moraes, Dror, Shaw, "Parallel random numbers:
// as easy as 1, 2, 3", SC'11) with key (seed, 0) and counter (K, w, c, 0),
// c = 0..3, gives 16 words r_0..r_15; bit j of r_b is bit b of world j's
// 16-bit uniform u_j, and the edge is positive iff u_j < k.  The comparison is
// evaluated for all 64 worlds at once on the bit planes (most significant
// plane first).
//
// Per-world counts are kept per lane as bit-sliced binary counters (plane t
// holds bit t of 64 counters), incremented by the XOR word of each triangle,
// and flushed to integer counts before they can overflow.
#include <algorithm>
#include <vector>

#include "ubt_traverse.cuh"

namespace ubt {

ubt_status make_trav_args(const ubt_graph* g, int64_t L, cudaStream_t s, TravArgs* out);

namespace {

// ------------------------------------------------------------ Philox4x64-10

struct U64x4 {
  unsigned long long x[4];
};

// Philox4x64-10 of counter (key, w, call, 0) with key (seed, 0), given the
// product of its first round that the four calls of an edge share.
struct FirstRound {
  unsigned long long lo, hi;  // M0 * key
};
constexpr unsigned long long kPhiloxM0 = 0xD2E7470EE14C6C93ull, kPhiloxM1 = 0xCA5A826395121157ull;
__device__ __forceinline__ FirstRound philox_first(uint32_t key) {
  return FirstRound{kPhiloxM0 * key, __umul64hi(kPhiloxM0, key)};
}
__device__ __forceinline__ U64x4 philox_call(const FirstRound& f, uint32_t w, uint32_t call, unsigned long long seed) {
  const unsigned long long W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
  unsigned long long k0 = seed, k1 = 0;
  U64x4 c;  // after the first round
  c.x[0] = __umul64hi(kPhiloxM1, (unsigned long long)call) ^ (unsigned long long)w ^ k0;
  c.x[1] = kPhiloxM1 * call;
  c.x[2] = f.hi ^ k1;
  c.x[3] = f.lo;
#pragma unroll
  for (int r = 1; r < 10; r++) {
    k0 += W0;
    k1 += W1;
    const unsigned long long lo0 = kPhiloxM0 * c.x[0], hi0 = __umul64hi(kPhiloxM0, c.x[0]);
    const unsigned long long lo1 = kPhiloxM1 * c.x[2], hi1 = __umul64hi(kPhiloxM1, c.x[2]);
    U64x4 n;
    n.x[0] = hi1 ^ c.x[1] ^ k0;
    n.x[1] = lo1;
    n.x[2] = hi0 ^ c.x[3] ^ k1;
    n.x[3] = lo0;
    c = n;
  }
  return c;
}

// u < k on the bit planes 4 call .. 4 call + 3, most significant first: lt are
// the worlds decided positive, eq the undecided ones
__device__ __forceinline__ void sign_planes(const U64x4& o, uint32_t call, uint32_t k, unsigned long long& lt,
                                            unsigned long long& eq) {
#pragma unroll
  for (int i = 3; i >= 0; i--) {
    const unsigned long long r = o.x[i];
    const unsigned long long bit = 0ull - (unsigned long long)((k >> (4 * call + i)) & 1u);  // all ones if set
    lt |= eq & ~r & bit;
    eq &= ~(r ^ bit);
  }
}

// X[pos * wp + i] = sign word (w0 + i) of the edge at CSR position pos, i < valid
// (wp a power of two): bit j = 1 iff positive in world 64 (w0 + i) + j.
//
// A world is decided at the first plane where u and k differ, so the lower
// planes' calls are needed for few words: after the first two calls (planes
// 15..8) 22 % of the words have an undecided world, after three 2 %.  Every
// word gets the first two calls, independent of each other; the undecided ones
// are queued per warp and finished 32 at a time, on full warps (2.4 calls a
// word; calling until a warp's 32 words are all decided took 3.4).  Bound by
// the 64-bit products' multiply instructions.
constexpr int kSignThreads = 256;
constexpr int kSignQueue = 64;
struct SignQueue {
  unsigned long long at[kSignQueue], lt[kSignQueue], eq[kSignQueue];
  uint32_t key[kSignQueue], w[kSignQueue], k[kSignQueue];
};
__global__ void __launch_bounds__(kSignThreads)
k_sign_table(int64_t m, const uint64_t* __restrict__ adj, const uint32_t* __restrict__ ekey, unsigned long long seed,
             uint32_t w0, uint32_t wp, uint32_t valid, unsigned long long* __restrict__ X) {
  __shared__ SignQueue queues[kSignThreads / 32];
  SignQueue& q = queues[threadIdx.x >> 5];
  const uint32_t lane = lane_id();
  uint32_t n = 0;  // queued words (warp-uniform, fewer than 32 between steps)
  auto finish = [&](uint32_t cnt) {  // the last cnt queued words
    __syncwarp();
    n -= cnt;
    if (lane < cnt) {
      const uint32_t i = n + lane, k = q.k[i];
      unsigned long long lt = q.lt[i], eq = q.eq[i];
      const FirstRound f = philox_first(q.key[i]);
#pragma unroll 1
      for (int call = 1; call >= 0 && eq; call--) sign_planes(philox_call(f, q.w[i], call, seed), call, k, lt, eq);
      X[q.at[i]] = lt;
    }
    __syncwarp();
  };
  const int lg = 31 - __clz((int)wp);
  const int64_t total = m << lg;
  for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; base < total;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + lane, pos = i >> lg;
    const uint32_t wi = (uint32_t)i & (wp - 1);
    const bool on = i < total && wi < valid;
    const uint32_t k = on ? (uint32_t)(32768 - adj_q(adj[pos])) : 0u, key = on ? ekey[pos] : 0u, w = w0 + wi;
    unsigned long long lt = k >= 65536u ? ~0ull : 0ull, eq = k == 0u || k >= 65536u ? 0ull : ~0ull;
    if (__any_sync(kFull, eq != 0ull)) {
      const FirstRound f = philox_first(key);
      const U64x4 o3 = philox_call(f, w, 3, seed), o2 = philox_call(f, w, 2, seed);
      sign_planes(o3, 3, k, lt, eq);
      sign_planes(o2, 2, k, lt, eq);
    }
    const bool more = on && eq != 0ull;
    if (on && !more) X[i] = lt;
    const unsigned mask = __ballot_sync(kFull, more);
    if (more) {
      const uint32_t at = n + __popc(mask & lanemask_lt());
      q.at[at] = (unsigned long long)i;
      q.lt[at] = lt;
      q.eq[at] = eq;
      q.key[at] = key;
      q.w[at] = w;
      q.k[at] = k;
    }
    n += __popc(mask);
    if (n >= 32) finish(32);
  }
  if (n) finish(n);
}

// ------------------------------------------------------------ bit-sliced counters

template <int K>
struct Planes {
  unsigned long long c[K];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int t = 0; t < K; t++) c[t] = 0;
  }
  // one word of weight 2^from
  __device__ __forceinline__ void inc(unsigned long long b, int from) {
#pragma unroll
    for (int t = 0; t < K; t++) {
      if (t < from) continue;
      const unsigned long long carry = c[t] & b;
      c[t] ^= b;
      b = carry;
    }
  }
  // All lanes' counters summed (32 lanes: 5 more planes), bit-sliced all the way:
  // every lane ends with the totals of all 64 counters in t[0 .. K + 4].
  __device__ __forceinline__ void warp_total(unsigned long long (&t)[K + 5]) const {
#pragma unroll
    for (int i = 0; i < K + 5; i++) t[i] = i < K ? c[i] : 0ull;
#pragma unroll
    for (int r = 0; r < 5; r++) {
      unsigned long long carry = 0;
#pragma unroll
      for (int i = 0; i < K + r; i++) {
        const unsigned long long o = __shfl_xor_sync(kFull, t[i], 1 << r), x = t[i];
        t[i] = x ^ o ^ carry;
        carry = (x & o) | (x & carry) | (o & carry);
      }
      t[K + r] = carry;
    }
  }
  // eight words at once (K > 3): a carry-save tree, three full adders' worth of
  // logic per word instead of a carry chain through every plane, whose carry of
  // weight 8 goes up the planes once
  __device__ __forceinline__ void add8(const unsigned long long (&w)[8]) {
    unsigned long long a, b, f0, f1, e;
    csa(a, c[0], w[0], w[1]);
    csa(b, c[0], w[2], w[3]);
    csa(f0, c[1], a, b);
    csa(a, c[0], w[4], w[5]);
    csa(b, c[0], w[6], w[7]);
    csa(f1, c[1], a, b);
    csa(e, c[2], f0, f1);
#pragma unroll
    for (int t = 3; t < K; t++) {
      const unsigned long long carry = c[t] & e;
      c[t] ^= e;
      e = carry;
    }
  }
  // sum + x + y: the sum bit stays, the carry goes out
  __device__ __forceinline__ static void csa(unsigned long long& carry, unsigned long long& sum, unsigned long long x,
                                             unsigned long long y) {
    const unsigned long long s = sum;
    carry = (s & x) | (s & y) | (x & y);
    sum = s ^ x ^ y;
  }
  // per-lane count of world j
  __device__ __forceinline__ uint32_t count(int j) const {
    uint32_t v = 0;
#pragma unroll
    for (int t = 0; t < K; t++) v |= (uint32_t)((c[t] >> j) & 1ull) << t;
    return v;
  }
};

// ------------------------------------------------------------ sign-world visitor

struct WorldsP {
  const unsigned long long* X;  // sign table of this pass: m x wp words
  uint32_t wp;                  // words per pass (1..64, power of two)
  uint32_t valid;               // of them wanted
  unsigned long long* out;      // counts of this pass's worlds: valid * 64
};

// SLOTS = words per lane: 1 when wp <= 32 (lanes grouped by word), 2 when wp = 64
template <int SLOTS>
struct Worlds {
  using P = WorldsP;
  using Item = uint4;  // table slot, positions of the pair edge and the streamed edge
  static constexpr bool kMore = false;
  static constexpr int kU = 2;
  static constexpr bool kPos = true;
  // the main kernel's form of Worlds<2> spills at this cap (964 bytes of stores,
  // 1,784 of loads a thread by the compiler's account): 24 planes and 16 words of
  // 64 bits are live beside the flush
  static constexpr int kRegCap = 128;
  // a block's counters are 32 KB that L1, where the owner's sign rows stay, loses
  // (R-MAT scale 20, 4,096 worlds: 94.7 ms in blocks of 128 threads, 76.7 of 256)
  static constexpr int kMinThreads = 256;
  static constexpr int K = SLOTS == 1 ? 14 : 12;      // planes per slot
  static constexpr uint32_t kLimit = (1u << K) - 1u;  // increments before a flush
  // counters + one list of 32 triangles per warp
  static __host__ __device__ int smem_bytes(const P&, int threads) { return 64 * 64 * 8 + (threads / 32) * 96 * 4; }
  P p;
  unsigned long long* cnt;  // shared: wp * 64 counters
  uint32_t* q;              // shared: this warp's triangles, 3 x 32 positions
  uint32_t since = 0;
  Planes<K> pl[SLOTS];
  __device__ Worlds(const P& p_, char* smem) : p(p_) {
    cnt = (unsigned long long*)smem;
    q = (uint32_t*)(smem + 64 * 64 * 8) + (threadIdx.x >> 5) * 96;
#pragma unroll
    for (int s = 0; s < SLOTS; s++) pl[s].clear();
  }
  __device__ void block_init() {
    for (int i = threadIdx.x; i < (int)p.wp * 64; i += blockDim.x) cnt[i] = 0;
  }
  __device__ __forceinline__ uint32_t word_of(int s) const {
    const int lane = (int)lane_id();
    return SLOTS == 2 ? (uint32_t)(2 * lane + s) : (uint32_t)lane % p.wp;
  }
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int s = 0; s < SLOTS; s++) {
      const uint32_t w = word_of(s);
#pragma unroll 1
      for (int j = 0; j < 64; j++) {
        const uint32_t v = pl[s].count(j);
        if (v) atomicAdd(&cnt[w * 64 + j], (unsigned long long)v);
      }
      pl[s].clear();
    }
    since = 0;
  }
  __device__ __forceinline__ static uint4 item(uint32_t slot, uint32_t, uint32_t, uint32_t, uint32_t puv, uint32_t pvw) {
    return make_uint4(slot, puv, pvw, 0u);
  }
  // The queued triangles' sign rows, 8 words a lane at a time (their loads all
  // issued before the adder tree); the streamed edge's row is not kept in L1,
  // so that the owner's and the pair's rows, which the next triangles reuse, stay.
  __device__ __forceinline__ void take(bool on, uint32_t qn, uint4 it, uint32_t, uint32_t, uint32_t, uint32_t puw,
                                       uint32_t) {
    const int lane = (int)lane_id();
    __syncwarp();
    if (on) {
      q[lane] = puw;
      q[32 + lane] = it.y;
      q[64 + lane] = it.z;
    }
    __syncwarp();
    const uint32_t wp = p.wp;
    if (SLOTS == 2) {
      // a row is 64 words = 32 16-byte pairs: lane l holds words 2l and 2l + 1
      const ulonglong2* __restrict__ X2 = reinterpret_cast<const ulonglong2*>(p.X) + lane;
#pragma unroll 1
      for (uint32_t t0 = 0; t0 < qn; t0 += 8) {
        unsigned long long w0[8], w1[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const uint32_t t = min(t0 + i, qn - 1);  // past the end: loaded again and not counted
          const ulonglong2 a = X2[(size_t)q[t] * 32], b = X2[(size_t)q[32 + t] * 32],
                           c = load_once(X2 + (size_t)q[64 + t] * 32);
          w0[i] = t0 + i < qn ? a.x ^ b.x ^ c.x : 0ull;
          w1[i] = t0 + i < qn ? a.y ^ b.y ^ c.y : 0ull;
        }
        if (since + 8 > kLimit) flush();
        pl[0].add8(w0);
        pl[SLOTS - 1].add8(w1);
        since += 8;
      }
    } else {
      const uint32_t per = 32 / wp;  // triangles per word of a lane
      const uint32_t grp = (uint32_t)lane / wp, w = (uint32_t)lane % wp;
      const unsigned long long* __restrict__ X = p.X + w;
#pragma unroll 1
      for (uint32_t t0 = grp; t0 < qn + grp; t0 += 8 * per) {  // as often in every lane
        unsigned long long x[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const uint32_t at = t0 + i * per, t = min(at, qn - 1);
          const unsigned long long v =
              X[(size_t)q[t] * wp] ^ X[(size_t)q[32 + t] * wp] ^ load_once(X + (size_t)q[64 + t] * wp);
          x[i] = at < qn ? v : 0ull;
        }
        if (since + 8 > kLimit) flush();
        pl[0].add8(x);
        since += 8;
      }
    }
  }
  __device__ __forceinline__ static unsigned long long load_once(const unsigned long long* a) {
    unsigned long long v;
    asm("ld.global.nc.L1::no_allocate.u64 %0, [%1];" : "=l"(v) : "l"(a));
    return v;
  }
  __device__ __forceinline__ static ulonglong2 load_once(const ulonglong2* a) {
    ulonglong2 v;
    asm("ld.global.nc.L1::no_allocate.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(a));
    return v;
  }
  __device__ void task_begin(uint32_t) {}
  __device__ void task_end(uint32_t) {}
  __device__ void block_end() {
    flush();
    __syncthreads();
    for (int i = threadIdx.x; i < (int)p.valid * 64; i += blockDim.x)
      if (cnt[i]) atomicAdd(&p.out[i], cnt[i]);
  }
};

__global__ void k_world_total(const unsigned long long* __restrict__ cnt, int64_t W, int64_t* total) {
  __shared__ unsigned long long s[1024];
  unsigned long long acc = 0;
  for (int64_t i = threadIdx.x; i < W; i += blockDim.x) acc += cnt[i];
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int d = blockDim.x / 2; d > 0; d >>= 1) {
    if ((int)threadIdx.x < d) s[threadIdx.x] += s[threadIdx.x + d];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = (int64_t)s[0];
}

// ------------------------------------------------------------ batch visitor

constexpr int kBatchTau = 8;

struct BatchP {
  int nt;
  int64_t B[kBatchTau];
  int64_t U[kBatchTau];
  const uint32_t* vgraph;
  const unsigned long long* X;  // one sign word per CSR position, or null
  unsigned long long* counts;   // per graph: 2 * nt
  unsigned long long* acc;      // per graph: T, sum_lo, sum_hi (or null)
  unsigned long long* worlds;   // per graph: 64 (or null)
};

// Per-graph answers; all tasks of a warp between two graph changes share
// their registers, which are flushed when the graph changes.
struct Batch {
  using P = BatchP;
  static constexpr bool kPos = true;
  using Item = uint4;  // table slot, product of two values, positions of the pair edge and the streamed edge
  static constexpr bool kMore = false;
  static constexpr int kU = 2;
  // 24 warps an SM instead of 16: the triangles' sign words and list entries are
  // waited on (batch of 1,000 graphs: 9.9 ms with up to 128 registers, 8.7 with
  // 85, 9.0 with 64; at 85 the compiler takes 80 and spills 568 bytes of stores,
  // 836 of loads a thread)
  static constexpr int kRegCap = 85;
  static __host__ __device__ int smem_bytes(const P&, int) { return 0; }
  static constexpr int K = 8;                        // planes: fewer than 256 words between two flushes
  static constexpr uint32_t kSumLimit = 1u << 17;    // |P| <= 2^45: so many fit a signed 64-bit sum
  P p;
  uint32_t g = kEmpty;
  uint32_t bal[kBatchTau], unbal[kBatchTau];
  uint32_t tri = 0;
  long long sum = 0;
  Planes<K> pl;
  unsigned long long ones = 0, twos = 0, fours = 0;  // words of weight 1, 2, 4 waiting for their second
  uint32_t since = 0, sums = 0;                      // triangles taken since the last flush (warp-uniform)
  __device__ Batch(const P& p_, char*) : p(p_) {
#pragma unroll
    for (int i = 0; i < kBatchTau; i++) bal[i] = unbal[i] = 0;
    pl.clear();
  }
  __device__ void block_init() {}
  // the world counters to the graph's counts: words still waiting go in first
  __device__ __forceinline__ void flush_worlds() {
    if (!since) return;
    pl.inc(since & 1u ? ones : 0ull, 0);
    pl.inc(since & 2u ? twos : 0ull, 1);
    pl.inc(since & 4u ? fours : 0ull, 2);
    unsigned long long t[K + 5];
    pl.warp_total(t);
    const int lane = (int)lane_id();
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int j = lane + 32 * h;
      uint32_t v = 0;
#pragma unroll
      for (int i = 0; i < K + 5; i++) v |= (uint32_t)((t[i] >> j) & 1ull) << i;
      if (v) atomicAdd(&p.worlds[(size_t)g * 64 + j], (unsigned long long)v);
    }
    pl.clear();
    since = 0;
  }
  __device__ __forceinline__ void flush_sums() {
    const uint32_t t = __reduce_add_sync(kFull, tri);
    unsigned long long lo = (unsigned long long)sum, hi = sum < 0 ? ~0ull : 0ull;  // 128-bit warp sum
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long l = __shfl_xor_sync(kFull, lo, d);
      const unsigned long long h = __shfl_xor_sync(kFull, hi, d);
      const unsigned long long o = lo;
      lo += l;
      hi += h + (lo < o ? 1ull : 0ull);
    }
    if (lane_id() == 0 && t) {
      unsigned long long* a = p.acc + (size_t)g * 3;
      atomicAdd(&a[0], (unsigned long long)t);
      const unsigned long long o = atomicAdd(&a[1], lo);
      atomicAdd(&a[2], hi + ((o + lo < o) ? 1ull : 0ull));
    }
    tri = 0;
    sum = 0;
    sums = 0;
  }
  __device__ void flush() {
    if (g == kEmpty) return;
    const int lane = (int)lane_id();
#pragma unroll
    for (int i = 0; i < kBatchTau; i++) {
      if (i < p.nt) {
        const uint32_t b = __reduce_add_sync(kFull, bal[i]);
        const uint32_t u = __reduce_add_sync(kFull, unbal[i]);
        if (lane == 0) {
          if (b) atomicAdd(&p.counts[(size_t)g * 2 * p.nt + i], (unsigned long long)b);
          if (u) atomicAdd(&p.counts[(size_t)g * 2 * p.nt + p.nt + i], (unsigned long long)u);
        }
        bal[i] = unbal[i] = 0;
      }
    }
    if (p.acc) flush_sums();
    if (p.worlds) flush_worlds();
  }
  __device__ __forceinline__ static uint4 item(uint32_t slot, uint32_t quv, uint32_t qvw, uint32_t, uint32_t puv,
                                               uint32_t pvw) {
    return make_uint4(slot, (uint32_t)((int32_t)quv * (int32_t)qvw), puv, pvw);
  }
  // One triangle a lane.  The world words go through carry-save adders a pair
  // at a time (`since` says which weights wait for their second word), so a
  // word costs two adders on average instead of a carry chain up the planes.
  __device__ __forceinline__ void take(bool on, uint32_t, uint4 it, uint32_t, uint32_t, uint32_t quw, uint32_t puw,
                                       uint32_t) {
    unsigned long long x = 0ull;
    if (on) {
      if (p.X) x = p.X[it.z] ^ p.X[puw] ^ p.X[it.w];
      const int64_t P = (int64_t)(int32_t)it.y * (int64_t)(int32_t)quw;
#pragma unroll
      for (int i = 0; i < kBatchTau; i++) {
        if (i < p.nt) {
          bal[i] += (P <= p.B[i]);
          unbal[i] += (P > p.U[i]);
        }
      }
      tri++;
      sum += P;
    }
    if (++sums == kSumLimit && p.acc) flush_sums();
    if (p.X) {
      if (!(since & 1u)) {
        ones = x;
      } else {
        Planes<K>::csa(x, pl.c[0], ones, x);
        if (!(since & 2u)) {
          twos = x;
        } else {
          Planes<K>::csa(x, pl.c[1], twos, x);
          if (!(since & 4u)) {
            fours = x;
          } else {
            Planes<K>::csa(x, pl.c[2], fours, x);
            pl.inc(x, 3);
          }
        }
      }
      if (++since == (1u << K) - 8u) flush_worlds();  // a multiple of 8: nothing waits
    }
  }
  __device__ void task_begin(uint32_t u) {
    const uint32_t gu = p.vgraph[u];
    if (gu != g) {
      flush();
      g = gu;
    }
  }
  __device__ void task_end(uint32_t) {}
  __device__ void block_end() { flush(); }
};

__global__ void k_batch_finish(int64_t ng, int nt, const unsigned long long* __restrict__ acc, double* expect) {
  for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < ng; gi += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long T = acc[3 * gi], lo = acc[3 * gi + 1], hi = acc[3 * gi + 2];
    const bool small = (hi == 0ull && !(lo >> 63)) || (hi == ~0ull && (lo >> 63));
    const double sum = (small ? (double)(long long)lo : (double)(long long)hi * 18446744073709551616.0 + (double)lo) *
                       0x1p-45;
    expect[2 * gi] = ((double)T - sum) * 0.5;
    expect[2 * gi + 1] = ((double)T + sum) * 0.5;
  }
}

ubt_status launch_sign_table(const ubt_graph* g, uint64_t seed, int64_t w0, int64_t wp, int64_t valid,
                             unsigned long long* X, cudaStream_t s) {
  if (g->m == 0) return UBT_OK;
  const int grid = (int)std::min<int64_t>((g->m * wp + kSignThreads - 1) / kSignThreads, (int64_t)g->sm_count * 32);
  k_sign_table<<<grid, kSignThreads, 0, s>>>(g->m, g->adj, g->ekey, seed, (uint32_t)w0, (uint32_t)wp, (uint32_t)valid, X);
  UBT_CUDA(cudaGetLastError());
  return UBT_OK;
}

template <class V>
ubt_status launch_w(const ubt_graph* g, const typename V::P& p, cudaStream_t s) {
  TravArgs a;
  const ubt_status st = make_trav_args(g, 0, s, &a);
  return st != UBT_OK ? st : launch_traversal<V>(g, a, p, s);
}

// Words of a pass over `left` words: a power of two (lanes are grouped by
// word), at most `most`.  More words a pass list the triangles fewer times and
// read longer rows (R-MAT scale 20, 64 words: one pass of 64 85 ms, eight of 8
// 143 ms).  The last pass may have words to spare rather than be cut into
// several.
int64_t pass_words(int64_t left, int64_t most) {
  int64_t wp = most;
  while (wp > 1 && 4 * left < 3 * wp) wp >>= 1;
  return wp;
}

// bytes of a workspace whose sign table has `words` words an edge
size_t worlds_workspace_bytes(const ubt_graph* g, int64_t words) {
  return (size_t)std::max<int64_t>(g->m, 1) * (size_t)words * 8 + 256;
}

// The most words a call needs room for: every workspace from this size on
// serves (the passes are the largest that fit it, with the same counts).
constexpr int64_t kLeastWords = 8;
int64_t least_words(int64_t words) {
  int64_t wp = std::min(kLeastWords, tuning().world_words_per_pass);
  while (wp > words) wp >>= 1;
  return wp;
}

// What ubt_sample_worlds_workspace_size asks for: the tuning's words, unless
// the table would take more than an eighth of the HBM or, above 1 GiB (where a
// call lasts long enough for the question to cost nothing), than 7/8 of the
// memory that is free now: a call beside other tenants of the GPU runs in
// smaller passes instead of failing to allocate.
constexpr int64_t kSignTableBytes = 36ll << 30, kSmallTableBytes = 1ll << 30;
int64_t wanted_words(const ubt_graph* g, int64_t words) {
  int64_t wp = pass_words(words, tuning().world_words_per_pass);
  const int64_t word_bytes = g->m * 8;
  if (wp <= kLeastWords || wp * word_bytes <= kSmallTableBytes) return wp;
  size_t free_bytes = 0, all = 0;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // the question is harmless inside a capture
  cudaThreadExchangeStreamCaptureMode(&mode);
  if (cudaMemGetInfo(&free_bytes, &all) != cudaSuccess) free_bytes = (size_t)kSignTableBytes;
  cudaThreadExchangeStreamCaptureMode(&mode);
  const int64_t room = std::min<int64_t>(kSignTableBytes, (int64_t)(free_bytes / 8 * 7));
  while (wp > kLeastWords && wp * word_bytes > room) wp >>= 1;
  return wp;
}

}  // namespace
}  // namespace ubt

using namespace ubt;

extern "C" ubt_status ubt_sample_worlds_workspace_size(const ubt_graph* g, int64_t W, size_t* h_bytes) {
  if (!g || !h_bytes || W < 64 || W % 64) return UBT_ERR_INVALID_ARG;
  *h_bytes = worlds_workspace_bytes(g, wanted_words(g, W / 64));
  return UBT_OK;
}

extern "C" ubt_status ubt_sample_worlds(ubt_graph* g, uint64_t seed, int64_t W, int64_t* d_bal_per_world,
                                        int64_t* d_total, void* d_workspace, size_t ws_bytes, void* stream) {
  UBT_RANGE("ubt_sample_worlds");
  if (!g || !d_bal_per_world || W < 64 || W % 64 || W / 64 > 0xFFFFFFFFll) return UBT_ERR_INVALID_ARG;
  if (g->kind != UBT_GRAPH_FIXED) return UBT_ERR_UNSUPPORTED;
  if (!d_workspace || ((uintptr_t)d_workspace & 255)) return UBT_ERR_INVALID_ARG;
  const int64_t words = W / 64;
  int64_t most = least_words(words);
  if (ws_bytes < worlds_workspace_bytes(g, most)) return UBT_ERR_WORKSPACE_TOO_SMALL;
  while (2 * most <= tuning().world_words_per_pass && ws_bytes >= worlds_workspace_bytes(g, 2 * most)) most *= 2;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* X = (unsigned long long*)d_workspace;
  UBT_CUDA(cudaMemsetAsync(d_bal_per_world, 0, sizeof(int64_t) * W, s));
  for (int64_t w0 = 0; w0 < words;) {
    const int64_t wp = pass_words(words - w0, most), valid = std::min(wp, words - w0);
    const ubt_status sst = launch_sign_table(g, seed, w0, wp, valid, X, s);
    if (sst != UBT_OK) return sst;
    WorldsP p{X, (uint32_t)wp, (uint32_t)valid, (unsigned long long*)(d_bal_per_world + w0 * 64)};
    const ubt_status st = wp == 64 ? launch_w<Worlds<2>>(g, p, s) : launch_w<Worlds<1>>(g, p, s);
    if (st != UBT_OK) return st;
    w0 += valid;
  }
  if (d_total) {
    k_world_total<<<1, 1024, 0, s>>>((const unsigned long long*)d_bal_per_world, W, d_total);
    UBT_CUDA(cudaGetLastError());
  }
  return UBT_OK;
}

extern "C" ubt_status ubt_batch_query(ubt_graph* g, const double* h_tau, int32_t n_tau, uint64_t seed,
                                      int64_t* d_counts, double* d_expect, int64_t* d_worlds, void* stream) {
  UBT_RANGE("ubt_batch_query");
  if (!g || !h_tau || !d_counts || n_tau < 1 || n_tau > kBatchTau) return UBT_ERR_INVALID_ARG;
  if (!g->vgraph) return UBT_ERR_INVALID_ARG;
  if (g->kind != UBT_GRAPH_FIXED) return UBT_ERR_UNSUPPORTED;
  BatchP p;
  p.nt = n_tau;
  for (int i = 0; i < n_tau; i++) {
    Level lv;
    if (!tau_level(h_tau[i], &lv)) return UBT_ERR_TAU_OOB;
    p.B[i] = lv.B;
    p.U[i] = lv.U;
  }
  for (int i = n_tau; i < kBatchTau; i++) p.B[i] = p.U[i] = 0;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t ng = g->n_graphs;
  p.vgraph = g->vgraph;
  p.counts = (unsigned long long*)d_counts;
  p.acc = d_expect ? g->bacc : nullptr;
  p.worlds = (unsigned long long*)d_worlds;
  p.X = nullptr;
  UBT_CUDA(cudaMemsetAsync(d_counts, 0, sizeof(int64_t) * ng * 2 * n_tau, s));
  if (d_expect) UBT_CUDA(cudaMemsetAsync(g->bacc, 0, sizeof(unsigned long long) * 3 * ng, s));
  if (d_worlds) {
    UBT_CUDA(cudaMemsetAsync(d_worlds, 0, sizeof(int64_t) * ng * 64, s));
    // one sign word per CSR position, kept in the backward accumulators
    const ubt_status sst = launch_sign_table(g, seed, 0, 1, 1, g->gacc, s);
    if (sst != UBT_OK) return sst;
    p.X = g->gacc;
  }
  ubt_status st = launch_w<Batch>(g, p, s);
  if (st != UBT_OK) return st;
  if (d_expect) {
    const int grid = (int)std::min<int64_t>((ng + 255) / 256, (int64_t)g->sm_count * 8);
    k_batch_finish<<<std::max(grid, 1), 256, 0, s>>>(ng, n_tau, g->bacc, d_expect);
    UBT_CUDA(cudaGetLastError());
  }
  return UBT_OK;
}
