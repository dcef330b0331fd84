// ubt_scan.cu -- exclusive prefix sum of uint32 counts (CSR offsets, list
// offsets).  Three passes over tiles of 4096 values: tile totals, a scan of
// the totals by one block, then a rescan of every tile with its offset.
#include "ubt_internal.cuh"

namespace ubt {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kTile = kScanThreads * kScanItems;

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* excl) {
  __shared__ uint32_t wsum[kScanThreads / 32];
  __shared__ uint32_t total_s;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t y = __shfl_up_sync(kFull, inc, d);
    if (lane >= d) inc += y;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    uint32_t t = wsum[lane];
    uint32_t ti = t;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      uint32_t y = __shfl_up_sync(kFull, ti, d);
      if (lane >= d) ti += y;
    }
    wsum[lane] = ti - t;
    if (lane == 31) total_s = ti;
  }
  __syncthreads();
  *excl = wsum[wid] + inc - x;
  const uint32_t total = total_s;
  __syncthreads();
  return total;
}

__global__ void k_tile_sums(const uint32_t* __restrict__ in, int64_t n, uint32_t* __restrict__ tile_sum) {
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; i++)
    if (base + i < n) s += in[base + i];
  uint32_t ex;
  uint32_t tot = block_exclusive_scan(s, &ex);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}

// One block: exclusive scan of the tile totals in place, total at [ntiles].
__global__ void k_scan_tiles(uint32_t* tile_sum, int64_t ntiles) {
  uint32_t carry = 0;
  for (int64_t start = 0; start < ntiles; start += kTile) {
    const int64_t base = start + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
      v[i] = (base + i < ntiles) ? tile_sum[base + i] : 0;
      s += v[i];
    }
    uint32_t ex;
    uint32_t tot = block_exclusive_scan(s, &ex);
    uint32_t run = carry + ex;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
      if (base + i < ntiles) tile_sum[base + i] = run;
      run += v[i];
    }
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) tile_sum[ntiles] = carry;
}

// The sums also go to `copy` and, as 64-bit words, to `wide` (either may be
// null): the build's fill cursors start as its offsets.
struct ScanOut {
  uint32_t* out;
  uint32_t* copy;
  unsigned long long* wide;
  __device__ __forceinline__ void put(int64_t i, uint32_t v) const {
    out[i] = v;
    if (copy) copy[i] = v;
    if (wide) wide[i] = v;
  }
};

__global__ void k_tile_apply(const uint32_t* in, int64_t n, const uint32_t* __restrict__ tile_off, ScanOut out) {
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; i++) {
    v[i] = (base + i < n) ? in[base + i] : 0;
    s += v[i];
  }
  uint32_t ex;
  block_exclusive_scan(s, &ex);
  uint32_t run = tile_off[blockIdx.x] + ex;
#pragma unroll
  for (int i = 0; i < kScanItems; i++) {
    if (base + i < n) out.put(base + i, run);
    run += v[i];
  }
}

// The scan of at most kSmallTiles tiles in one launch, total at out[n].
constexpr int64_t kSmallTiles = 4;
__global__ void k_scan_small(const uint32_t* in, int64_t n, ScanOut out) {
  uint32_t carry = 0;
  for (int64_t start = 0; start < n; start += kTile) {
    const int64_t base = start + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
      v[i] = (base + i < n) ? in[base + i] : 0;
      s += v[i];
    }
    uint32_t ex;
    const uint32_t tot = block_exclusive_scan(s, &ex);
    uint32_t run = carry + ex;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
      if (base + i < n) out.put(base + i, run);
      run += v[i];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) out.out[n] = carry;
}

// Kept entries (|q| >= qmin) per tile of row entries, and, with the scanned
// tile counts, keep[i] = kept entries before i and the kept entries themselves
// in order.  Both stream the rows once (8 bytes an entry); the second pass
// mostly reads them from L2.
__device__ __forceinline__ bool entry_kept(uint64_t e, uint32_t qmin) {
  const int32_t q = adj_q(e);
  return (uint32_t)(q < 0 ? -q : q) >= qmin;
}
__global__ void k_keep_count(const uint64_t* __restrict__ adj, int64_t m, uint32_t qmin, uint32_t* __restrict__ tile_sum) {
  const int64_t base = (int64_t)blockIdx.x * kTile;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; i++) {
    const int64_t at = base + i * kScanThreads + threadIdx.x;
    if (at < m && entry_kept(adj[at], qmin)) s++;
  }
  uint32_t ex;
  const uint32_t tot = block_exclusive_scan(s, &ex);
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = tot;
}
__global__ void k_keep_apply(const uint64_t* __restrict__ adj, int64_t m, uint32_t qmin,
                             const uint32_t* __restrict__ tile_off, uint32_t* __restrict__ keep,
                             uint64_t* __restrict__ kept) {
  uint32_t run = tile_off[blockIdx.x];
  const int64_t base = (int64_t)blockIdx.x * kTile;
#pragma unroll
  for (int i = 0; i < kScanItems; i++) {  // coalesced: kScanThreads consecutive entries at a time
    const int64_t at = base + i * kScanThreads + threadIdx.x;
    const uint64_t e = at < m ? adj[at] : 0ull;
    const uint32_t on = at < m && entry_kept(e, qmin) ? 1u : 0u;
    uint32_t ex;
    const uint32_t tot = block_exclusive_scan(on, &ex);
    if (at < m) keep[at] = run + ex;
    if (on) kept[run + ex] = e;
    run += tot;
  }
}

__global__ void k_write_total(const uint32_t* tile_off, int64_t ntiles, uint32_t* out, int64_t n) {
  out[n] = tile_off[ntiles];
}

}  // namespace

size_t scan_tmp_words(int64_t n) { return (size_t)((n + kTile - 1) / kTile) + 2; }

// out[0..n] = exclusive prefix sums of in[0..n), out[n] = total; copy[0..n) and
// wide[0..n), where given, the sums again.  `in` may alias `out` or `copy`.
// tmp holds scan_tmp_words(n) words.
cudaError_t exclusive_scan_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* tmp, cudaStream_t s,
                               uint32_t* copy, unsigned long long* wide) {
  const ScanOut to{out, copy, wide};
  const int64_t ntiles = (n + kTile - 1) / kTile;
  if (ntiles <= kSmallTiles) {
    k_scan_small<<<1, kScanThreads, 0, s>>>(in, n, to);
    return cudaGetLastError();
  }
  k_tile_sums<<<(unsigned)ntiles, kScanThreads, 0, s>>>(in, n, tmp);
  k_scan_tiles<<<1, kScanThreads, 0, s>>>(tmp, ntiles);
  k_tile_apply<<<(unsigned)ntiles, kScanThreads, 0, s>>>(in, n, tmp, to);
  k_write_total<<<1, 1, 0, s>>>(tmp, ntiles, out, n);
  return cudaGetLastError();
}

// keep[0..m]: kept entries before each position, and the kept entries in
// order.  tmp holds scan_tmp_words(m) words.
cudaError_t keep_entries(const uint64_t* adj, int64_t m, uint32_t qmin, uint32_t* keep, uint64_t* kept, uint32_t* tmp,
                         cudaStream_t s) {
  const int64_t ntiles = (m + kTile - 1) / kTile;
  if (ntiles > 0) k_keep_count<<<(unsigned)ntiles, kScanThreads, 0, s>>>(adj, m, qmin, tmp);
  k_scan_tiles<<<1, kScanThreads, 0, s>>>(tmp, ntiles);
  if (ntiles > 0) k_keep_apply<<<(unsigned)ntiles, kScanThreads, 0, s>>>(adj, m, qmin, tmp, keep, kept);
  k_write_total<<<1, 1, 0, s>>>(tmp, ntiles, keep, m);
  return cudaGetLastError();
}

}  // namespace ubt
