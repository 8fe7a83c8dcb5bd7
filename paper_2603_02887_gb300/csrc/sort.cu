// Device radix sort (stable LSD, 8-bit digits), exclusive scan of tile counts, and tile ranges.
//
// The sort works on `nseg` equal segments of seg_len items at once, each sorted on its own (the depth sort
// of a batch sorts every view's Gaussians in one launch per kernel). Each pass runs three kernels:
//   upsweep   per block of 1024 (or 4096) items of a segment: digit histogram -> hist[segment][digit][block]
//   scan      one block per (segment, digit): exclusive scan of that row in place, total -> totals
//   downsweep per block: stable rank of every item within the block (warp multi-split: the lanes with
//             the same digit from one ballot per digit bit; warps in order), reorder in shared memory so
//             that items of one digit are contiguous, then a coalesced scatter to
//             segment start + base(digit) + hist[segment][digit][block] + rank, base = exclusive scan of
//             the segment's digit totals.
// Stability (equal digits keep their input order) makes the LSD passes a correct sort, and it is what
// orders equal depths by Gaussian index (the pairs are emitted in index order within one depth).
// A count known only on the device (the number of pairs, inside a captured graph) is read by every
// kernel: blocks past it contribute empty histograms and move nothing.
#include <algorithm>

#include "ngs_internal.cuh"

namespace ngs {
namespace {

// Exclusive prefix sum over a block (warp shuffles, then one warp scans the warp totals).
// `s_warp` needs THREADS/32 entries; all threads must call it. Returns the exclusive prefix of `v`;
// *total receives the block's sum.
template <int THREADS, typename T>
__device__ __forceinline__ T block_exclusive_sum(T v, T* s_warp, T* total) {
  constexpr int NW = THREADS / 32;
  static_assert(NW <= 32, "block too large");
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T w = lane < NW ? s_warp[lane] : (T)0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xFFFFFFFFu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < NW) s_warp[lane] = w;
  }
  __syncthreads();
  T prefix = warp > 0 ? s_warp[warp - 1] : (T)0;
  *total = s_warp[NW - 1];
  __syncthreads();
  return prefix + x - v;
}

constexpr int kThreads = 256;
// Items per thread: 4 (1024 per CTA) up to kSmallSort items per segment, where the passes are latency-bound
// and more CTAs hide more latency (a sweep of 4..16 on GB300 at 0.5-3.3 M items); 16 above it, where the
// per-digit scans over the CTAs' counts would otherwise grow long.
constexpr int kSmallSort = 1 << 23;
template <int ITEMS>
struct SortTile {
  static constexpr int kTile = kThreads * ITEMS;
};
__host__ __device__ constexpr int tile_items(uint32_t seg_len) { return seg_len <= (uint32_t)kSmallSort ? 1024 : 4096; }
constexpr int kWarps = kThreads / 32;
constexpr int kDigits = 256;

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K key, int shift) {
  return (uint32_t)(key >> shift) & 0xFFu;
}

__device__ __forceinline__ uint32_t segment_count(uint32_t seg_len, const uint32_t* n_dev) {
  return n_dev ? min(*n_dev, seg_len) : seg_len;
}

template <typename K, int ITEMS>
__global__ void __launch_bounds__(kThreads) upsweep_kernel(const K* __restrict__ keys, uint32_t seg_len,
                                                           const uint32_t* __restrict__ n_dev, int shift,
                                                           uint32_t* __restrict__ hist, uint32_t nblocks) {
  pdl_wait();
  __shared__ uint32_t s_hist[kWarps][kDigits];
  int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t seg = blockIdx.x / nblocks, blk = blockIdx.x - seg * nblocks;
  const uint32_t n = segment_count(seg_len, n_dev);
  keys += (size_t)seg * seg_len;
  hist += (size_t)seg * kDigits * nblocks;
  for (int i = tid; i < kWarps * kDigits; i += kThreads) (&s_hist[0][0])[i] = 0;
  __syncthreads();
  constexpr int kTile = SortTile<ITEMS>::kTile;
  uint32_t base = blk * (uint32_t)kTile;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    uint32_t idx = base + j * kThreads + tid;
    // a plain shared-memory atomic per item (measured on GB300: faster than aggregating the warp's equal
    // digits with __match_any_sync first, by 11 % on the depth sort and 18 % on the tile sort)
    if (idx < n) atomicAdd(&s_hist[warp][digit_of(keys[idx], shift)], 1u);
  }
  __syncthreads();
  for (int d = tid; d < kDigits; d += kThreads) {
    uint32_t sum = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sum += s_hist[w][d];
    hist[(size_t)d * nblocks + blk] = sum;
  }
}

// One block per (segment, digit): exclusive scan of that digit's per-block counts; the digit's total goes
// to totals[segment][digit] (stored after the histograms).
__global__ void __launch_bounds__(1024) scan_digit_kernel(uint32_t* hist, uint32_t nblocks, uint32_t* totals) {
  pdl_wait();
  __shared__ uint32_t s_warp[32];
  uint32_t* row = hist + (size_t)blockIdx.x * nblocks;
  uint32_t carry = 0;
  for (uint32_t base = 0; base < nblocks; base += 1024) {
    uint32_t i = base + threadIdx.x;
    uint32_t v = i < nblocks ? row[i] : 0u, agg;
    uint32_t ex = block_exclusive_sum<1024>(v, s_warp, &agg);
    if (i < nblocks) row[i] = ex + carry;
    carry += agg;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

template <typename K, int ITEMS>
__global__ void __launch_bounds__(kThreads) downsweep_kernel(const K* __restrict__ keys_in,
                                                             const uint32_t* __restrict__ vals_in,
                                                             K* __restrict__ keys_out, uint32_t* __restrict__ vals_out,
                                                             uint32_t seg_len, const uint32_t* __restrict__ n_dev,
                                                             int shift, const uint32_t* __restrict__ hist,
                                                             const uint32_t* __restrict__ totals, uint32_t nblocks) {
  pdl_wait();
  constexpr int kTile = SortTile<ITEMS>::kTile, kItems = ITEMS;
  const uint32_t seg = blockIdx.x / nblocks, blk = blockIdx.x - seg * nblocks;
  const uint32_t n = segment_count(seg_len, n_dev);
  if (blk * (uint32_t)kTile >= n) return;  // the whole block is past the segment's items
  {
    const size_t off = (size_t)seg * seg_len;
    keys_in += off;
    vals_in += off;
    keys_out += off;
    vals_out += off;
    hist += (size_t)seg * kDigits * nblocks;
    totals += (size_t)seg * kDigits;
  }
  extern __shared__ __align__(16) unsigned char smem[];
  K* s_keys = reinterpret_cast<K*>(smem);
  uint32_t* s_vals = reinterpret_cast<uint32_t*>(smem + sizeof(K) * kTile);
  __shared__ uint32_t s_cnt[kWarps][kDigits];  // per-warp digit counters, then per-warp offsets
  __shared__ uint32_t s_local[kDigits];         // block-local start of each digit
  __shared__ uint32_t s_global[kDigits];        // global start of this block's run of each digit
  __shared__ uint32_t s_warp[kWarps];

  int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < kWarps * kDigits; i += kThreads) (&s_cnt[0][0])[i] = 0;
  __syncthreads();

  uint32_t base = blk * (uint32_t)kTile + warp * (kTile / kWarps);
  K key[kItems];
  uint32_t val[kItems], rank[kItems], dig[kItems];
  uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    uint32_t idx = base + r * 32 + lane;
    bool valid = idx < n;
    key[r] = valid ? keys_in[idx] : (K)0;
    val[r] = valid ? vals_in[idx] : 0u;
    uint32_t d = valid ? digit_of(key[r], shift) : (uint32_t)kDigits;  // kDigits = "no item"
    dig[r] = d;
    // lanes holding the same digit (0..255, or 256 for "no item"): one ballot per bit of d (measured on
    // GB300: 2-4 % faster sorts than __match_any_sync)
    uint32_t peers = 0xFFFFFFFFu;
#pragma unroll
    for (int bit = 0; bit < 9; ++bit) {
      const bool one = (d >> bit) & 1u;
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, one);
      peers &= one ? bal : ~bal;
    }
    uint32_t before = valid ? s_cnt[warp][d] : 0u;
    rank[r] = before + __popc(peers & lt);
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) s_cnt[warp][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // per digit: exclusive offsets over warps, block total, block-local digit start, global start
  uint32_t total = 0;
  {
    int d = tid;  // kThreads == kDigits
    for (int w = 0; w < kWarps; ++w) {
      uint32_t c = s_cnt[w][d];
      s_cnt[w][d] = total;
      total += c;
    }
    uint32_t agg;
    s_local[d] = block_exclusive_sum<kThreads>(total, s_warp, &agg);
  }
  {
    // global digit base = exclusive scan of the digit totals; this block's run starts hist[d][b] into it
    uint32_t agg;
    uint32_t ex = block_exclusive_sum<kThreads>(totals[tid], s_warp, &agg);
    s_global[tid] = ex + hist[(size_t)tid * nblocks + blk];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    if (dig[r] < (uint32_t)kDigits) {
      uint32_t pos = s_local[dig[r]] + s_cnt[warp][dig[r]] + rank[r];
      s_keys[pos] = key[r];
      s_vals[pos] = val[r];
    }
  }
  __syncthreads();
  uint32_t count = min((uint32_t)kTile, n - blk * (uint32_t)kTile);
  for (uint32_t i = tid; i < count; i += kThreads) {
    K k = s_keys[i];
    uint32_t d = digit_of(k, shift);
    uint32_t g = s_global[d] + (i - s_local[d]);
    keys_out[g] = k;
    vals_out[g] = s_vals[i];
  }
}

template <typename K, int ITEMS>
int radix_sort(K* keys[2], uint32_t* vals[2], uint32_t seg_len, uint32_t nseg, const uint32_t* n_dev, int begin_bit,
               int end_bit, uint32_t* hist, cudaStream_t s, int* launches) {
  constexpr int kTile = SortTile<ITEMS>::kTile;
  int cur = 0;
  if (seg_len <= 1 || nseg == 0 || begin_bit >= end_bit) return cur;
  uint32_t nblocks = (seg_len + kTile - 1) / kTile;
  uint32_t grid = nblocks * nseg;
  uint32_t* totals = hist + (size_t)kDigits * nblocks * nseg;
  // at most 24 KB of dynamic shared memory (for 64-bit keys), within the default limit without an opt-in
  size_t smem = (sizeof(K) + sizeof(uint32_t)) * kTile;
  for (int shift = begin_bit; shift < end_bit; shift += 8) {
    launch_pdl(upsweep_kernel<K, ITEMS>, grid, kThreads, 0, s, keys[cur], seg_len, n_dev, shift, hist, nblocks);
    launch_pdl(scan_digit_kernel, kDigits * nseg, 1024, 0, s, hist, nblocks, totals);
    launch_pdl(downsweep_kernel<K, ITEMS>, grid, kThreads, smem, s, keys[cur], vals[cur], keys[cur ^ 1],
               vals[cur ^ 1], seg_len, n_dev, shift, hist, totals, nblocks);
    cur ^= 1;
    *launches += 3;
  }
  return cur;
}

// ---- exclusive scan of tile counts taken in depth order ---------------------------------------------

constexpr int kScanThreads = 512;
// Items per thread: 2 up to kScanSmall items, where the scan is a few hundred CTAs of gathers and more
// CTAs hide their latency; 8 above, which keeps the per-CTA sums that one CTA scans short.
constexpr uint32_t kScanSmall = 1u << 21;
constexpr int scan_items(uint32_t n) { return n <= kScanSmall ? 2 : 8; }

template <int kScanItems>
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const uint32_t* __restrict__ count,
                                                                   const uint32_t* __restrict__ order, uint32_t n,
                                                                   uint64_t* __restrict__ block_sums) {
  pdl_wait();
  __shared__ uint64_t s_warp[kScanThreads / 32];
  constexpr int kScanTile = kScanThreads * kScanItems;
  uint64_t sum = 0;
  uint32_t base = blockIdx.x * (uint32_t)kScanTile;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    uint32_t i = base + j * kScanThreads + threadIdx.x;
    if (i < n) sum += count[order[i]];
  }
  uint64_t agg;
  block_exclusive_sum<kScanThreads>(sum, s_warp, &agg);
  if (threadIdx.x == 0) block_sums[blockIdx.x] = agg;
}

__global__ void __launch_bounds__(1024) scan_block_sums_kernel(uint64_t* block_sums, uint32_t nblocks, uint64_t* total) {
  pdl_wait();
  __shared__ uint64_t s_warp[32];
  uint64_t carry = 0;
  for (uint32_t base = 0; base < nblocks; base += 1024) {
    uint32_t i = base + threadIdx.x;
    uint64_t v = i < nblocks ? block_sums[i] : 0, agg;
    uint64_t ex = block_exclusive_sum<1024>(v, s_warp, &agg);
    if (i < nblocks) block_sums[i] = ex + carry;
    carry += agg;
  }
  if (threadIdx.x == 0) *total = carry;
}

template <int kScanItems>
__global__ void __launch_bounds__(kScanThreads) scan_final_kernel(const uint32_t* __restrict__ count,
                                                                  const uint32_t* __restrict__ order, uint32_t n,
                                                                  const uint64_t* __restrict__ block_offsets,
                                                                  uint32_t* __restrict__ offsets) {
  pdl_wait();
  constexpr int kScanTile = kScanThreads * kScanItems;
  __shared__ uint32_t s_warp[kScanThreads / 32];
  uint32_t base = blockIdx.x * (uint32_t)kScanTile + threadIdx.x * kScanItems;  // blocked arrangement
  uint32_t v[kScanItems], local = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    uint32_t i = base + j;
    v[j] = i < n ? count[order[i]] : 0u;
    local += v[j];
  }
  uint32_t agg;
  uint32_t run = (uint32_t)block_offsets[blockIdx.x] + block_exclusive_sum<kScanThreads>(local, s_warp, &agg);
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    uint32_t i = base + j;
    if (i < n) offsets[i] = run;
    run += v[j];
    if (i == n - 1) offsets[n] = run;
  }
}

__global__ void tile_ranges_kernel(const uint32_t* __restrict__ tiles, const uint32_t* __restrict__ vals,
                                   const ViewParams* __restrict__ views, uint32_t n_per_view, uint32_t n_views,
                                   uint32_t npairs_cap, const uint32_t* __restrict__ npairs_dev, uint32_t ntiles,
                                   uint2* __restrict__ ranges, uint32_t* check) {
  pdl_wait();
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t npairs = npairs_dev ? min(*npairs_dev, npairs_cap) : npairs_cap;
  if (i >= npairs) return;
  if (n_views == 1) {
    const uint32_t t = tiles[i];
    if (t >= ntiles) {  // never from a correct sort: skipped and reported
      atomicOr(check, kCheckTile);
      return;
    }
    if (i == 0 || tiles[i - 1] != t) ranges[t].x = i;
    if (i == npairs - 1 || tiles[i + 1] != t) ranges[t].y = i + 1;
    return;
  }
  // a batch: a run is a (view-local tile, view) pair, compared without the view table; only the first and
  // last pair of a run look up the view's first tile
  const uint32_t n_records = n_per_view * n_views;
  const uint32_t v = vals[i];
  if (v >= n_records) {  // never from a correct sort: skipped and reported (the compositing checks it too)
    atomicOr(check, kCheckIndex);
    return;
  }
  const uint32_t loc = tiles[i], view = v / n_per_view;
  auto same = [&](uint32_t j) { return tiles[j] == loc && vals[j] / n_per_view == view; };
  const bool first = i == 0 || !same(i - 1), last = i == npairs - 1 || !same(i + 1);
  if (!(first || last)) return;
  const uint32_t t = __ldg(&views[view].tile_base) + loc;
  if (t >= ntiles) {
    atomicOr(check, kCheckTile);
    return;
  }
  if (first) ranges[t].x = i;
  if (last) ranges[t].y = i + 1;
}

// One warp per tile: the 64-bit keys of its list (diagnostics).
__global__ void __launch_bounds__(256) compose_keys_kernel(const uint2* __restrict__ ranges, uint32_t ntiles,
                                                           const uint32_t* __restrict__ ids,
                                                           const float4* __restrict__ rec,
                                                           uint64_t* __restrict__ keys) {
  const uint32_t t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= ntiles) return;
  const uint2 r = ranges[t];
  for (uint32_t i = r.x + (threadIdx.x & 31); i < r.y; i += 32)
    keys[i] = ((uint64_t)t << 32) | (uint64_t)__float_as_uint(rec[3 * (size_t)ids[i] + 2].y);
}

// ---- tile work order for the persistent composite: descending pair count ---------------------------

__device__ __forceinline__ uint32_t cost_bucket(uint2 r) {
  const uint32_t c = r.y - r.x;
  return (uint32_t)(kCostBuckets - 1) - (c ? 32u - (uint32_t)__clz(c) : 0u);  // 0 = most pairs
}

__global__ void __launch_bounds__(256) tile_bucket_count_kernel(const uint2* __restrict__ ranges, uint32_t ntiles,
                                                                uint32_t* __restrict__ counts) {
  pdl_wait();
  __shared__ uint32_t s_cnt[kCostBuckets];
  if (threadIdx.x < kCostBuckets) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < ntiles) atomicAdd(&s_cnt[cost_bucket(ranges[t])], 1u);
  __syncthreads();
  if (threadIdx.x < kCostBuckets && s_cnt[threadIdx.x]) atomicAdd(&counts[threadIdx.x], s_cnt[threadIdx.x]);
}

__global__ void __launch_bounds__(256) tile_bucket_scatter_kernel(const uint2* __restrict__ ranges, uint32_t ntiles,
                                                                  const uint32_t* __restrict__ counts,
                                                                  uint32_t* __restrict__ cursors,
                                                                  uint32_t* __restrict__ work) {
  pdl_wait();
  __shared__ uint32_t s_start[kCostBuckets];
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int b = 0; b < kCostBuckets; ++b) {
      s_start[b] = run;
      run += counts[b];
    }
  }
  __syncthreads();
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t b = t < ntiles ? cost_bucket(ranges[t]) : (uint32_t)kCostBuckets;
  const uint32_t peers = __match_any_sync(0xFFFFFFFFu, b);
  const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
  uint32_t base = 0;
  if (b < (uint32_t)kCostBuckets && lane == leader) base = atomicAdd(&cursors[b], (uint32_t)__popc(peers));
  base = __shfl_sync(0xFFFFFFFFu, base, leader);
  if (b < (uint32_t)kCostBuckets) work[s_start[b] + base + __popc(peers & ((1u << lane) - 1u))] = t;
}

// ---- per-tile lists by counting ------------------------------------------------------------------------
//
// The lists of all tiles without a global sort: the projection counts every tile's splats, a scan of the
// counts gives each tile its segment of the pair array, the emission drops each (depth, record) pair at the
// next free slot of its tile's segment, in any order, and tile_sort_kernel sorts every segment by
// (depth, record index). That is the order the two stable radix sorts give, with each pair written and read
// once (8 B) and 4 B written, instead of 3 radix passes' worth of 16 B, and 3 kernels instead of about 20.

constexpr int kBinThreads = 256;
static_assert(kBinBlock == 4 * kBinThreads, "four tiles per thread");
static_assert(kCostBuckets == 33, "a warp and one more");
constexpr int kSortThreads = 256;
constexpr int kWarpList = 256;     // longest list sorted by one warp
constexpr int kWarpBuckets = 256;  // its buckets
constexpr int kCtaList = kWarpList * (kSortThreads / 32);  // keys a CTA holds in shared memory
constexpr int kCtaBuckets = kWarpBuckets * (kSortThreads / 32);
// With more keys in one bucket, a list is sorted by the network, not by comparing each key with its bucket's: the
// network of a CTA is 66 steps with a barrier each, so that it pays later.
constexpr uint32_t kHeavy = 48, kHeavyCta = 160;

// ranges[t].y holds tile t's count; afterwards ranges[t] = (o, o) with o the number of pairs in the tiles
// before t of its block of kBinBlock tiles. `bases` receives the blocks' first pairs, *total the pair count:
// the block that finishes last scans the blocks' sums, so that no block waits on another. Tiles whose lists are
// too long for one warp are listed in `big` (as far as its big_cap entries go; total[kTotalBig] counts them all).
// With `sched`, the work list's first entry of each cost bucket is left in the bucket's cursor. The count and the
// device error word are published in the host mirror.
__global__ void __launch_bounds__(kBinThreads) tile_scan_kernel(uint2* __restrict__ ranges, uint32_t ntiles,
                                                                uint64_t* bases, uint64_t* total,
                                                                uint32_t* __restrict__ big, uint32_t big_cap,
                                                                uint32_t* sched, uint64_t* mirror) {
  pdl_wait();
  __shared__ uint32_t s_warp[kBinThreads / 32];
  __shared__ uint64_t s_warp64[kBinThreads / 32];
  __shared__ uint32_t s_cost[kCostBuckets];
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  if (sched) {
    if (tid < kCostBuckets) s_cost[tid] = 0;
    __syncthreads();
  }
  const uint32_t t0 = blockIdx.x * (uint32_t)kBinBlock + 4 * tid;
  uint32_t c[4], sum = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c[k] = t0 + k < ntiles ? ranges[t0 + k].y : 0u;
    if (sched && t0 + k < ntiles) atomicAdd(&s_cost[cost_bucket(make_uint2(0, c[k]))], 1u);
    sum += c[k];
    if (c[k] > (uint32_t)kWarpList) {
      const uint32_t at = atomicAdd(reinterpret_cast<uint32_t*>(total + kTotalBig), 1u);
      if (at < big_cap) big[at] = t0 + k;
    }
  }
  uint32_t agg;
  uint32_t run = block_exclusive_sum<kBinThreads>(sum, s_warp, &agg);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (t0 + k < ntiles) ranges[t0 + k] = make_uint2(run, run);
    run += c[k];
  }
  if (sched && tid < kCostBuckets && s_cost[tid]) {
    atomicAdd(&sched[2 + tid], s_cost[tid]);
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) {
    bases[blockIdx.x] = agg;
    __threadfence();
    s_last = atomicAdd(reinterpret_cast<uint32_t*>(total + kTotalTicket), 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  uint64_t carry = 0;
  for (uint32_t b = 0; b < gridDim.x; b += kBinThreads) {
    const uint32_t i = b + tid;
    const uint64_t v = i < gridDim.x ? __ldcg(reinterpret_cast<unsigned long long*>(bases) + i) : 0ull;
    uint64_t a64;
    const uint64_t ex = block_exclusive_sum<kBinThreads>(v, s_warp64, &a64);
    if (i < gridDim.x) bases[i] = ex + carry;
    carry += a64;
  }
  if (sched && tid < 32) {  // kCostBuckets == 33: lane l takes bucket l, the last bucket follows the others
    const uint32_t v = __ldcg(&sched[2 + tid]);
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (tid >= o) incl += y;
    }
    sched[2 + kCostBuckets + tid] = incl - v;
    if (tid == 31) sched[2 + kCostBuckets + 32] = incl;
  }
  if (tid == 0) {
    total[0] = carry;
    mirror[0] = carry;
    mirror[1] = total[1];
    __threadfence_system();
  }
}

// Sorts a[0, n) ascending in place: a bitonic network whose comparators all point up, so that the elements
// past n (as if infinite) never move. The group of `size` threads that calls it (member `me`) synchronises
// with `sync`. For lists the bucket sort below cannot split.
template <typename Sync>
__device__ __forceinline__ void bitonic_sort(unsigned long long* a, uint32_t n, uint32_t me, uint32_t size, Sync sync) {
  for (uint32_t k = 2; k != 0 && (k >> 1) < n; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      const uint32_t mask = j == (k >> 1) ? k - 1 : j;  // the first step of a merge mirrors its second half
      for (uint32_t i = me; i < n; i += size) {
        const uint32_t p = i ^ mask;
        if (p > i && p < n) {
          const unsigned long long x = a[i], y = a[p];
          if (y < x) {
            a[i] = y;
            a[p] = x;
          }
        }
      }
      sync();
    }
  }
}

// A key's bucket: linear over the list's range of depth bits (or of record indices, where all depths are
// equal), so that equal keys share one and buckets ascend with the keys.
struct BucketMap {
  uint32_t lo;
  float scale;
  bool by_id;
  __device__ __forceinline__ BucketMap(uint32_t hmin, uint32_t hmax, uint32_t lmin, uint32_t lmax, uint32_t nb)
      : lo(hmin == hmax ? lmin : hmin),
        scale((float)nb / ((float)(hmin == hmax ? lmax - lmin : hmax - hmin) + 1.0f)),
        by_id(hmin == hmax) {}
  __device__ __forceinline__ uint32_t operator()(unsigned long long key, uint32_t nb) const {
    const uint32_t v = (by_id ? (uint32_t)key : (uint32_t)(key >> 32)) - lo;
    return min((uint32_t)(__uint2float_rz(v) * scale), nb - 1);
  }
};

// The position of key a[i] among the keys of its bucket a[first, last).
__device__ __forceinline__ uint32_t rank_in_bucket(const unsigned long long* a, uint32_t first, uint32_t last,
                                                   unsigned long long key) {
  uint32_t r = first;
  if (last - first > 1)
    for (uint32_t q = first; q < last; ++q) r += a[q] < key ? 1u : 0u;
  return r;
}

// One warp sorts keys[0, n), n <= kWarpList, and writes the record indices to out. One bucket per key or more:
// count, scan, scatter into shared memory, then each key's place within its bucket by comparison.
__device__ __forceinline__ void warp_sort_list(const unsigned long long* __restrict__ keys, uint32_t n,
                                               uint32_t* __restrict__ out, unsigned long long* s_key, uint32_t* s_cnt) {
  constexpr int kPer = kWarpList / 32;
  const uint32_t full = 0xFFFFFFFFu, lane = threadIdx.x & 31;
  unsigned long long k[kPer];
  uint32_t hmin = full, hmax = 0, lmin = full, lmax = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    if (j * 32u >= n) break;
    if (j * 32 + lane < n) {
      k[j] = keys[j * 32 + lane];
      hmin = min(hmin, (uint32_t)(k[j] >> 32));
      hmax = max(hmax, (uint32_t)(k[j] >> 32));
      lmin = min(lmin, (uint32_t)k[j]);
      lmax = max(lmax, (uint32_t)k[j]);
    }
  }
  hmin = __reduce_min_sync(full, hmin);
  hmax = __reduce_max_sync(full, hmax);
  if (hmin == hmax) {
    lmin = __reduce_min_sync(full, lmin);
    lmax = __reduce_max_sync(full, lmax);
  }
  const BucketMap bucket(hmin, hmax, lmin, lmax, kWarpBuckets);
  uint4* cnt4 = reinterpret_cast<uint4*>(s_cnt);
  cnt4[2 * lane] = cnt4[2 * lane + 1] = make_uint4(0, 0, 0, 0);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    if (j * 32u >= n) break;
    if (j * 32 + lane < n) atomicAdd(&s_cnt[bucket(k[j], kWarpBuckets)], 1u);
  }
  __syncwarp();
  uint4 c0 = cnt4[2 * lane], c1 = cnt4[2 * lane + 1];
  const uint32_t most = __reduce_max_sync(full, max(max(max(c0.x, c0.y), max(c0.z, c0.w)), max(max(c1.x, c1.y), max(c1.z, c1.w))));
  const uint32_t sum = c0.x + c0.y + c0.z + c0.w + c1.x + c1.y + c1.z + c1.w;
  uint32_t run = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(full, run, o);
    if (lane >= (uint32_t)o) run += y;
  }
  run -= sum;
  uint4 e0, e1;
  e0.x = run;
  e0.y = e0.x + c0.x;
  e0.z = e0.y + c0.y;
  e0.w = e0.z + c0.z;
  e1.x = e0.w + c0.w;
  e1.y = e1.x + c1.x;
  e1.z = e1.y + c1.y;
  e1.w = e1.z + c1.z;
  cnt4[2 * lane] = e0;
  cnt4[2 * lane + 1] = e1;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    if (j * 32u >= n) break;
    if (j * 32 + lane < n) s_key[atomicAdd(&s_cnt[bucket(k[j], kWarpBuckets)], 1u)] = k[j];
  }
  __syncwarp();  // s_cnt[b] is now the end of bucket b
  if (most > kHeavy) {
    bitonic_sort(s_key, n, lane, 32, [] { __syncwarp(); });
    for (uint32_t i = lane; i < n; i += 32) out[i] = (uint32_t)s_key[i];
  } else {
    for (uint32_t i = lane; i < n; i += 32) {
      const unsigned long long key = s_key[i];
      const uint32_t b = bucket(key, kWarpBuckets);
      out[rank_in_bucket(s_key, b ? s_cnt[b - 1] : 0u, s_cnt[b], key)] = (uint32_t)key;
    }
  }
}

// Exclusive prefix sums of the CTA's kCtaBuckets counts, in place; the largest count is returned to every thread.
__device__ __forceinline__ uint32_t cta_scan_buckets(uint32_t* s_cnt, uint32_t* s_red) {
  const uint32_t tid = threadIdx.x;
  uint4* cnt4 = reinterpret_cast<uint4*>(s_cnt);
  const uint4 c0 = cnt4[2 * tid], c1 = cnt4[2 * tid + 1];
  uint32_t most = max(max(max(c0.x, c0.y), max(c0.z, c0.w)), max(max(c1.x, c1.y), max(c1.z, c1.w)));
  most = __reduce_max_sync(0xFFFFFFFFu, most);
  if ((tid & 31) == 0) s_red[8 + (tid >> 5)] = most;
  const uint32_t sum = c0.x + c0.y + c0.z + c0.w + c1.x + c1.y + c1.z + c1.w;
  uint32_t agg;
  const uint32_t run = block_exclusive_sum<kSortThreads>(sum, s_red, &agg);
#pragma unroll
  for (int w = 0; w < kSortThreads / 32; ++w) most = max(most, s_red[8 + w]);
  uint4 e0, e1;
  e0.x = run;
  e0.y = e0.x + c0.x;
  e0.z = e0.y + c0.y;
  e0.w = e0.z + c0.z;
  e1.x = e0.w + c0.w;
  e1.y = e1.x + c1.x;
  e1.z = e1.y + c1.y;
  e1.w = e1.z + c1.z;
  cnt4[2 * tid] = e0;
  cnt4[2 * tid + 1] = e1;
  __syncthreads();
  return most;
}

// The range of the CTA's keys (each thread has reduced its own), and zeroed bucket counts.
__device__ __forceinline__ BucketMap cta_bucket_map(uint32_t hmin, uint32_t hmax, uint32_t lmin, uint32_t lmax,
                                                    uint32_t* s_cnt, uint32_t* s_red) {
  const uint32_t full = 0xFFFFFFFFu, tid = threadIdx.x, warp = tid >> 5;
  hmin = __reduce_min_sync(full, hmin);
  hmax = __reduce_max_sync(full, hmax);
  lmin = __reduce_min_sync(full, lmin);
  lmax = __reduce_max_sync(full, lmax);
  __syncthreads();  // the previous list's use of the shared arrays is over
  if ((tid & 31) == 0) {
    s_red[warp] = hmin;
    s_red[8 + warp] = hmax;
    s_red[16 + warp] = lmin;
    s_red[24 + warp] = lmax;
  }
  uint4* cnt4 = reinterpret_cast<uint4*>(s_cnt);
  cnt4[2 * tid] = cnt4[2 * tid + 1] = make_uint4(0, 0, 0, 0);
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSortThreads / 32; ++w) {
    hmin = min(hmin, s_red[w]);
    hmax = max(hmax, s_red[8 + w]);
    lmin = min(lmin, s_red[16 + w]);
    lmax = max(lmax, s_red[24 + w]);
  }
  return BucketMap(hmin, hmax, lmin, lmax, kCtaBuckets);
}

// The keys of a run of buckets stand in s_key[0, m), the run starting at list position `first`; s_cnt holds each
// bucket's end. Writes their record indices in order.
__device__ __forceinline__ void cta_write_run(unsigned long long* s_key, const uint32_t* s_cnt, uint32_t m, uint32_t first,
                                              const BucketMap& bucket, bool heavy, uint32_t* __restrict__ out) {
  if (heavy) {
    bitonic_sort(s_key, m, threadIdx.x, kSortThreads, [] { __syncthreads(); });
    for (uint32_t i = threadIdx.x; i < m; i += kSortThreads) out[first + i] = (uint32_t)s_key[i];
    return;
  }
  for (uint32_t i = threadIdx.x; i < m; i += kSortThreads) {
    const unsigned long long key = s_key[i];
    const uint32_t b = bucket(key, kCtaBuckets);
    const uint32_t from = b ? s_cnt[b - 1] : 0u;
    out[first + rank_in_bucket(s_key, from - first, s_cnt[b] - first, key)] = (uint32_t)key;
  }
}

// A CTA sorts keys[0, n), n <= kCtaList, as the warps do; the keys stay in registers between the passes.
__device__ __forceinline__ void cta_sort_list(const unsigned long long* __restrict__ keys, uint32_t n,
                                              uint32_t* __restrict__ out, unsigned long long* s_key, uint32_t* s_cnt,
                                              uint32_t* s_red) {
  constexpr int kPer = kCtaList / kSortThreads;
  const uint32_t full = 0xFFFFFFFFu, tid = threadIdx.x;
  unsigned long long k[kPer];
  uint32_t hmin = full, hmax = 0, lmin = full, lmax = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (j * kSortThreads + tid < n) k[j] = keys[j * kSortThreads + tid];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    if (j * kSortThreads + tid < n) {
      hmin = min(hmin, (uint32_t)(k[j] >> 32));
      hmax = max(hmax, (uint32_t)(k[j] >> 32));
      lmin = min(lmin, (uint32_t)k[j]);
      lmax = max(lmax, (uint32_t)k[j]);
    }
  }
  const BucketMap bucket = cta_bucket_map(hmin, hmax, lmin, lmax, s_cnt, s_red);
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (j * kSortThreads + tid < n) atomicAdd(&s_cnt[bucket(k[j], kCtaBuckets)], 1u);
  __syncthreads();
  const uint32_t most = cta_scan_buckets(s_cnt, s_red);
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (j * kSortThreads + tid < n) s_key[atomicAdd(&s_cnt[bucket(k[j], kCtaBuckets)], 1u)] = k[j];
  __syncthreads();
  cta_write_run(s_key, s_cnt, n, 0, bucket, most > kHeavyCta, out);
}

// Calls f(index, key) for every key, eight loads of a thread on their way at a time.
template <typename F>
__device__ __forceinline__ void for_keys(const unsigned long long* __restrict__ keys, uint32_t n, F f) {
  constexpr int kFlight = 8;
  for (uint32_t i0 = 0; i0 < n; i0 += kFlight * kSortThreads) {
    unsigned long long k[kFlight];
#pragma unroll
    for (int j = 0; j < kFlight; ++j) {
      const uint32_t i = i0 + j * kSortThreads + threadIdx.x;
      k[j] = i < n ? keys[i] : 0ull;
    }
#pragma unroll
    for (int j = 0; j < kFlight; ++j) {
      const uint32_t i = i0 + j * kSortThreads + threadIdx.x;
      if (i < n) f(i, k[j]);
    }
  }
}

// A list of any length: the keys' places by bucket go to `tmp` (n words), and runs of consecutive buckets that shared
// memory holds are then sorted one after another. A bucket that alone exceeds it leaves the list to the network, in
// place in global memory.
__device__ __noinline__ void cta_sort_long_list(unsigned long long* keys, uint32_t n, uint32_t* __restrict__ out,
                                                uint32_t* tmp, unsigned long long* s_key, uint32_t* s_cnt,
                                                uint32_t* s_red) {
  const uint32_t full = 0xFFFFFFFFu, tid = threadIdx.x;
  uint32_t hmin = full, hmax = 0, lmin = full, lmax = 0;
  for_keys(keys, n, [&](uint32_t, unsigned long long k) {
    hmin = min(hmin, (uint32_t)(k >> 32));
    hmax = max(hmax, (uint32_t)(k >> 32));
    lmin = min(lmin, (uint32_t)k);
    lmax = max(lmax, (uint32_t)k);
  });
  const BucketMap bucket = cta_bucket_map(hmin, hmax, lmin, lmax, s_cnt, s_red);
  for_keys(keys, n, [&](uint32_t, unsigned long long k) { atomicAdd(&s_cnt[bucket(k, kCtaBuckets)], 1u); });
  __syncthreads();
  const uint32_t most = cta_scan_buckets(s_cnt, s_red);
  if (most > (uint32_t)kCtaList) {
    bitonic_sort(keys, n, tid, kSortThreads, [] { __syncthreads(); });
    for (uint32_t i = tid; i < n; i += kSortThreads) out[i] = (uint32_t)keys[i];
    return;
  }
  for_keys(keys, n,
           [&](uint32_t i, unsigned long long k) { tmp[atomicAdd(&s_cnt[bucket(k, kCtaBuckets)], 1u)] = i; });
  __syncthreads();  // s_cnt[b] is now the end of bucket b
  for (uint32_t b0 = 0, first = 0; first < n;) {
    // buckets [b0, l] hold at most kCtaList keys, list positions [first, first + m): no bucket is larger
    uint32_t l = b0, h = kCtaBuckets - 1;
    while (l < h) {
      const uint32_t mid = (l + h + 1) >> 1;
      if (s_cnt[mid] - first <= (uint32_t)kCtaList) l = mid;
      else h = mid - 1;
    }
    const uint32_t m = s_cnt[l] - first;
    for (uint32_t i0 = 0; i0 < m; i0 += 4 * kSortThreads) {
      uint32_t at[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t i = i0 + j * kSortThreads + tid;
        at[j] = i < m ? tmp[first + i] : 0u;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t i = i0 + j * kSortThreads + tid;
        if (i < m) s_key[i] = keys[at[j]];
      }
    }
    __syncthreads();
    cta_write_run(s_key, s_cnt, m, first, bucket, most > kHeavyCta, out);
    __syncthreads();
    b0 = l + 1;
    first += m;
  }
}

// Tile t's segment of the pair array: an asynchronous render's lists may run past the capacity.
__device__ __forceinline__ uint2 tile_segment(const uint64_t* __restrict__ bases, uint2 local, uint32_t t, uint32_t cap) {
  const uint64_t base = bases[t / kBinBlock];
  const uint2 r = make_uint2((uint32_t)min(base + local.x, (uint64_t)cap), (uint32_t)min(base + local.y, (uint64_t)cap));
  return r.y > r.x ? r : make_uint2(0, 0);
}

// Sorts every tile's segment and finishes its range: [start, end), or (0, 0) for an empty tile. The first
// `big_ctas` CTAs take the lists of more than kWarpList keys (from `big`, or, where that overflowed, among all
// tiles), each sorted by the whole CTA; the warps of the others take one tile each. With `sched`, each tile takes
// its place in the work list of descending cost.
__global__ void __launch_bounds__(kSortThreads, 5)
    tile_sort_kernel(unsigned long long* keys, uint32_t cap, const uint64_t* __restrict__ bases, uint32_t ntiles,
                     const uint2* local, uint2* __restrict__ ranges, uint32_t* __restrict__ out, uint32_t* tmp, uint32_t big_ctas,
                     const uint32_t* __restrict__ big, uint32_t big_cap, const uint64_t* __restrict__ total,
                     uint32_t* __restrict__ sched, uint32_t* __restrict__ work) {
  pdl_wait();
  __shared__ __align__(16) unsigned long long s_key[kCtaList];
  __shared__ __align__(16) uint32_t s_cnt[kCtaBuckets];
  __shared__ uint32_t s_red[32];
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto finish = [&](uint32_t t, uint2 l, uint2 r) {  // by one thread, after the tile's offsets have been read
    ranges[t] = r;
    // the cost bucket counted by the scan: the whole list, also where the capacity cuts it
    if (sched) work[atomicAdd(&sched[2 + kCostBuckets + cost_bucket(l)], 1u)] = t;
  };
  if (blockIdx.x < big_ctas) {
    const uint32_t listed = (uint32_t)total[kTotalBig];
    const uint32_t items = listed <= big_cap ? listed : ntiles;
    for (uint32_t i = blockIdx.x; i < items; i += big_ctas) {
      const uint32_t t = listed <= big_cap ? big[i] : i;
      const uint2 l = local[t];
      if (l.y - l.x <= (uint32_t)kWarpList) continue;
      const uint2 r = tile_segment(bases, l, t, cap);
      const uint32_t n = r.y - r.x;
      if (n > (uint32_t)kCtaList) cta_sort_long_list(keys + r.x, n, out + r.x, tmp + r.x, s_key, s_cnt, s_red);
      else if (n) cta_sort_list(keys + r.x, n, out + r.x, s_key, s_cnt, s_red);
      __syncthreads();
      if (threadIdx.x == 0) finish(t, l, r);
    }
    return;
  }
  const uint32_t t = (blockIdx.x - big_ctas) * (kSortThreads / 32) + warp;
  if (t >= ntiles) return;
  const uint2 l = local[t];
  __syncwarp();  // lane 0 overwrites it below
  if (l.y - l.x > (uint32_t)kWarpList) return;
  const uint2 r = tile_segment(bases, l, t, cap);
  const uint32_t n = r.y - r.x;
  if (n > 1)
    warp_sort_list(keys + r.x, n, out + r.x, s_key + warp * kWarpList, s_cnt + warp * kWarpBuckets);
  else if (n == 1 && lane == 0)
    out[r.x] = (uint32_t)keys[r.x];
  if (lane == 0) finish(t, l, r);
}

}  // namespace

void launch_tile_order(const uint2* ranges, uint32_t ntiles, uint32_t* sched, uint32_t* work, cudaStream_t s,
                       int* launches) {
  if (ntiles == 0) return;
  const unsigned blocks = (ntiles + 255) / 256;
  launch_pdl(tile_bucket_count_kernel, blocks, 256, 0, s, ranges, ntiles, sched + 2);
  launch_pdl(tile_bucket_scatter_kernel, blocks, 256, 0, s, ranges, ntiles, sched + 2, sched + 2 + kCostBuckets, work);
  *launches += 2;
}

size_t radix_hist_words(uint32_t seg_len, uint32_t nseg) {
  const uint32_t tile = (uint32_t)tile_items(seg_len);
  uint32_t nblocks = (seg_len + tile - 1) / tile;
  return (size_t)kDigits * (nblocks + 1) * nseg;
}

int radix_sort_u32(uint32_t* keys[2], uint32_t* vals[2], uint32_t seg_len, uint32_t nseg, const uint32_t* n_dev,
                   int begin_bit, int end_bit, uint32_t* hist, cudaStream_t s, int* launches) {
  if (tile_items(seg_len) == SortTile<4>::kTile)
    return radix_sort<uint32_t, 4>(keys, vals, seg_len, nseg, n_dev, begin_bit, end_bit, hist, s, launches);
  return radix_sort<uint32_t, 16>(keys, vals, seg_len, nseg, n_dev, begin_bit, end_bit, hist, s, launches);
}



size_t scan_tmp_words(uint32_t n) {
  const uint32_t tile = (uint32_t)(kScanThreads * scan_items(n));
  return (size_t)(n + tile - 1) / tile + 1;
}

cudaError_t launch_scan_counts(const uint32_t* tile_count, const uint32_t* order, uint32_t n, uint32_t* offsets,
                               uint64_t* block_sums, uint64_t* total, cudaStream_t s, int* launches) {
  if (n == 0) {
    cudaError_t e = cudaMemsetAsync(offsets, 0, sizeof(uint32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(total, 0, sizeof(uint64_t), s);
    return e;
  }
  const int items = scan_items(n);
  const uint32_t tile = (uint32_t)(kScanThreads * items);
  const uint32_t nblocks = (n + tile - 1) / tile;
  if (items == 2) launch_pdl(scan_reduce_kernel<2>, nblocks, kScanThreads, 0, s, tile_count, order, n, block_sums);
  else launch_pdl(scan_reduce_kernel<8>, nblocks, kScanThreads, 0, s, tile_count, order, n, block_sums);
  launch_pdl(scan_block_sums_kernel, 1, 1024, 0, s, block_sums, nblocks, total);
  if (items == 2)
    launch_pdl(scan_final_kernel<2>, nblocks, kScanThreads, 0, s, tile_count, order, n, block_sums, offsets);
  else
    launch_pdl(scan_final_kernel<8>, nblocks, kScanThreads, 0, s, tile_count, order, n, block_sums, offsets);
  *launches += 3;
  return cudaSuccess;
}

void launch_tile_ranges(const uint32_t* tiles, const uint32_t* vals, const ViewParams* views, uint32_t n_per_view,
                        uint32_t n_views, uint32_t npairs_cap, const uint32_t* npairs_dev, uint32_t ntiles,
                        uint2* ranges, uint32_t* check, cudaStream_t s) {
  if (npairs_cap == 0) return;
  launch_pdl(tile_ranges_kernel, (npairs_cap + 255) / 256, 256, 0, s, tiles, vals, views, n_per_view, n_views,
             npairs_cap, npairs_dev, ntiles, ranges, check);
}

void launch_compose_keys(const uint2* ranges, uint32_t ntiles, const uint32_t* ids, const float4* rec, uint64_t* keys,
                         cudaStream_t s) {
  if (ntiles == 0) return;
  compose_keys_kernel<<<(ntiles + 7) / 8, 256, 0, s>>>(ranges, ntiles, ids, rec, keys);
}

size_t bin_bases_words(uint64_t ntiles) { return (size_t)((ntiles + kBinBlock - 1) / kBinBlock); }

void launch_tile_scan(uint2* ranges, uint32_t ntiles, uint64_t* bases, uint64_t* total, uint32_t* big, uint32_t big_cap,
                      uint32_t* sched, uint64_t* mirror, cudaStream_t s) {
  launch_pdl(tile_scan_kernel, (ntiles + kBinBlock - 1) / kBinBlock, kBinThreads, 0, s, ranges, ntiles, bases, total, big,
             big_cap, sched, mirror);
}

void launch_tile_sort(uint64_t* keys, uint32_t cap, const uint64_t* bases, uint32_t ntiles, uint2* ranges, uint32_t* out,
                      uint32_t* tmp, const uint32_t* big, uint32_t big_cap, const uint64_t* total, uint32_t* sched, uint32_t* work,
                      int num_sms, cudaStream_t s) {
  constexpr uint32_t kTiles = kSortThreads / 32;
  const uint32_t big_ctas = std::min(ntiles, 4u * (uint32_t)std::max(num_sms, 1));  // one wave
  launch_pdl(tile_sort_kernel, big_ctas + (ntiles + kTiles - 1) / kTiles, kSortThreads, 0, s,
             reinterpret_cast<unsigned long long*>(keys), cap, bases, ntiles, ranges, ranges, out, tmp, big_ctas, big,
             big_cap, total, sched, work);
}

}  // namespace ngs
