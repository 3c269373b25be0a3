// Tile binning: the per-tile Gaussian lists ordered by depth (Sec. 3.1, the
// depth-ordered sets K(p)) as a counting sort on the active-tile rank and a
// sort of (depth | id) keys within each tile:
//   1. blocks take consecutive chunks of Gaussians, count their pairs per
//      active tile in shared memory and reserve their runs in each tile's
//      list with one atomic per tile they touch (a block x tile table of
//      offsets),
//   2. each block scans the tiles' totals (their starts; one launch before it
//      where there are many pairs) and scatters (depth bits << 32 | id) into its
//      runs with shared-memory cursors,
//   3. one block per tile orders its list (k_tile_sort).
// Positive float depths order like their bit patterns, so the result is the
// order (tile, depth, Gaussian id).  With more active tiles than the shared
// counters hold, counts and cursors are global atomics.
#include "scan.cuh"

namespace tgs {

// Most chunks per SM in the count and scatter passes, two blocks of 1024
// threads: more chunks reserve and look up more runs (a chunk and tile each)
// and write shorter ones.
constexpr int kHistBlocksPerSm = 2;
constexpr int kHistChunk = 1536;          // Gaussians per chunk below that (before the rounding to SM waves)
constexpr int kHistMaxRanks = 49152;      // shared-memory table limit (192 KB)

// Chunks of about kHistChunk Gaussians, rounded up to whole waves of the SMs
// (every SM then holds the same number of chunks).
static int hist_blocks(int64_t n) {
  const int64_t c = (n + kHistChunk - 1) / kHistChunk;
  const int64_t sms = std::max(1, device_sm_count());
  return (int)std::max<int64_t>(1, std::min<int64_t>(kHistBlocksPerSm * sms, (c + sms - 1) / sms * sms));
}

struct BinWs {
  int32_t* tile_cnt;   // [R] pairs per rank
  int32_t* tile_fill;  // [R] scatter cursors (global-atomic path)
  int64_t* tile_start; // [R]
  int32_t* table;      // [G * R] offsets of each block's run in each rank's list (shared-memory path)
  uint64_t* keys;      // [C] (depth bits << 32 | id), grouped by tile
  int32_t* inv_rank;   // [R] tile id of each rank
  int64_t* scan_sums;
};

static BinWs carve_bin(void* base, int64_t n, int64_t cap, int32_t n_ranks, size_t* total) {
  Carver c(base);
  BinWs w;
  const size_t R = (size_t)std::max(n_ranks, 1), C = (size_t)std::max<int64_t>(cap, 1);
  const size_t RG = R * (size_t)hist_blocks(n);
  w.tile_cnt = c.take<int32_t>(R);
  w.tile_fill = c.take<int32_t>(R);
  w.tile_start = c.take<int64_t>(R);
  w.table = c.take<int32_t>(RG);
  w.keys = c.take<uint64_t>(C);
  w.inv_rank = c.take<int32_t>(R);
  w.scan_sums = c.take<int64_t>((size_t)std::max(1, scan_blocks((int64_t)R)));
  *total = c.size();
  return w;
}

struct BinGeom {
  int tx, ty;
  int n_ranks;  // ranks >= n_ranks count as inactive
};

// Rank of tile t, from the view's table in global memory (nullptr: the id).
struct RankGlobal {
  static constexpr bool kMasked = false;
  const int32_t* tile_rank;
  int n_ranks;
  __device__ __forceinline__ int operator()(int t) const {
    const int r = tile_rank ? __ldg(tile_rank + t) : t;
    return (r >= 0 && r < n_ranks) ? r : -1;
  }
};
// The same from a copy in shared memory: 16 bits a tile, 0xFFFF for none.  32
// lanes look up 32 tiles, which costs the L1 a tag lookup a line and shared
// memory a few bank conflicts.
struct RankShared {
  static constexpr bool kMasked = false;
  const uint16_t* rank;
  __device__ __forceinline__ int operator()(int t) const {
    const uint32_t r = rank[t];
    return r == 0xFFFFu ? -1 : (int)r;
  }
};
// The same with a bit per tile, set where it has a rank.
struct RankMasked {
  static constexpr bool kMasked = true;
  const uint16_t* rank;
  const uint32_t* bits;  // one word past the last tile's
  __device__ __forceinline__ int operator()(int t) const {
    const uint32_t r = rank[t];
    return r == 0xFFFFu ? -1 : (int)r;
  }
  __device__ __forceinline__ uint32_t row(int t, int w) const {  // tiles t .. t + w - 1, w <= 32
    return __funnelshift_r(bits[t >> 5], bits[(t >> 5) + 1], t & 31) & (0xffffffffu >> (32 - w));
  }
};

// Calls f(rank, Gaussian, depth bits) for every (Gaussian, active tile) pair of
// the block's Gaussians [i0, i1).  A lane walks its Gaussian's rectangle by
// itself, a dozen instructions a tile; rectangles of more than kLaneTiles
// tiles are walked by the whole warp, so that a few large splats do not leave
// the other lanes idle.  (Numbering the pairs of a warp's Gaussians by a prefix
// and dealing them out evenly takes a binary search and a division a pair.)
// With the ranks looked up in shared memory: count 14.5 -> 10.1 and scatter
// 17.2 -> 12.2 us at 500k Gaussians and 720 tiles, 71 -> 27 and 163 -> 109 at 1M
// and every tile of 1957x1091.
// Where only some tiles are active (RankMasked) the lane first gathers the
// active tiles of its rectangle as one word, a row of the bit table at a time,
// and takes only those, count and scatter: 720 of 3600 tiles, 500k Gaussians
// 10.1 -> 9.0 and 12.2 -> 10.1 us; 1340 of 6700, 2M 34.5 -> 24.7 and 41.0 -> 36.6;
// eight views of 3M with 15 to 55 % of the tiles 494 -> 359 and 776 -> 677.
constexpr int kLaneTiles = 16;
constexpr int kLaneTilesMasked = 32;  // bits of a word

template <bool DEPTH, typename Rank, typename F>
__device__ __forceinline__ void for_each_pair(const float2* __restrict__ xy, const int32_t* __restrict__ radius,
                                              const float* __restrict__ depth, int64_t i0, int64_t i1,
                                              const BinGeom& geo, const Rank rank_of, F f) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  for (int64_t base = i0 + (threadIdx.x & ~31); base < i1; base += blockDim.x) {
    const int64_t pos = base + lane;
    const uint32_t id = (uint32_t)pos;
    int x0 = 0, x1 = 0, y0 = 0, y1 = 0;
    uint32_t d = 0;
    const int r = pos < i1 ? radius[pos] : 0;
    if (r > 0) {
      const float2 p = xy[pos];
      if (DEPTH) d = __float_as_uint(depth[pos]);
      tile_span(p.x, r, geo.tx, x0, x1);
      tile_span(p.y, r, geo.ty, y0, y1);
    }
    const int w = x1 - x0, area = w * (y1 - y0);
    constexpr int kLane = Rank::kMasked ? kLaneTilesMasked : kLaneTiles;
    if constexpr (Rank::kMasked) {
      const int t0 = y0 * geo.tx + x0;
      uint32_t on = 0u;
      if (area <= kLane)
        for (int t = t0, b = 0; b < area; t += geo.tx, b += w) on |= rank_of.row(t, w) << b;
      const uint32_t inv = w > 0 ? 65536u / (uint32_t)w + 1u : 0u;  // b / w = b inv >> 16 for b < 32
      for (; on; on &= on - 1u) {
        const int b = __ffs(on) - 1, y = (int)(((uint32_t)b * inv) >> 16);
        f((int)rank_of.rank[t0 + b + y * (geo.tx - w)], id, d);
      }
    } else {
      int t = y0 * geo.tx + x0, row_end = t + w;
      for (int left = area <= kLane ? area : 0; left > 0; --left) {
        const int k = rank_of(t);
        if (k >= 0) f(k, id, d);
        if (++t == row_end) {
          t += geo.tx - w;
          row_end = t + w;
        }
      }
    }
    __syncwarp();
    for (unsigned big = __ballot_sync(full, area > kLane); big; big &= big - 1) {
      const int src = __ffs(big) - 1;
      const int o_area = __shfl_sync(full, area, src), o_w = __shfl_sync(full, w, src);
      const int o_t = __shfl_sync(full, y0 * geo.tx + x0, src);
      const uint32_t o_id = __shfl_sync(full, id, src), o_d = DEPTH ? __shfl_sync(full, d, src) : 0u;
      for (int q = lane; q < o_area; q += 32) {
        const int ty = q / o_w;
        const int k = rank_of(o_t + ty * geo.tx + (q - ty * o_w));
        if (k >= 0) f(k, o_id, o_d);
      }
      __syncwarp();
    }
  }
}

// 1''. pairs per active tile with global atomics, 256 Gaussians per block.
__global__ void __launch_bounds__(256) k_count_pairs(const float2* __restrict__ xy,
                                                     const int32_t* __restrict__ radius, int64_t n, BinGeom geo,
                                                     const int32_t* __restrict__ tile_rank,
                                                     int32_t* __restrict__ tile_cnt) {
  const int64_t i0 = (int64_t)blockIdx.x * 256, i1 = min(n, i0 + 256);
  for_each_pair<false>(xy, radius, nullptr, i0, i1, geo, RankGlobal{tile_rank, geo.n_ranks},
                       [&](int k, uint32_t, uint32_t) { atomicAdd(tile_cnt + k, 1); });
}

// 3''. scatter with global cursors (order inside a tile arbitrary: the
// per-tile sort that follows orders it).
__global__ void __launch_bounds__(256) k_scatter_pairs(const float2* __restrict__ xy,
                                                       const int32_t* __restrict__ radius,
                                                       const float* __restrict__ depth, int64_t n, BinGeom geo,
                                                       const int32_t* __restrict__ tile_rank,
                                                       const int64_t* __restrict__ tile_start,
                                                       int32_t* __restrict__ tile_fill, uint64_t* __restrict__ keys,
                                                       int64_t cap) {
  const int64_t i0 = (int64_t)blockIdx.x * 256, i1 = min(n, i0 + 256);
  for_each_pair<true>(xy, radius, depth, i0, i1, geo, RankGlobal{tile_rank, geo.n_ranks},
                      [&](int k, uint32_t i, uint32_t d) {
    const int64_t pos = tile_start[k] + atomicAdd(tile_fill + k, 1);
    if (pos < cap) keys[pos] = ((uint64_t)d << 32) | (uint64_t)i;
  });
}

// 1. shared-memory path: block b counts the pairs of its chunk of Gaussians
// per rank and reserves its run in each rank's list (table[b * R + r] = the
// run's offset in the list; blocks land in any order, the lists are sorted
// whole).
constexpr int kHistThreads = 1024;
constexpr size_t kHistStaticSmem = 1024;  // at least the kernels' statically allocated shared memory

__device__ __forceinline__ void chunk_of(int64_t n, int64_t& i0, int64_t& i1) {
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  i0 = (int64_t)blockIdx.x * chunk;
  i1 = min(n, i0 + chunk);
}

// The view's ranks as 16-bit values in shared memory (at p), and behind them a
// bit per tile (MASKED; whole blocks call it).
enum { kRankGlobal = 0, kRankShared = 1, kRankMasked = 2 };
__host__ __device__ inline size_t rank_smem(int kind, int tiles) {
  const size_t words = ((size_t)tiles + 1) / 2;
  return kind == kRankGlobal ? 0 : 4 * (words + (kind == kRankMasked ? (size_t)(tiles + 31) / 32 + 1 : 0));
}
template <bool MASKED>
__device__ __forceinline__ RankMasked stage_ranks(uint32_t* p, const int32_t* __restrict__ tile_rank,
                                                  const BinGeom& geo) {
  uint16_t* out = reinterpret_cast<uint16_t*>(p);
  const int T = geo.tx * geo.ty;
  uint32_t* bits = p + (T + 1) / 2;
  for (int t0 = threadIdx.x & ~31; t0 < T; t0 += blockDim.x) {
    const int t = t0 + (threadIdx.x & 31);
    const int r = t < T ? tile_rank[t] : -1;
    const bool in = r >= 0 && r < geo.n_ranks;
    if (t < T) out[t] = in ? (uint16_t)r : (uint16_t)0xFFFFu;
    if (MASKED) {
      const uint32_t b = __ballot_sync(0xffffffffu, in);
      if ((threadIdx.x & 31) == 0) bits[t0 >> 5] = b;
    }
  }
  if (MASKED && threadIdx.x == 0) bits[(T + 31) / 32] = 0u;
  return RankMasked{out, bits};
}

// Walks the block's chunk with ranks of the given kind (staged at p).
template <int KIND, bool DEPTH, typename F>
__device__ __forceinline__ void walk_chunk(const float2* __restrict__ xy, const int32_t* __restrict__ radius,
                                           const float* __restrict__ depth, int64_t n, const BinGeom& geo,
                                           const int32_t* __restrict__ tile_rank, const RankMasked& staged, F f) {
  int64_t i0, i1;
  chunk_of(n, i0, i1);
  if constexpr (KIND == kRankMasked) for_each_pair<DEPTH>(xy, radius, depth, i0, i1, geo, staged, f);
  else if constexpr (KIND == kRankShared)
    for_each_pair<DEPTH>(xy, radius, depth, i0, i1, geo, RankShared{staged.rank}, f);
  else for_each_pair<DEPTH>(xy, radius, depth, i0, i1, geo, RankGlobal{tile_rank, geo.n_ranks}, f);
}

template <int KIND>
__global__ void __launch_bounds__(kHistThreads) k_hist_count(const float2* __restrict__ xy,
                                                             const int32_t* __restrict__ radius, int64_t n,
                                                             BinGeom geo, const int32_t* __restrict__ tile_rank,
                                                             int32_t* __restrict__ table,
                                                             int32_t* __restrict__ rank_cnt) {
  extern __shared__ uint32_t sh[];
  const int R = geo.n_ranks;
  for (int r = threadIdx.x; r < R; r += blockDim.x) sh[r] = 0;
  RankMasked staged{};
  if constexpr (KIND != kRankGlobal) staged = stage_ranks<KIND == kRankMasked>(sh + R, tile_rank, geo);
  __syncthreads();
  walk_chunk<KIND, false>(xy, radius, nullptr, n, geo, tile_rank, staged,
                          [&](int k, uint32_t, uint32_t) { atomicAdd(sh + k, 1u); });
  __syncthreads();
  int32_t* row = table + (size_t)blockIdx.x * R;
  for (int r = threadIdx.x; r < R; r += blockDim.x)
    if (sh[r]) row[r] = atomicAdd(rank_cnt + r, (int32_t)sh[r]);
}

// 2'. shared-memory path, many pairs: the ranks' starts and the pairs' total,
// once, and the keys' places overwritten with whole lines before the scatter.
// The scatter writes 8 bytes here and there; a first write to a part of a
// 32-byte sector that the L2 does not hold fetches the sector from memory, so
// with the keys of the last call long evicted the scatter waited for a read of
// the whole array: 6.7M pairs, 8487 tiles: 92 us, 49 where the lines are in the
// L2.
// Taken from kStartsPairs of capacity (48 MB of keys).  Scatter alone, and with
// this launch before it: 720 tiles of 500k Gaussians 12 us, 14; 1340 tiles of 2M
// 41, 45; every tile of 500k 26, 25; every tile of 1M at 1957x1091 109, 73; eight
// views of 3M (4 to 15M pairs each) 1072, 881.
constexpr int kStartThreads = 1024;
constexpr int64_t kStartsPairs = 6ll << 20;

__global__ void __launch_bounds__(kStartThreads) k_hist_starts(const int32_t* __restrict__ rank_cnt, int R,
                                                               int64_t* __restrict__ rank_start,
                                                               int64_t* __restrict__ n_total,
                                                               uint64_t* __restrict__ keys, int64_t cap) {
  __shared__ int64_t s_wt[32];
  int64_t total;
  if (blockIdx.x == 0) {
    const int per = (R + (int)blockDim.x - 1) / (int)blockDim.x;
    const int r0 = min(R, (int)threadIdx.x * per), r1 = min(R, r0 + per);
    int64_t run = 0;
    for (int r = r0; r < r1; ++r) run += rank_cnt[r];
    int64_t pre = block_exclusive_scan<int64_t>(run, s_wt, total);
    for (int r = r0; r < r1; ++r) {
      rank_start[r] = pre;
      pre += rank_cnt[r];
    }
    if (threadIdx.x == 0) *n_total = total;
  } else {
    int64_t run = 0;
    for (int r = threadIdx.x; r < R; r += blockDim.x) run += rank_cnt[r];
    block_exclusive_scan<int64_t>(run, s_wt, total);
  }
  const int64_t m = min(total, cap);
  uint4* k2 = reinterpret_cast<uint4*>(keys);
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < m / 2; p += (int64_t)gridDim.x * blockDim.x)
    k2[p] = make_uint4(0u, 0u, 0u, 0u);
  if ((m & 1) && blockIdx.x == 0 && threadIdx.x == 0) keys[m - 1] = 0;
}

// 2. shared-memory path: scatters with shared cursors that start at the block's
// runs (clamped to the capacity; positions at or past it are dropped).  The
// ranks' starts come from k_hist_starts (STARTS), or the block takes the
// exclusive prefix of the ranks' totals itself (R values, from L2) instead of a
// launch of its own (block 0 writes them to rank_start and their sum to n_total
// for what follows).  Entries of ranks that the block has no pair in are not
// used as positions.
template <int KIND, bool STARTS>
__global__ void __launch_bounds__(kHistThreads) k_hist_scatter(const float2* __restrict__ xy,
                                                               const int32_t* __restrict__ radius,
                                                               const float* __restrict__ depth, int64_t n,
                                                               BinGeom geo, const int32_t* __restrict__ tile_rank,
                                                               const int32_t* __restrict__ table,
                                                               int64_t* __restrict__ rank_start,
                                                               const int32_t* __restrict__ rank_cnt,
                                                               int64_t* __restrict__ n_total,
                                                               uint64_t* __restrict__ keys, int64_t cap) {
  extern __shared__ uint32_t sh[];
  __shared__ int64_t s_wt[32];
  static_assert(sizeof(s_wt) <= kHistStaticSmem, "shared memory asked for");
  const int R = geo.n_ranks, b = blockIdx.x;
  const int32_t* row = table + (size_t)b * R;
  if (STARTS) {
    for (int r = threadIdx.x; r < R; r += blockDim.x) sh[r] = (uint32_t)min(row[r] + rank_start[r], cap);
  } else {
    // thread t scans the contiguous run [t * per, (t + 1) * per) of the totals
    const int per = (R + (int)blockDim.x - 1) / (int)blockDim.x;
    const int r0 = (int)threadIdx.x * per, r1 = min(R, r0 + per);
    int64_t run = 0;
    for (int r = r0; r < r1; ++r) run += rank_cnt[r];
    int64_t total;
    int64_t pre = block_exclusive_scan<int64_t>(run, s_wt, total);
    for (int r = r0; r < r1; ++r) {
      const int64_t c = rank_cnt[r];
      if (b == 0) rank_start[r] = pre;
      sh[r] = (uint32_t)min(row[r] + pre, cap);
      pre += c;
    }
    if (b == 0 && threadIdx.x == 0) *n_total = total;
  }
  RankMasked staged{};
  if constexpr (KIND != kRankGlobal) staged = stage_ranks<KIND == kRankMasked>(sh + R, tile_rank, geo);
  __syncthreads();
  walk_chunk<KIND, true>(xy, radius, depth, n, geo, tile_rank, staged, [&](int k, uint32_t i, uint32_t d) {
    const uint32_t pos = atomicAdd(sh + k, 1u);
    if ((int64_t)pos < cap) keys[pos] = ((uint64_t)d << 32) | (uint64_t)i;
  });
}

// ---------------------------------------------------------------------------
// 4. one block per active rank: its keys in order, ids (and full keys) out.
//
// A list of up to CAP = T E keys is spread over buckets of equal key width (a
// power of two) between its smallest and largest key, in shared memory (one
// histogram, one scan, one scatter); each key then finds its place by counting
// the smaller keys of its bucket, about one on average.  A bucket of more than
// kRankMax keys (depths crowded in a small part of the range) is spread again
// over its own range, and so on: keys are distinct, so a range always splits.
// That is a few dozen instructions a key, where a bitonic network over the
// list takes log^2 n compare-exchanges of 64-bit keys.  1340 tiles of 2M
// Gaussians: 339 us with the network, 57 here; every tile of 1M Gaussians at
// 1957x1091: 182, 98; 720 tiles of 500k Gaussians: 21, 10.  Lists of thousands
// (eight views of 3M Gaussians, up to 8200 keys a tile) needed the Gaussians
// sorted by depth first and then every chunk's segment of every list: 3.1 ms of
// radix passes, table scans and segment sorts, 0.72 ms here.
//
// Longer lists are taken in runs of consecutive keys that fit: a histogram of
// the keys not yet out gives the next run's upper bound, and the run is
// gathered from the list and sorted as above.
// ---------------------------------------------------------------------------
constexpr int kRankMax = 48;     // longest bucket ordered by counting
constexpr int kSortBins = 2048;  // buckets of a pass

// Range of rank r: its start and count of pairs.
struct RangeSrc {
  const int64_t* start;
  const int32_t* cnt;
  __device__ __forceinline__ void get(int r, int64_t& s0, int64_t& e0) const {
    s0 = start[r];
    e0 = s0 + cnt[r];
  }
};

template <int T, int E>
struct __align__(16) SortSmem {
  uint64_t key[T * E];
  uint32_t fill[kSortBins];  // a bucket's count, then its next free place
  uint64_t red[2][32];
  uint32_t wt[32];
  int2 seg[T * E / kRankMax + 2];  // (first place, keys) of the buckets to spread again
  int n_seg;
  int cursor;
};

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t y = __shfl_xor_sync(0xffffffffu, v, o);
    v = y < v ? y : v;
  }
  return v;
}

// Block-wide minimum of lo and maximum of hi.
template <int T, int E>
__device__ __forceinline__ void block_min_max(uint64_t& lo, uint64_t& hi, SortSmem<T, E>& S) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  lo = warp_min_u64(lo);
  hi = ~warp_min_u64(~hi);
  if (lane == 0) {
    S.red[0][w] = lo;
    S.red[1][w] = hi;
  }
  __syncthreads();
  lo = lane < T / 32 ? S.red[0][lane] : ~0ull;
  hi = lane < T / 32 ? S.red[1][lane] : 0ull;
  lo = warp_min_u64(lo);
  hi = ~warp_min_u64(~hi);
}

// Bucket width (a shift) that spreads [0, span] over at most `bins` buckets.
__device__ __forceinline__ int bucket_shift(uint64_t span, int bins) {
  const int top = 64 - __clzll(span | 1ull), b = 31 - __clz(bins);
  return max(0, top - b);
}

// Exclusive prefix of S.fill[0 .. bins - 1] in place (all threads; bins a
// multiple of T or at most T), `base` added.
template <int T, int E>
__device__ __forceinline__ void scan_buckets(SortSmem<T, E>& S, int bins, uint32_t base) {
  constexpr int P = kSortBins / T;
  const int per = max(1, bins / T);
  const int b0 = threadIdx.x * per;
  uint32_t v[P], sum = 0;
#pragma unroll
  for (int k = 0; k < P; ++k) {
    v[k] = k < per && b0 + k < bins ? S.fill[b0 + k] : 0u;
    sum += v[k];
  }
  uint32_t total;
  uint32_t run = base + block_exclusive_scan<uint32_t>(sum, S.wt, total);
#pragma unroll
  for (int k = 0; k < P; ++k)
    if (k < per && b0 + k < bins) {
      S.fill[b0 + k] = run;
      run += v[k];
    }
  __syncthreads();
}

// Orders n keys (n <= T E) from `src` (global memory, or nullptr: S.key
// itself) and hands key number p to emit(p, key).
template <int T, int E, class Emit>
__device__ __forceinline__ void sort_run(SortSmem<T, E>& S, const uint64_t* __restrict__ src, int n, Emit emit) {
  const int t = threadIdx.x;
  if (t == 0) {
    S.seg[0] = make_int2(0, n);
    S.n_seg = 1;
  }
  const uint64_t* from = src ? src : S.key;
  for (;;) {
    __syncthreads();
    const int q = S.n_seg - 1;
    if (q < 0) break;
    const int2 g = S.seg[q];
    __syncthreads();
    if (t == 0) S.n_seg = q;  // the last in is the first out: the waiting buckets are disjoint
    uint64_t k[E];
    uint64_t lo = ~0ull, hi = 0ull;
#pragma unroll
    for (int r = 0; r < E; ++r) {
      if (r * T >= g.y) break;
      const int i = r * T + t;
      k[r] = i < g.y ? from[i] : 0ull;
      if (i < g.y) {
        lo = k[r] < lo ? k[r] : lo;
        hi = k[r] > hi ? k[r] : hi;
      }
    }
    int bins = 256;
    while (bins < g.y && bins < kSortBins) bins *= 2;
    for (int b = t; b < bins; b += T) S.fill[b] = 0;
    block_min_max<T, E>(lo, hi, S);  // its barrier also ends the reads of S.key and the clearing
    const int sh = bucket_shift(hi - lo, bins);
#pragma unroll
    for (int r = 0; r < E; ++r) {
      if (r * T >= g.y) break;
      if (r * T + t < g.y) atomicAdd(&S.fill[(uint32_t)((k[r] - lo) >> sh)], 1u);
    }
    __syncthreads();
    scan_buckets<T, E>(S, bins, (uint32_t)g.x);
#pragma unroll
    for (int r = 0; r < E; ++r) {
      if (r * T >= g.y) break;
      if (r * T + t < g.y) S.key[atomicAdd(&S.fill[(uint32_t)((k[r] - lo) >> sh)], 1u)] = k[r];
    }
    __syncthreads();
    // neighbours in S.key share their bucket, so a warp's counting loops stay together
    for (int i = g.x + t; i < g.x + g.y; i += T) {
      const uint64_t key = S.key[i];
      const uint32_t b = (uint32_t)((key - lo) >> sh);
      const int b0 = b ? S.fill[b - 1] : g.x, b1 = S.fill[b];  // filled: a bucket ends where the next begins
      if (b1 - b0 > kRankMax && b1 - b0 < g.y) {
        if (i == b0) S.seg[atomicAdd(&S.n_seg, 1)] = make_int2(b0, b1 - b0);
        continue;
      }
      int p = b0;
      for (int m = b0; m < b1; ++m) p += S.key[m] < key;
      emit(p, key);
    }
    __syncthreads();
    if (S.n_seg > 0) from = S.key + S.seg[S.n_seg - 1].x;
  }
}

// 64 registers at 256 threads (four blocks an SM), 40 at 512 (three): the
// sort waits on shared memory and barriers, so it wants warps.  Sixteen keys a
// thread then spill, 8 bytes at 256 threads and 268 at 512.
template <int T, int E>
__global__ void __launch_bounds__(T, T == 512 ? 3 : 4) k_tile_sort(const uint64_t* __restrict__ keys, RangeSrc src,
                                                 const int32_t* __restrict__ inv_rank, int64_t cap,
                                                 int32_t* __restrict__ vals, uint64_t* __restrict__ full_keys,
                                                 int2* __restrict__ ranges) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem<T, E>& S = *reinterpret_cast<SortSmem<T, E>*>(smem_raw);
  constexpr int CAP = T * E;
  const int r = blockIdx.x, t = threadIdx.x;
  int64_t s0, e0;
  src.get(r, s0, e0);
  const int64_t s = min(s0, cap), e = min(e0, cap);  // pairs past the capacity are dropped
  if (t == 0) ranges[r] = make_int2((int)s, (int)e);
  const int n = (int)(e - s);
  if (n <= 0) return;
  const uint64_t tile_hi = full_keys ? ((uint64_t)(uint32_t)inv_rank[r] << 32) : 0;
  const uint64_t* K = keys + s;
  auto put = [&](int64_t pos, uint64_t k) {
    vals[pos] = (int32_t)(uint32_t)k;
    if (full_keys) full_keys[pos] = tile_hi | (k >> 32);
  };
  if (n <= CAP) {
    sort_run<T, E>(S, K, n, [&](int p, uint64_t k) { put(s + p, k); });
    return;
  }
  uint64_t first = ~0ull, top = 0ull;
  for (int i = t; i < n; i += T) {
    const uint64_t k = K[i];
    first = k < first ? k : first;
    top = k > top ? k : top;
  }
  block_min_max<T, E>(first, top, S);
  for (int out = 0; out < n;) {  // keys >= first are not yet out: n - out of them
    uint64_t bound = top;        // the run: keys in [first, bound]
    int run = n - out;
    while (run > CAP) {
      // narrow [first, bound] until its leading buckets make a run that fits
      const int sh = bucket_shift(bound - first, kSortBins);
      __syncthreads();
      for (int b = t; b < kSortBins; b += T) S.fill[b] = 0;
      __syncthreads();
      for (int i = t; i < n; i += T) {
        const uint64_t k = K[i];
        if (k >= first && k <= bound) atomicAdd(&S.fill[(uint32_t)((k - first) >> sh)], 1u);
      }
      __syncthreads();
      scan_buckets<T, E>(S, kSortBins, 0u);
      if (t == 0) {  // the most leading buckets with at most CAP keys: fill[b] counts those before b
        int lo = 0, hi = kSortBins - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) / 2;
          if (S.fill[mid] <= (uint32_t)CAP) lo = mid;
          else hi = mid - 1;
        }
        S.cursor = lo;
      }
      __syncthreads();
      const int b = S.cursor;
      const int before = (int)S.fill[b];
      if (before > 0) {
        bound = first + ((uint64_t)b << sh) - 1;
        run = before;
      } else {  // all before bucket b are empty and it alone is too long: look into it
        first += (uint64_t)b << sh;
        const uint64_t last = first + ((1ull << sh) - 1);
        bound = last < bound ? last : bound;
      }
      __syncthreads();
    }
    if (t == 0) S.cursor = 0;
    __syncthreads();
    for (int i = t; i < n; i += T) {
      const uint64_t k = K[i];
      if (k >= first && k <= bound) S.key[atomicAdd(&S.cursor, 1)] = k;
    }
    __syncthreads();
    sort_run<T, E>(S, nullptr, run, [&](int p, uint64_t k) { put(s + out + p, k); });
    out += run;
    first = bound + 1;
  }
}

__global__ void k_inv_rank(const int32_t* __restrict__ tile_rank, int T, int32_t* __restrict__ inv, int n_max) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  const int r = tile_rank ? tile_rank[t] : t;
  if (r >= 0 && r < n_max) inv[r] = t;
}

}  // namespace tgs

using namespace tgs;

template <int T, int E>
static void launch_tile_sort(int R, const BinWs& w, const RangeSrc& src, int64_t cap, int32_t* vals, uint64_t* keys,
                             int2* ranges, cudaStream_t s) {
  constexpr int smem = (int)sizeof(SortSmem<T, E>);
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (smem > 48 * 1024 && (dev < 0 || dev >= 64 || !attr[dev])) {
    cudaFuncSetAttribute(k_tile_sort<T, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  k_tile_sort<T, E><<<R, T, smem, s>>>(w.keys, src, w.inv_rank, cap, vals, keys, ranges);
}

extern "C" size_t tgs_bin_tiles_workspace_size(int64_t n, int64_t capacity, int32_t n_active_max) {
  size_t total = 0;
  carve_bin(nullptr, n, capacity, n_active_max, &total);
  return total;
}

extern "C" tgs_status tgs_bin_tiles(const tgs_projected* proj, int64_t n, const tgs_camera* cam,
                                    const int32_t* tile_rank, int32_t n_active_max, void* workspace,
                                    size_t workspace_bytes, int64_t capacity, int32_t* vals, uint64_t* keys,
                                    int32_t* tile_ranges, int64_t* n_isect, tgs_stream stream) {
  if (!proj || !cam || n < 0 || capacity < 0 || capacity >= (int64_t)INT32_MAX || n >= (int64_t)INT32_MAX ||
      cam->width <= 0 || cam->height <= 0 || !n_isect || !tile_ranges || n_active_max < 0)
    return TGS_ERR_INVALID_ARG;
  const int T = tiles_x(cam->width) * tiles_y(cam->height);
  if (!tile_rank && n_active_max < T) return TGS_ERR_INVALID_ARG;
  if (n > 0 && (!proj->xy || !proj->radius || !proj->depth || !aligned8(proj->xy))) return TGS_ERR_INVALID_ARG;
  if (capacity > 0 && !vals) return TGS_ERR_INVALID_ARG;
  if (!aligned8(tile_ranges) || (keys && !aligned8(keys))) return TGS_ERR_INVALID_ARG;
  size_t need = tgs_bin_tiles_workspace_size(n, capacity, n_active_max);
  if (!workspace || workspace_bytes < need) return TGS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  size_t tot;
  BinWs w = carve_bin(workspace, n, capacity, n_active_max, &tot);
  BinGeom geo{tiles_x(cam->width), tiles_y(cam->height), n_active_max};
  const int R = n_active_max;
  // the scan writes n_isect and the per-rank sort writes every range; they
  // are cleared here only where those kernels do not run
  if (n == 0 || R == 0) {
    if (R > 0) cudaMemsetAsync(tile_ranges, 0, sizeof(int2) * (size_t)R, s);
    cudaMemsetAsync(n_isect, 0, sizeof(int64_t), s);
    return check_launch();
  }
  const float2* xy = reinterpret_cast<const float2*>(proj->xy);
  const RangeSrc src{w.tile_start, w.tile_cnt};
  // Per-chunk histograms in shared memory and an offset table, while the
  // ranks fit in shared memory: global per-tile counters and cursors take
  // every pair's atomic on a few hundred addresses, several times slower.
  const bool shared_path = R <= kHistMaxRanks;
  const int G = hist_blocks(n);
  // the view's rank table beside the counters, where both fit twice on an SM;
  // with a bit table where some tile is inactive (with every tile active its
  // rows save nothing: 500k Gaussians 11.5 and 26.9 us without, 12.5 and 28.4)
  const size_t counters = sizeof(int32_t) * (size_t)R;
  int kind = tile_rank ? (R < T ? kRankMasked : kRankShared) : kRankGlobal;
  if (counters + rank_smem(kind, T) > 100 * 1024) kind = kRankGlobal;  // R < 0xFFFF
  // nor where a block stages a large table for a few Gaussians: 14 a block, 14400
  // tiles 31.9 us staged, 29.8 not; 34560 tiles 50.3, 42.1, and 74.9, 64.6 with a fifth
  // of them active; but 8160 tiles 23.7, 25.7, and 53 a block and 34560 tiles 57.5, 64.6
  if (T > 8192 && T > 1000 * ((n + G - 1) / G)) kind = kRankGlobal;
  const size_t smem = counters + rank_smem(kind, T);
  cudaMemsetAsync(w.tile_cnt, 0, sizeof(int32_t) * (size_t)R, s);
  if (shared_path) {
    // opt in to more than 48 KB of shared memory a block (per device); the
    // scatter's own arrays count too
    if (smem + kHistStaticSmem > 48 * 1024) {
      static bool attr_set[64] = {};
      int dev = 0;
      cudaGetDevice(&dev);
      if (dev < 0 || dev >= 64) return TGS_ERR_DEVICE;
      if (!attr_set[dev]) {
        for (auto f : {k_hist_count<0>, k_hist_count<1>, k_hist_count<2>})
          cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistMaxRanks * 4);
        for (auto f : {k_hist_scatter<0, false>, k_hist_scatter<0, true>, k_hist_scatter<1, false>,
                       k_hist_scatter<1, true>, k_hist_scatter<2, false>, k_hist_scatter<2, true>})
          cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistMaxRanks * 4);
        attr_set[dev] = true;
      }
    }
    auto count = kind == kRankMasked ? k_hist_count<2> : kind == kRankShared ? k_hist_count<1> : k_hist_count<0>;
    count<<<G, kHistThreads, smem, s>>>(xy, proj->radius, n, geo, tile_rank, w.table, w.tile_cnt);
  } else {
    cudaMemsetAsync(w.tile_fill, 0, sizeof(int32_t) * (size_t)R, s);
    k_count_pairs<<<(int)((n + 255) / 256), 256, 0, s>>>(xy, proj->radius, n, geo, tile_rank, w.tile_cnt);
  }
  if (!shared_path || capacity == 0) {  // else the scatter scans the totals itself
    const int32_t* cnt = w.tile_cnt;
    int64_t* start = w.tile_start;
    auto load = [=] __device__(int64_t r) -> int64_t { return cnt[r]; };
    auto store = [=] __device__(int64_t r, int64_t pre, int64_t) { start[r] = pre; };
    exclusive_scan<int64_t>(load, store, nullptr, R, w.scan_sums, n_isect, s);
  }
  if (capacity == 0) {
    cudaMemsetAsync(tile_ranges, 0, sizeof(int2) * (size_t)R, s);
    return check_launch();
  }
  if (shared_path) {
    // it writes the keys 16 bytes at a time; a workspace is taken from any 8-byte boundary
    const bool starts = capacity >= kStartsPairs && aligned16(w.keys);
    if (starts)
      k_hist_starts<<<2 * std::max(1, device_sm_count()), kStartThreads, 0, s>>>(w.tile_cnt, R, w.tile_start, n_isect,
                                                                                 w.keys, capacity);
    auto scatter = kind == kRankMasked   ? (starts ? k_hist_scatter<2, true> : k_hist_scatter<2, false>)
                   : kind == kRankShared ? (starts ? k_hist_scatter<1, true> : k_hist_scatter<1, false>)
                                         : (starts ? k_hist_scatter<0, true> : k_hist_scatter<0, false>);
    scatter<<<G, kHistThreads, smem, s>>>(xy, proj->radius, proj->depth, n, geo, tile_rank, w.table, w.tile_start,
                                          w.tile_cnt, n_isect, w.keys, capacity);
  } else {
    k_scatter_pairs<<<(int)((n + 255) / 256), 256, 0, s>>>(xy, proj->radius, proj->depth, n, geo, tile_rank,
                                                           w.tile_start, w.tile_fill, w.keys, capacity);
  }
  if (keys) k_inv_rank<<<(T + 255) / 256, 256, 0, s>>>(tile_rank, T, w.inv_rank, R);
  // The sort's block by the lists' mean length, as far as the capacity tells it:
  // lists past its CAP are sorted in several runs, and a larger block leaves
  // fewer of them on an SM.  A training view's capacity is sized from the pairs of
  // all tiles.  The differentiable render's is sized from those of its active
  // tiles only, so there the mean comes out too small by the share of the tiles that
  // are active (1340 of 6700 tiles of 2M Gaussians: 453 for lists of 2270, most of
  // which then take two or three runs).
  const int64_t mean = capacity / T;
  int2* rg = reinterpret_cast<int2*>(tile_ranges);
  if (mean <= 512) launch_tile_sort<256, 8>(R, w, src, capacity, vals, keys, rg, s);
  else if (mean <= 2048) launch_tile_sort<256, 16>(R, w, src, capacity, vals, keys, rg, s);
  else launch_tile_sort<512, 16>(R, w, src, capacity, vals, keys, rg, s);
  return check_launch();
}
