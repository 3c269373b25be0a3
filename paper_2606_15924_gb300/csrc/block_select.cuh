// Block-wide exact k-selection shared by the tile selection (Sec. 3.5) and
// the view sampling (Sec. 3.4).
#pragma once
#include "tgs_common.cuh"

namespace tgs {

// Exclusive prefix over threads of v (thread order); total receives the sum.
__device__ __forceinline__ int64_t block_excl_sum(int64_t v, int64_t* s64, int64_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s64[w] = x;
  __syncthreads();
  int64_t t = lane < nw ? s64[lane] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += y;
  }
  const int64_t upto = __shfl_sync(0xffffffffu, t, w > 0 ? w - 1 : 0);  // warps 0 .. w - 1
  total = __shfl_sync(0xffffffffu, t, nw - 1);
  __syncthreads();
  return (w > 0 ? upto : 0) + x - v;
}

constexpr int kSelThreads = 1024;  // threads of a selecting block, and buckets of a pass
constexpr int kSelCand = 64;       // keys of the last bucket that are ordered by counting

struct SelectSmem {
  uint32_t hist[kSelThreads];
  uint32_t lo[32], hi[32];
  int32_t cnt[32];
  uint32_t wsum[32];
  uint64_t ckey[kSelCand];
  int32_t cidx[kSelCand];
  int32_t n_cand;
};

__device__ __forceinline__ uint32_t warp_incl_sum(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Exact block-wide k-selection: of the items in elig (bit j: item t * ITEMS + j
// of thread t, 1024 threads), the k smallest by (full key, index), as the same
// kind of mask.  key[j] is the leading 32 bits of the full key, full(j) all of
// it (MORE: it has 32 more bits; else the same value).
// A pass spreads the keys in play over up to 1024 buckets of equal key width (a
// power of two) between their smallest and largest, one shared-memory count
// each, and finds the bucket that holds the k-th smallest: the keys below it
// are taken, those above are not.  Its own keys are all taken when that many
// are wanted, ordered by counting when there are few (a dozen of some thousand
// well spread keys after the first pass), taken by their low words or in index
// order when they are equal, and else spread again.  Every thread of the block
// must call it (it synchronises); k is the same on all threads.
// Bound by the instructions of one SM and by its chain of barriers and warp
// sums, five barriers for a selection of one pass; a radix selection of 64-bit
// keys by 8-bit digits took two a digit.  The tile selection (three selections
// and the compaction), 256 tiles: 16 -> 7 us; 4056: 19 -> 12; 8160
// tiles: 38 -> 25.
template <int ITEMS, bool MORE, class Full>
__device__ __forceinline__ uint32_t block_select(const uint32_t (&key)[ITEMS], const Full& full_key, uint32_t elig,
                                                 int k, SelectSmem& sm, int64_t* s64) {
  const unsigned full = 0xffffffffu;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  if (k <= 0) return 0u;
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j)
    if ((elig >> j) & 1u) {
      lo = min(lo, key[j]);
      hi = max(hi, key[j]);
    }
  const int mine = __reduce_add_sync(full, __popc(elig));
  lo = __reduce_min_sync(full, lo);
  hi = __reduce_max_sync(full, hi);
  __syncthreads();  // the selection before this one has been read
  if (lane == 0) {
    sm.lo[w] = lo;
    sm.hi[w] = hi;
    sm.cnt[w] = mine;
  }
  sm.hist[t] = 0;
  if (t == 0) sm.n_cand = 0;
  __syncthreads();
  const int n_elig = __reduce_add_sync(full, sm.cnt[lane]);
  if (k >= n_elig) return elig;
  lo = __reduce_min_sync(full, sm.lo[lane]);
  hi = __reduce_max_sync(full, sm.hi[lane]);
  uint32_t in = elig, below = 0u;  // items in [lo, hi], and below lo
  int kk = k;                      // rank (from 1) of the sought key among the items in play
  for (;;) {
    const int sh = max(0, 22 - __clz((int)((hi - lo) | 1u)));
    const uint32_t nb = ((hi - lo) >> sh) + 1u;
    if (nb <= 8u) {  // few buckets (equal ages): counted by ballots, a shared counter would serialise
      uint32_t c = 0;
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const uint32_t d = (in >> j) & 1u ? (key[j] - lo) >> sh : 8u;
        for (uint32_t q = 0; q < nb; ++q) {
          const uint32_t b = __ballot_sync(full, d == q);
          if ((uint32_t)lane == q) c += __popc(b);
        }
      }
      if (c) atomicAdd(&sm.hist[lane], c);
    } else {
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if ((in >> j) & 1u) atomicAdd(&sm.hist[(key[j] - lo) >> sh], 1u);
    }
    __syncthreads();
    const uint32_t ws = __reduce_add_sync(full, sm.hist[t]);
    if (lane == 0) sm.wsum[w] = ws;
    __syncthreads();
    // every warp: the 32 buckets, then the bucket, where the running count reaches kk
    const uint32_t s1 = sm.wsum[lane], i1 = warp_incl_sum(s1);
    const int at1 = __ffs(__ballot_sync(full, i1 >= (uint32_t)kk)) - 1;
    const uint32_t base = __shfl_sync(full, i1 - s1, at1);
    const uint32_t s2 = sm.hist[32 * at1 + lane], i2 = base + warp_incl_sum(s2);
    const int at2 = __ffs(__ballot_sync(full, i2 >= (uint32_t)kk)) - 1;
    const int count = (int)__shfl_sync(full, s2, at2);
    kk -= (int)__shfl_sync(full, i2 - s2, at2);
    lo += (uint32_t)(32 * at1 + at2) << sh;
    const uint32_t width = (1u << sh) - 1u;
    hi = hi - lo > width ? lo + width : hi;
    uint32_t lt = 0u, gt = 0u;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      lt |= (key[j] < lo ? 1u : 0u) << j;
      gt |= (key[j] > hi ? 1u : 0u) << j;
    }
    below |= in & lt;
    in &= ~(lt | gt);
    if (kk == count) return below | in;
    if (count <= kSelCand) {
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if ((in >> j) & 1u) {
          const int p = atomicAdd(&sm.n_cand, 1);
          sm.ckey[p] = full_key(j);
          sm.cidx[p] = t * ITEMS + j;
        }
      __syncthreads();
      for (uint32_t rem = in; rem; rem &= rem - 1u) {
        const int j = __ffs(rem) - 1, i = t * ITEMS + j;
        const uint64_t mk = full_key(j);
        int r = 0;
        for (int q = 0; q < count; ++q) r += sm.ckey[q] < mk || (sm.ckey[q] == mk && sm.cidx[q] < i);
        if (r < kk) below |= 1u << j;
      }
      return below;
    }
    if (sh == 0) break;  // equal leading words
    __syncthreads();
    sm.hist[t] = 0;
    __syncthreads();
  }
  if constexpr (MORE) {
    uint32_t low[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) low[j] = (uint32_t)full_key(j);
    return below | block_select<ITEMS, false>(low, [&](int j) { return full_key(j); }, in, kk, sm, s64);
  } else {
    int64_t all_ties;
    int before = (int)block_excl_sum(__popc(in), s64, all_ties);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if ((in >> j) & 1u) {
        if (before < kk) below |= 1u << j;
        ++before;
      }
    return below;
  }
}

}  // namespace tgs
