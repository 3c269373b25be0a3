// Tile selection and tile-wise error-guided pixel sampling (Sec. 3.5).
//
// Both levels choose n items as: round(r_hard n) by the error-proportional
// draw without replacement, round(r_stable n) of the rest with the largest age,
// the remainder uniformly.  The weighted draw is realised as the
// Efraimidis-Spirakis order (ascending E_i / w_i with E_i = -log2 U_i an
// exponential clock in 32-bit fixed point), so every item's fate is decided
// by counting the items that precede it in a total order - no sequential
// loop.  The keys are exact (integers, and correctly rounded quotients of them),
// hence bit-identical on every run; the pixel draw orders by fp32 quotients first,
// and by the exact keys wherever the bounds on their error leave a choice open.
#include "block_select.cuh"
#include "scan.cuh"

namespace tgs {

struct SelWs {
  uint64_t* tile_w;   // [T] sum of pixel weights
  uint64_t* tile_key; // [T] hard key: bits of the double L / w (exponential clock over weight)
  uint64_t* tile_u;   // [T] uniform key
  uint32_t* tile_age; // [T] smallest pixel age
  int32_t* rank_h;    // [T]
  int32_t* rank_s;    // [T]
  int32_t* rank_u;    // [T]
  int64_t* scan_sums;
  int64_t* total;     // [1]
};

static SelWs carve_sel(void* base, int T, size_t* total) {
  Carver c(base);
  SelWs w;
  w.tile_w = c.take<uint64_t>(T);
  w.tile_key = c.take<uint64_t>(T);
  w.tile_u = c.take<uint64_t>(T);
  w.tile_age = c.take<uint32_t>(T);
  w.rank_h = c.take<int32_t>(3 * (size_t)T);
  w.rank_s = w.rank_h + T;
  w.rank_u = w.rank_h + 2 * T;
  w.scan_sums = c.take<int64_t>((size_t)std::max(1, scan_blocks(T)));
  w.total = c.take<int64_t>(1);
  *total = c.size();
  return w;
}

struct SelGeom {
  int W, H, tx, T;
};

__device__ __forceinline__ int tile_valid(const SelGeom& g, int t) {
  int tx = t % g.tx, ty = t / g.tx;
  return min(TGS_TILE, g.W - tx * TGS_TILE) * min(TGS_TILE, g.H - ty * TGS_TILE);
}

// Hard order: ascending L / w in IEEE double (exact operands, correctly
// rounded division, so every machine computes the same key); weight 0 maps to
// L * 2^900, after every positive weight.  Positive doubles order like their
// bit patterns, so the key is used as an unsigned 64-bit integer; equal keys
// go to the lower index.
__device__ __forceinline__ uint64_t hard_key(uint64_t w, uint64_t L) {
  const double k = w ? __ddiv_rn(__ull2double_rn(L), __ull2double_rn(w)) : __ull2double_rn(L) * 0x1p900;
  return (uint64_t)__double_as_longlong(k);
}

// Per-tile weight (sum), age (min) and the tile's random keys.
// Hash prefixes of the call: the iteration comes from the host or, for graph
// replays, from device memory.
struct HashKeys {
  uint64_t seed, iter;
  const uint64_t* iter_dev;
  uint32_t view;
  __device__ __forceinline__ uint64_t prefix(uint32_t stream) const {
    return hash_prefix(seed, iter_dev ? *iter_dev : iter, view, stream);
  }
};

// 8 tiles per block of 8 warps, one per warp: lane l sums the error
// weights and takes the minimum age of eight pixels (row l / 2, columns
// 8 (l % 2) .. + 7; one 16-byte load per map where the row allows it), then the
// warp reduces.  The draws (-log2 of a hash, 32 dependent squarings) then run
// one tile per lane of the first warp.  Bound by latency: the loads, then the
// draws.  With four tiles a warp (32 a block) a view of 4056 tiles had fewer
// blocks than the chip has SMs: 12.8 us, 8.3 with two, 7.1 with one; 256 tiles
// 6.2, 4.6, 3.9; 8160 tiles 8.6, 7.9, 7.4.
constexpr int kStatsTiles = 8;
constexpr int kStatsPerWarp = kStatsTiles / 8;
static_assert(kStatsTiles % 8 == 0 && kStatsTiles <= 32, "whole tiles per warp, and a lane of the first warp each");

__device__ __forceinline__ void pixel_row8(const uint16_t* __restrict__ err, const uint16_t* __restrict__ age,
                                           const SelGeom& g, int t, int lane, bool vec, uint64_t& wv,
                                           uint32_t& av) {
  wv = 0;
  av = 0xFFFFFFFFu;
  if (t >= g.T) return;
  const int y = (t / g.tx) * TGS_TILE + (lane >> 1), x0 = (t % g.tx) * TGS_TILE + 8 * (lane & 1);
  if (y >= g.H) return;
  const size_t p = (size_t)y * g.W + x0;
  uint16_t e[8], a[8];
  if (vec && x0 + 8 <= g.W) {  // 16-byte aligned: both maps are, and x0 and W are multiples of 8
    const uint4 ev = *reinterpret_cast<const uint4*>(err + p), avv = *reinterpret_cast<const uint4*>(age + p);
    const uint32_t ew[4] = {ev.x, ev.y, ev.z, ev.w}, aw[4] = {avv.x, avv.y, avv.z, avv.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      e[2 * u] = (uint16_t)(ew[u] & 0xFFFFu);
      e[2 * u + 1] = (uint16_t)(ew[u] >> 16);
      a[2 * u] = (uint16_t)(aw[u] & 0xFFFFu);
      a[2 * u + 1] = (uint16_t)(aw[u] >> 16);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      wv += err_weight(e[u]);
      av = min(av, (uint32_t)a[u]);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (x0 + u < g.W) {
        wv += err_weight(err[p + u]);
        av = min(av, (uint32_t)age[p + u]);
      }
  }
}

// The views of a launch; its second grid dimension counts them.
constexpr int kMaxSelViews = 16;
struct SelView {
  const uint16_t* err;
  const uint16_t* age;
  SelGeom g;
  HashKeys hk;
  SelWs w;
  int n_sel, kh, ks;  // tiles to choose, of them by error and by age
  int n_pix, hard_pm, stable_pm;
  bool vec;           // 16-byte loads of the maps are aligned
  int32_t* active_tiles;
  int32_t* n_active;
  int32_t* tile_rank;
  int32_t* pix_off;
  uint8_t* pix_idx;
};
template <int V>
struct SelBatch {
  SelView v[V];
};

template <int V>
__global__ void __launch_bounds__(256) k_tile_stats(const __grid_constant__ SelBatch<V> batch) {
  const SelView& a = batch.v[V == 1 ? 0 : blockIdx.y];
  const SelGeom& g = a.g;
  const HashKeys& hk = a.hk;
  const SelWs& w = a.w;
  __shared__ uint64_t s_w[kStatsTiles];
  __shared__ uint32_t s_a[kStatsTiles];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t0 = blockIdx.x * kStatsTiles;
  uint64_t wv[kStatsPerWarp];
  uint32_t av[kStatsPerWarp];
#pragma unroll
  for (int q = 0; q < kStatsPerWarp; ++q)
    pixel_row8(a.err, a.age, g, t0 + kStatsPerWarp * warp + q, lane, a.vec, wv[q], av[q]);
#pragma unroll
  for (int q = 0; q < kStatsPerWarp; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      wv[q] += __shfl_xor_sync(0xffffffffu, wv[q], o);
      av[q] = min(av[q], __shfl_xor_sync(0xffffffffu, av[q], o));
    }
  }
  if (lane < kStatsPerWarp) {
    // lane q keeps tile q of the warp (register arrays indexed by constants)
    uint64_t ww = wv[0];
    uint32_t aa = av[0];
#pragma unroll
    for (int q = 1; q < kStatsPerWarp; ++q)
      if (lane == q) {
        ww = wv[q];
        aa = av[q];
      }
    s_w[kStatsPerWarp * warp + lane] = ww;
    s_a[kStatsPerWarp * warp + lane] = aa;
  }
  __syncthreads();
  const int t = t0 + lane;
  if (warp == 0 && lane < kStatsTiles && t < g.T) {
    w.tile_w[t] = s_w[lane];
    w.tile_age[t] = s_a[lane];
    // the FP64 division runs here, spread over the grid, and not in the
    // single-block selection (FP64 throughput is low on this part)
    w.tile_key[t] = hard_key(s_w[lane], neglog2_q32(hash_item(hk.prefix(STREAM_TILE_HARD), (uint32_t)t, 0)));
    w.tile_u[t] = hash_item(hk.prefix(STREAM_TILE_UNIF), (uint32_t)t, 0);
  }
}

// Every tile selected: ranks are the tile ids, and the pixels before a tile
// follow from its row and column (only the last row and column have tiles of
// other sizes).  The single-block compaction took 6.3 us at 3600 tiles and 17.8
// at 8487, this 2.8 and 1.5.
__global__ void __launch_bounds__(256) k_select_all(SelGeom g, int n_pix, int32_t* __restrict__ active_tiles,
                                                    int32_t* __restrict__ n_active, int32_t* __restrict__ tile_rank,
                                                    int32_t* __restrict__ pix_off) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= g.T) return;
  const int x = t % g.tx, y = t / g.tx, ty = g.T / g.tx;
  const int w_last = g.W - (g.tx - 1) * TGS_TILE, h_last = g.H - (ty - 1) * TGS_TILE;
  const int h = y == ty - 1 ? h_last : TGS_TILE, w = x == g.tx - 1 ? w_last : TGS_TILE;
  const int row = (g.tx - 1) * min(n_pix, TGS_TILE * TGS_TILE) + min(n_pix, w_last * TGS_TILE);  // of a whole row
  const int off = y * row + x * min(n_pix, TGS_TILE * h);
  active_tiles[t] = t;
  tile_rank[t] = t;
  pix_off[t] = off;
  if (t == g.T - 1) {
    pix_off[g.T] = off + min(n_pix, w * h);
    *n_active = g.T;
  }
}

// rank[i] += #{j in this block's chunk, eligible, preceding i} for the phase.
// phase 0: hard order among all; 1: age order among those not taken by phase
// 0; 2: uniform order among those not taken by phases 0 and 1.
constexpr int RANK_CHUNK = 64;

__global__ void __launch_bounds__(256) k_rank_tiles(SelWs w, int T, int phase, int kh, int ks) {
  __shared__ uint64_t s_k[RANK_CHUNK];
  __shared__ uint8_t s_e[RANK_CHUNK];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j0 = blockIdx.y * RANK_CHUNK;
  // phase key, ascending, ties to the lower index:
  //  0: hard key; 1: (2^32 - 1 - age) (older first); 2: top 32 hash bits
  auto key = [&](int t) -> uint64_t {
    if (phase == 0) return w.tile_key[t];
    if (phase == 1) return 0xFFFFFFFFull - w.tile_age[t];
    return w.tile_u[t] >> 32;
  };
  if (threadIdx.x < RANK_CHUNK) {
    const int j = j0 + threadIdx.x;
    bool e = j < T;
    if (e && phase >= 1) e = w.rank_h[j] >= kh;
    if (e && phase >= 2) e = w.rank_s[j] >= ks;
    s_e[threadIdx.x] = e;
    s_k[threadIdx.x] = j < T ? key(j) : 0;
  }
  __syncthreads();
  if (i >= T) return;
  if (phase >= 1 && w.rank_h[i] < kh) return;
  if (phase >= 2 && w.rank_s[i] < ks) return;
  const uint64_t ki = key(i);
  int cnt = 0;
  const int jn = min(RANK_CHUNK, T - j0);
  for (int k = 0; k < jn; ++k) {
    const uint64_t kj = s_k[k];
    cnt += s_e[k] && (kj < ki || (kj == ki && j0 + k < i));
  }
  if (cnt) atomicAdd(phase == 0 ? &w.rank_h[i] : phase == 1 ? &w.rank_s[i] : &w.rank_u[i], cnt);
}

// Tile level in one block of 1024 threads (up to 1024 * ITEMS tiles): the
// three phases, then the ascending compaction into active_tiles, tile_rank,
// pix_off and n_active.
constexpr int kSelBlockMaxTiles = kSelThreads * 16;

template <int ITEMS, int V>
__global__ void __launch_bounds__(kSelThreads, 1) k_select_block(const __grid_constant__ SelBatch<V> batch) {
  const SelView& a = batch.v[V == 1 ? 0 : blockIdx.y];
  const SelGeom& g = a.g;
  const SelWs& w = a.w;
  const int n_sel = a.n_sel, kh = a.kh, ks = a.ks, n_pix = a.n_pix;
  int32_t* __restrict__ active_tiles = a.active_tiles;
  int32_t* __restrict__ tile_rank = a.tile_rank;
  int32_t* __restrict__ pix_off = a.pix_off;
  __shared__ SelectSmem sm;
  __shared__ int64_t s64[32];
  const int T = g.T;
  const int i0 = threadIdx.x * ITEMS;
  const uint32_t valid = i0 < T ? (ITEMS < T - i0 ? (1u << ITEMS) - 1u : (1u << (T - i0)) - 1u) : 0u;
  uint32_t taken = 0u;
  if (n_sel > 0) {
    uint32_t key[ITEMS];
    // the hard keys are read again where their low words are wanted
    auto hard = [&](int j) -> uint64_t { return (valid >> j) & 1u ? w.tile_key[i0 + j] : 0ull; };
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = (uint32_t)(hard(j) >> 32);
    const uint32_t th = block_select<ITEMS, true>(key, hard, valid, kh, sm, s64);
    auto same = [&](int j) -> uint64_t {
      uint32_t v = key[0];
#pragma unroll
      for (int q = 1; q < ITEMS; ++q) v = j == q ? key[q] : v;
      return v;
    };
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = (valid >> j) & 1u ? 0xFFFFu - min(w.tile_age[i0 + j], 0xFFFFu) : 0u;
    const uint32_t ts = block_select<ITEMS, false>(key, same, valid & ~th, ks, sm, s64);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) key[j] = (valid >> j) & 1u ? (uint32_t)(w.tile_u[i0 + j] >> 32) : 0u;
    const uint32_t tu = block_select<ITEMS, false>(key, same, valid & ~th & ~ts, n_sel - kh - ks, sm, s64);
    taken = th | ts | tu;
  }
  // compaction: (taken count << 32 | pixel count) prefix in tile order; the
  // tile's place in the image follows from the thread's first by steps
  const int x0 = i0 % g.tx, y0 = i0 / g.tx;
  auto each = [&](auto f) {
    int x = x0, y = y0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int nv = min(TGS_TILE, g.W - x * TGS_TILE) * min(TGS_TILE, g.H - y * TGS_TILE);
      f(j, (1ll << 32) | (int64_t)min(n_pix, nv));
      if (++x == g.tx) {
        x = 0;
        ++y;
      }
    }
  };
  int64_t mine = 0;
  each([&](int j, int64_t v) { mine += (taken >> j) & 1u ? v : 0; });
  int64_t total;
  int64_t pre = block_excl_sum(mine, s64, total);
  each([&](int j, int64_t v) {
    const int i = i0 + j;
    if ((taken >> j) & 1u) {
      const int r = (int)(pre >> 32);
      tile_rank[i] = r;
      active_tiles[r] = i;
      pix_off[r] = (int)(pre & 0xFFFFFFFFll);
      pre += v;
    } else if ((valid >> j) & 1u) {
      tile_rank[i] = -1;
    }
  });
  if (threadIdx.x == 0) {
    *a.n_active = (int32_t)(total >> 32);
    pix_off[total >> 32] = (int32_t)(total & 0xFFFFFFFFll);
  }
}

// ---------------------------------------------------------------------------
// Pixel sampling inside the chosen tiles: one warp per tile, lane l on the
// local pixels l, l + 32, ..., l + 224 (two rows of the tile at a time), so
// that every count is a ballot or a warp sum and nothing waits at a barrier.
//
// The error-proportional draw takes the kh smallest of L / w, in the exact
// order of hard_key: L a logarithm by 32 squarings of 64-bit integers and a
// quotient in FP64, about 500 instructions a pixel.  Which pixels those are is
// nearly always clear from a few digits, so the warp first orders the pixels by
// an approximate quotient in fp32 with a bound on its error, and takes the kh
// smallest of these if the largest bound of the taken lies below the smallest
// bound of the others (then the exact order takes the same); otherwise the
// pixels between those two bounds, two as a rule, are ordered by their exact
// keys.  With one block of 256 threads per tile, exact keys throughout and a
// block-wide radix selection, the kernel was bound by its instructions (73 % of
// the issue slots, 15000 warp instructions a tile; 2600 here): every tile of
// 1280x720, 85 of 256 pixels: 66 -> 19 us; 1420 tiles 30 -> 12; eight views of
// 1200 to 4500 tiles 436 -> 125.
// ---------------------------------------------------------------------------
constexpr int kPix = 256 / 32;  // pixels a lane

// The k smallest (key, index) of the warp's eligible pixels, as a bit mask per
// lane (bit j: pixel lane + 32 j).  The k-th smallest key is found one bit at
// a time from the first bit in which the eligible keys differ; once the keys
// that match the bits found are exactly those still wanted, the rest decides
// nothing.  Ties at the last key go to the lower index.
template <typename Key>
__device__ __forceinline__ uint32_t warp_select(const Key (&key)[kPix], uint32_t elig, int k) {
  const unsigned full = 0xffffffffu;
  if (k <= 0) return 0u;
  int play = __reduce_add_sync(full, __popc(elig));  // keys that match the bits found
  if (k >= play) return elig;
  // the bits in which they differ
  Key any = 0, all = ~(Key)0;
#pragma unroll
  for (int j = 0; j < kPix; ++j)
    if ((elig >> j) & 1u) {
      any |= key[j];
      all &= key[j];
    }
  Key diff;
  if (sizeof(Key) == 8) {
    const uint32_t lo = __reduce_or_sync(full, (uint32_t)any) ^ __reduce_and_sync(full, (uint32_t)all);
    const uint32_t hi = __reduce_or_sync(full, (uint32_t)((uint64_t)any >> 32)) ^
                        __reduce_and_sync(full, (uint32_t)((uint64_t)all >> 32));
    diff = (Key)(((uint64_t)hi << 32) | lo);
  } else {
    diff = (Key)(__reduce_or_sync(full, (uint32_t)any) ^ __reduce_and_sync(full, (uint32_t)all));
  }
  uint32_t in = elig, below = 0u;  // pixels that match the bits found; pixels below them
  int kk = k;
  while (diff && kk < play) {
    const int bit = sizeof(Key) == 8 ? 63 - __clzll((long long)diff) : 31 - __clz((int)diff);
    uint32_t zero = 0u;
#pragma unroll
    for (int j = 0; j < kPix; ++j) zero |= (((key[j] >> bit) & 1u) ? 0u : 1u) << j;
    zero &= in;
    const int c = __reduce_add_sync(full, __popc(zero));
    if (kk <= c) {
      in = zero;
      play = c;
    } else {
      below |= zero;
      in &= ~zero;
      kk -= c;
      play -= c;
    }
    diff &= ~((Key)1 << bit);
  }
  if (kk < play) {  // equal keys: the first kk in index order
    uint32_t t = 0u;
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
#pragma unroll
    for (int j = 0; j < kPix; ++j) {
      const uint32_t b = __ballot_sync(full, (in >> j) & 1u);
      if (((in >> j) & 1u) && __popc(b & lt) < kk) t |= 1u << j;
      kk = max(0, kk - __popc(b));
    }
    in = t;
  }
  return below | in;
}

// -log2 of the hash, in units of 1, to within kLogErr and 2^-24 of itself (the
// difference's rounding): the top 24 bits of the mantissa (2^-22.5), the fast
// logarithm of a value in [1, 2) (2^-21.4) and the truncations of neglog2_q32
// (2^-31) are together below half of kLogErr.
constexpr float kLogErr = 0x1p-19f;
__device__ __forceinline__ float neglog2_approx(uint64_t h) {
  const uint64_t u = h | 1ull;
  const int lz = __clzll((long long)u);
  return fmaxf((float)(lz + 1) - __log2f((float)(uint32_t)((u << lz) >> 40) * 0x1p-23f), 0.f);
}

constexpr int kSampleWarps = 4;  // tiles per block

template <int V>
__global__ void __launch_bounds__(32 * kSampleWarps) k_sample_pixels(const __grid_constant__ SelBatch<V> batch) {
  const SelView& a = batch.v[V == 1 ? 0 : blockIdx.y];
  const SelGeom& g = a.g;
  const HashKeys& hk = a.hk;
  const uint16_t* __restrict__ err = a.err;
  const uint16_t* __restrict__ age = a.age;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * kSampleWarps + (threadIdx.x >> 5);
  if (j0 >= a.n_sel || j0 >= *a.n_active) return;
  const int t = a.active_tiles[j0];
  const int x = (t % g.tx) * TGS_TILE + (lane & 15), y = (t / g.tx) * TGS_TILE + (lane >> 4);  // pixel j: row y + 2 j
  uint32_t valid = 0u;
#pragma unroll
  for (int j = 0; j < kPix; ++j)
    if (x < g.W && y + 2 * j < g.H) valid |= 1u << j;
  const int nv = tile_valid(g, t);
  const int n = min(a.n_pix, nv);
  int kh, ks;
  split_counts(n, a.hard_pm, a.stable_pm, kh, ks);
  uint32_t taken = valid;  // n >= nv: every valid pixel
  if (n < nv) {
    const size_t p0 = (size_t)y * g.W + x;
    uint16_t ev[kPix], av[kPix];
#pragma unroll
    for (int j = 0; j < kPix; ++j) {
      const bool in = (valid >> j) & 1u;
      ev[j] = in && kh > 0 ? err[p0 + (size_t)(2 * j) * g.W] : (uint16_t)0;
      av[j] = in && ks > 0 ? age[p0 + (size_t)(2 * j) * g.W] : (uint16_t)0;
    }
    uint32_t th = 0u;
    if (kh > 0) {
      const uint64_t pre = hk.prefix(STREAM_PIX_HARD);
      uint32_t key[kPix];
      float d[kPix];
#pragma unroll
      for (int j = 0; j < kPix; ++j) {
        const float l = neglog2_approx(hash_item(pre, (uint32_t)t, (uint32_t)(lane + 32 * j)));
        // weight 0 comes after every positive weight, whose quotients are at most 65
        const float w = (float)err_weight(ev[j]);
        const float rw = w > 0.f ? __fdividef(1.f, w) : 0x1p60f;
        key[j] = __float_as_uint(l * rw);  // l >= 0: ordered like its bits
        d[j] = kLogErr * rw;
      }
      th = warp_select<uint32_t>(key, valid, kh);
      // taken and not taken, apart by their bounds (2^-19 of the quotient covers the roundings of the weight, the division and L)
      float top = 0.f, low = 0x1p126f;
#pragma unroll
      for (int j = 0; j < kPix; ++j) {
        const float c = __uint_as_float(key[j]);
        if ((th >> j) & 1u) top = fmaxf(top, c + (c * 0x1p-19f + d[j]));
        else if ((valid >> j) & 1u) low = fminf(low, c - (c * 0x1p-19f + d[j]));
      }
      const float t_top = __uint_as_float(__reduce_max_sync(full, __float_as_uint(top)));
      const float t_low = __uint_as_float(__reduce_min_sync(full, __float_as_uint(fmaxf(low, 0.f))));
      if (t_top >= t_low) {
        // in doubt: the taken whose bound reaches the lowest of the others, and the others that reach the highest of
        // the taken; the rest is as the approximate order has it
        uint32_t doubt = 0u;
#pragma unroll
        for (int j = 0; j < kPix; ++j) {
          const float c = __uint_as_float(key[j]), e = c * 0x1p-19f + d[j];
          if ((th >> j) & 1u ? c + e >= t_low : ((valid >> j) & 1u) && c - e <= t_top) doubt |= 1u << j;
        }
        const int kk = __reduce_add_sync(full, __popc(doubt & th));
        uint64_t exact[kPix];
#pragma unroll
        for (int q = 0; q < kPix; ++q) exact[q] = 0;
#pragma unroll 1
        for (uint32_t rem = doubt; __any_sync(full, rem); rem &= rem - 1u) {  // each lane's next one
          const int j = __ffs(rem) - 1;
          uint16_t e = 0;
#pragma unroll
          for (int q = 0; q < kPix; ++q) e = j == q ? ev[q] : e;
          const uint64_t v =
              hard_key(err_weight(e), neglog2_q32(hash_item(pre, (uint32_t)t, (uint32_t)(lane + 32 * j))));
#pragma unroll
          for (int q = 0; q < kPix; ++q) exact[q] = j == q ? v : exact[q];
        }
        th = (th & ~doubt) | warp_select<uint64_t>(exact, doubt, kk);
      }
    }
    // the oldest of the rest, then the uniform draw of the rest
    uint32_t ts = 0u, tu = 0u;
    if (ks > 0) {
      uint32_t key[kPix];
#pragma unroll
      for (int j = 0; j < kPix; ++j) key[j] = 0xFFFFu - av[j];
      ts = warp_select<uint32_t>(key, valid & ~th, ks);
    }
    if (n - kh - ks > 0) {
      const uint64_t pre = hk.prefix(STREAM_PIX_UNIF);
      uint32_t key[kPix];
#pragma unroll
      for (int j = 0; j < kPix; ++j)
        key[j] = (uint32_t)(hash_item(pre, (uint32_t)t, (uint32_t)(lane + 32 * j)) >> 32);
      tu = warp_select<uint32_t>(key, valid & ~th & ~ts, n - kh - ks);
    }
    taken = th | ts | tu;
  }
  // the taken local indices, ascending
  uint8_t* out = a.pix_idx + a.pix_off[j0];
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int j = 0; j < kPix; ++j) {
    const uint32_t b = __ballot_sync(full, (taken >> j) & 1u);
    if ((taken >> j) & 1u) out[__popc(b & lt)] = (uint8_t)(lane + 32 * j);
    out += __popc(b);
  }
}

__global__ void k_sel_finish(const int64_t* __restrict__ total, int32_t* __restrict__ n_active,
                             int32_t* __restrict__ pix_off) {
  const int64_t v = *total;
  *n_active = (int32_t)(v >> 32);
  pix_off[v >> 32] = (int32_t)(v & 0xFFFFFFFFll);
}

}  // namespace tgs

using namespace tgs;

// One view's arguments (checked) as the kernels take them.
static SelView make_view(const uint16_t* err_map, const uint16_t* age_map, int32_t width, int32_t height,
                         int32_t n_select, int32_t n_pix, const tgs_sampling* cfg, uint64_t seed, uint64_t iter,
                         const uint64_t* iter_dev, uint32_t view, void* scratch, int32_t* active_tiles,
                         int32_t* n_active, int32_t* tile_rank, int32_t* pix_off, uint8_t* pix_idx) {
  const int T = tiles_x(width) * tiles_y(height);
  SelView a;
  size_t tot;
  a.err = err_map;
  a.age = age_map;
  a.g = SelGeom{width, height, tiles_x(width), T};
  a.hk = HashKeys{seed, iter, iter_dev, view};
  a.w = carve_sel(scratch, T, &tot);
  a.n_sel = std::min(n_select, T);
  split_counts(a.n_sel, cfg->tile_hard_pm, cfg->tile_stable_pm, a.kh, a.ks);
  a.n_pix = n_pix;
  a.hard_pm = cfg->pix_hard_pm;
  a.stable_pm = cfg->pix_stable_pm;
  a.vec = aligned16(err_map) && aligned16(age_map) && width % 8 == 0;
  a.active_tiles = active_tiles;
  a.n_active = n_active;
  a.tile_rank = tile_rank;
  a.pix_off = pix_off;
  a.pix_idx = pix_idx;
  return a;
}

// The tiles of the batch's first `count` views, each of at most max_T <=
// kSelBlockMaxTiles tiles and fewer chosen: the statistics, and one block per
// view for the three phases and the compaction.
template <int V>
static void launch_block_select(const SelBatch<V>& b, int count, int max_T, bool any, cudaStream_t s) {
  if (any) k_tile_stats<V><<<dim3((max_T + kStatsTiles - 1) / kStatsTiles, count), 256, 0, s>>>(b);
  const dim3 grid(1, count);
  if (max_T <= kSelThreads) k_select_block<1, V><<<grid, kSelThreads, 0, s>>>(b);
  else if (max_T <= kSelThreads * 4) k_select_block<4, V><<<grid, kSelThreads, 0, s>>>(b);
  else if (max_T <= kSelThreads * 8) k_select_block<8, V><<<grid, kSelThreads, 0, s>>>(b);
  else k_select_block<16, V><<<grid, kSelThreads, 0, s>>>(b);
}

static bool block_selects(const SelView& a) { return a.n_sel < a.g.T && a.g.T <= kSelBlockMaxTiles; }

// The tiles of one view.
static void launch_tiles(const SelView& a, cudaStream_t s) {
  const int T = a.g.T, n_sel = a.n_sel;
  if (n_sel >= T) {
    k_select_all<<<(T + 255) / 256, 256, 0, s>>>(a.g, a.n_pix, a.active_tiles, a.n_active, a.tile_rank, a.pix_off);
    return;
  }
  const SelBatch<1> one{{a}};
  if (T <= kSelBlockMaxTiles) {
    launch_block_select<1>(one, 1, T, n_sel > 0, s);
    return;
  }
  // many tiles: ranks by pairwise counting, then a device-wide scan.  A
  // tile is taken when rank_h < kh, or (not hard) rank_s < ks, or
  // (neither) rank_u < n_sel - kh - ks.
  const SelWs& w = a.w;
  const int kh = a.kh, ks = a.ks;
  if (n_sel > 0) k_tile_stats<1><<<(T + kStatsTiles - 1) / kStatsTiles, 256, 0, s>>>(one);
  cudaMemsetAsync(w.rank_h, 0, sizeof(int32_t) * 3 * (size_t)T, s);
  if (n_sel > 0) {
    dim3 grid((T + 255) / 256, (T + RANK_CHUNK - 1) / RANK_CHUNK);
    if (kh > 0) k_rank_tiles<<<grid, 256, 0, s>>>(w, T, 0, kh, ks);
    if (ks > 0) k_rank_tiles<<<grid, 256, 0, s>>>(w, T, 1, kh, ks);
    if (n_sel - kh - ks > 0) k_rank_tiles<<<grid, 256, 0, s>>>(w, T, 2, kh, ks);
  }
  const int32_t* rh = w.rank_h;
  const int32_t* rs = w.rank_s;
  const int32_t* ru = w.rank_u;
  const int none = n_sel == 0 ? 1 : 0;
  const int ku = n_sel - kh - ks;
  const int npx = a.n_pix;
  const SelGeom g = a.g;
  int32_t* at = a.active_tiles;
  int32_t* tr = a.tile_rank;
  int32_t* po = a.pix_off;
  auto load = [=] __device__(int64_t t) -> int64_t {
    const bool taken = !none && (rh[t] < kh || rs[t] < ks || (rs[t] >= ks && ru[t] < ku));
    if (!taken) return 0;
    return (1ll << 32) | (int64_t)min(npx, tile_valid(g, (int)t));
  };
  auto store = [=] __device__(int64_t t, int64_t pre, int64_t v) {
    if (v) {
      const int r = (int)(pre >> 32);
      tr[t] = r;
      at[r] = (int)t;
      po[r] = (int)(pre & 0xFFFFFFFFll);
    } else {
      tr[t] = -1;
    }
  };
  exclusive_scan<int64_t>(load, store, nullptr, T, w.scan_sums, w.total, s);
  k_sel_finish<<<1, 1, 0, s>>>(w.total, a.n_active, a.pix_off);
}

// The launch sequence of the one-view entry points.
static tgs_status launch_select(const SelView& a, cudaStream_t s) {
  launch_tiles(a, s);
  if (a.n_sel > 0)
    k_sample_pixels<1><<<(a.n_sel + kSampleWarps - 1) / kSampleWarps, 32 * kSampleWarps, 0, s>>>(SelBatch<1>{{a}});
  return check_launch();
}

// What every entry point refuses.
static bool select_args_ok(const uint16_t* err_map, const uint16_t* age_map, int32_t width, int32_t height,
                           int32_t n_select, int32_t n_pix, const tgs_sampling* cfg, const int32_t* n_active,
                           const int32_t* tile_rank, const int32_t* pix_off) {
  if (width <= 0 || height <= 0 || width > (1 << 16) || height > (1 << 16) || n_select < 0 || n_pix < 1 ||
      n_pix > 256 || !cfg || !err_map || !age_map || !n_active || !tile_rank || !pix_off)
    return false;
  const int pms[4] = {cfg->tile_hard_pm, cfg->tile_stable_pm, cfg->pix_hard_pm, cfg->pix_stable_pm};
  for (int k = 0; k < 4; ++k)
    if (pms[k] < 0 || pms[k] > 1000) return false;
  return true;
}
static bool select_outputs_ok(int32_t n_select, const int32_t* active_tiles, const uint8_t* pix_idx) {
  return n_select == 0 || (active_tiles && pix_idx);
}

extern "C" size_t tgs_select_tiles_workspace_size(int32_t width, int32_t height) {
  size_t total = 0;
  if (width <= 0 || height <= 0) return 0;
  carve_sel(nullptr, tiles_x(width) * tiles_y(height), &total);
  return total;
}

extern "C" tgs_status tgs_select_tiles(const uint16_t* err_map, const uint16_t* age_map, int32_t width,
                                       int32_t height, int32_t n_select, int32_t n_pix, const tgs_sampling* cfg,
                                       uint64_t seed, uint64_t iter, const uint64_t* iter_dev, uint32_t view,
                                       void* workspace, size_t workspace_bytes, int32_t* active_tiles, int32_t* n_active,
                                       int32_t* tile_rank, int32_t* pix_off, uint8_t* pix_idx,
                                       tgs_stream stream) {
  if (!select_args_ok(err_map, age_map, width, height, n_select, n_pix, cfg, n_active, tile_rank, pix_off) ||
      !select_outputs_ok(n_select, active_tiles, pix_idx) || !workspace || workspace_bytes < tgs_select_tiles_workspace_size(width, height))
    return TGS_ERR_INVALID_ARG;
  return launch_select(make_view(err_map, age_map, width, height, n_select, n_pix, cfg, seed, iter, iter_dev, view,
                                 workspace, active_tiles, n_active, tile_rank, pix_off, pix_idx),
                       (cudaStream_t)stream);
}

// Views chosen by one block each share the launches; a view with every tile, or
// with more tiles than a block takes, is chosen by itself.  Eight views of 8160
// tiles, 1200 to 4500 chosen, statistics, tiles and pixels: 380 -> 135 us.
extern "C" tgs_status tgs_select_tiles_batched(int32_t n_views, const tgs_select_view* views, const tgs_sampling* cfg,
                                               uint64_t iter, const uint64_t* iter_dev, tgs_stream stream) {
  if (n_views < 1 || n_views > kMaxSelViews || !views) return TGS_ERR_INVALID_ARG;
  SelBatch<kMaxSelViews> all, block;
  int in_block = 0, max_T = 0, max_sel = 0;
  bool any = false;
  for (int k = 0; k < n_views; ++k) {
    const tgs_select_view& v = views[k];
    if (!select_args_ok(v.err_map, v.age_map, v.width, v.height, v.n_select, v.n_pix, cfg, v.n_active, v.tile_rank,
                        v.pix_off) ||
        !select_outputs_ok(v.n_select, v.active_tiles, v.pix_idx) || !v.workspace || v.workspace_bytes < tgs_select_tiles_workspace_size(v.width, v.height))
      return TGS_ERR_INVALID_ARG;
    all.v[k] = make_view(v.err_map, v.age_map, v.width, v.height, v.n_select, v.n_pix, cfg, v.seed, iter, iter_dev,
                         v.view, v.workspace, v.active_tiles, v.n_active, v.tile_rank, v.pix_off, v.pix_idx);
    max_sel = std::max(max_sel, all.v[k].n_sel);
    if (block_selects(all.v[k])) {
      max_T = std::max(max_T, all.v[k].g.T);
      any = any || all.v[k].n_sel > 0;
      block.v[in_block++] = all.v[k];
    }
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (n_views == 1) return launch_select(all.v[0], s);
  for (int k = 0; k < n_views; ++k)
    if (!block_selects(all.v[k])) launch_tiles(all.v[k], s);
  if (in_block) launch_block_select<kMaxSelViews>(block, in_block, max_T, any, s);
  if (max_sel > 0)
    k_sample_pixels<kMaxSelViews>
        <<<dim3((max_sel + kSampleWarps - 1) / kSampleWarps, n_views), 32 * kSampleWarps, 0, s>>>(all);
  return check_launch();
}

// ---------------------------------------------------------------------------
// select_tiles without a caller workspace.
//
// For callers that cannot allocate device memory - for example code running
// inside a host framework that hands out all device memory from its own fixed
// pool and forbids any other allocation, or a latency-critical path where an
// allocation could block or synchronise the device.  The scratch that
// tgs_select_tiles carves out of `workspace` lives here in one file-scope
// device array of fixed size instead; every GPU that loads this library holds
// it until the process exits.
// ---------------------------------------------------------------------------
#include <mutex>

namespace {

__device__ __align__(256) unsigned char g_select_scratch[TGS_SELECT_NOALLOC_SCRATCH_BYTES];

std::mutex g_scratch_mu;
void* g_scratch_ptr[TGS_SELECT_NOALLOC_MAX_DEVICES] = {};

// Device address of g_select_scratch on the current device.  In host code the
// array's name is only a host-side stand-in, so the address is looked up once
// per device (with that device current) and cached.
tgs_status select_scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    tgs::set_cuda_error(e);
    return TGS_ERR_CUDA;
  }
  if (dev < 0 || dev >= TGS_SELECT_NOALLOC_MAX_DEVICES) return TGS_ERR_CAPACITY;  // the cache's size
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_select_scratch);
    if (e != cudaSuccess || !p) {
      tgs::set_cuda_error(e);
      return TGS_ERR_CUDA;
    }
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return TGS_OK;
}

}  // namespace

extern "C" tgs_status tgs_select_tiles_noalloc(const uint16_t* err_map, const uint16_t* age_map, int32_t width,
                                               int32_t height, int32_t n_select, int32_t n_pix,
                                               const tgs_sampling* cfg, uint64_t seed, uint64_t iter,
                                               const uint64_t* iter_dev, uint32_t view, int32_t* active_tiles,
                                               int32_t* n_active, int32_t* tile_rank, int32_t* pix_off,
                                               uint8_t* pix_idx, tgs_stream stream) {
  if (!select_args_ok(err_map, age_map, width, height, n_select, n_pix, cfg, n_active, tile_rank, pix_off))
    return TGS_ERR_INVALID_ARG;
  const int T = tiles_x(width) * tiles_y(height);
  if (T > TGS_SELECT_NOALLOC_MAX_TILES) return TGS_ERR_CAPACITY;
  size_t need = 0;
  carve_sel(nullptr, T, &need);
  if (need > sizeof(g_select_scratch)) return TGS_ERR_CAPACITY;
  if (!select_outputs_ok(n_select, active_tiles, pix_idx)) return TGS_ERR_INVALID_ARG;
  void* scratch = nullptr;
  tgs_status st = select_scratch_address(&scratch);
  if (st != TGS_OK) return st;
  return launch_select(make_view(err_map, age_map, width, height, n_select, n_pix, cfg, seed, iter, iter_dev, view,
                                 scratch, active_tiles, n_active, tile_rank, pix_off, pix_idx),
                       (cudaStream_t)stream);
}
