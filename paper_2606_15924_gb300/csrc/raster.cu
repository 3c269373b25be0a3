// Sparse forward rasterization and its adjoint (Sec. 3.6, Eq. 1).
//
// One thread block per active tile, one warp per 32 (or 64) sampled pixels of
// the tile, so a tile sampled at rate 0.1 runs as one warp; each warp walks the
// tile's depth-ordered splat list until its pixels have saturated, two splats
// at a time.  The backward replays the same walk in
// reverse from the stored final transmittance, recovering T_k by division, one
// warp per group of pixels and piece of the list, two splats at a time.
#include <climits>

#include "tgs_common.cuh"

namespace tgs {

void launch_project_bwd(const tgs_gaussians& g, const tgs_camera& cam, const int32_t* radius, const float* grad2d,
                        const tgs_param_ptrs& grads, uint8_t* touched, int write_untouched, int accumulate,
                        float* row, cudaStream_t s);
bool gaussians_ok(const tgs_gaussians* g);
bool camera_ok(const tgs_camera* c);

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTStop = 1e-4f;
constexpr int kUnroll = 4;  // splats per step of the forward walk
constexpr int kCkptEvery = 32;  // list positions per checkpoint slot (a multiple of kUnroll)

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct Splat {
  float2 xy;
  float2 yr;   // the rows [y0, y1] outside which alpha < 1/255 (with a margin)
  float4 co;   // the conic pre-scaled to base-2 exponents: (-a/2, -b, -c/2) log2(e), then the opacity
  float4 rgb;  // r, g, b, (unused)
};

// Staging scale of the conic: with a' = -a log2(e) / 2, b' = -b log2(e) and
// c' = -c log2(e) / 2 the exponent of Eq. 1's Gaussian in base 2 is
// p = a' dx^2 + b' dx dy + c' dy^2 = log2(e) power.
constexpr float kPow2A = -0.5f * kLog2e;
constexpr float kPow2B = -kLog2e;
// back to the conic: a = a' kInvA, b = b' kInvB, c = c' kInvA
constexpr float kInvA = -1.3862943611198906f;  // -2 ln 2
constexpr float kInvB = -0.6931471805599453f;  // -ln 2

// p = log2(e) power at offset (dx, dy) from the splat's centre, with the
// pre-scaled conic: (a' dx + b' dy) dx + c' dy^2 (explicitly rounded, so
// every kernel takes the same decisions for the same splat and pixel).
__device__ __forceinline__ float splat_pow2(const float4& co, float dx, float dy) {
  const float t = __fmaf_rn(co.x, dx, __fmul_rn(co.y, dy));
  return __fmaf_rn(t, dx, __fmul_rn(__fmul_rn(co.z, dy), dy));
}

// alpha of a splat at offset (dx, dy) from its centre; G receives exp(power).
// Returns false when the splat is skipped (power > 0 or alpha < 1/255).
__device__ __forceinline__ bool splat_alpha(const float4& co, float dx, float dy, float& alpha, float& G) {
  const float p = splat_pow2(co, dx, dy);
  if (p > 0.f) return false;
  G = ex2_approx(p);
  alpha = fminf(kAlphaMax, __fmul_rn(co.w, G));
  return alpha >= kAlphaMin;
}

// The same decision without a branch: alpha and G are computed in every case
// (for power > 0, G may be +inf and alpha 0.99, finite either way), and the
// return value says whether the splat counts.
__device__ __forceinline__ bool splat_alpha_nb(const float4& co, float dx, float dy, float& alpha, float& G) {
  const float p = splat_pow2(co, dx, dy);
  G = ex2_approx(p);
  alpha = fminf(kAlphaMax, __fmul_rn(co.w, G));
  return p <= 0.f && alpha >= kAlphaMin;
}

struct RasterArgs {
  const float2* xy;
  const float4* conic_opac;
  const float* rgb;
  const int2* ranges;
  const int32_t* vals;
  const int32_t* active_tiles;
  const int32_t* n_active;
  const int32_t* pix_off;
  const uint8_t* pix_idx;
  int tiles_x;
  float bg[3];
};

// Rows a splat can reach: alpha >= 1/255 needs power >= -tau with
// tau = ln(255 o), i.e. the ellipse a dx^2 + 2 b dx dy + c dy^2 <= 2 tau,
// whose half-height is sqrt(2 tau a / (a c - b^2)).  The margin (1e-3
// relative + 1e-3 px) covers the rounding of the kernels' own alpha test, so
// a pixel outside [y0, y1] never passes it.  Empty when o <= 1/255.
__device__ __forceinline__ float2 splat_rows(float y, const float4& c) {
  const float tau = logf(255.f * c.w);
  if (!(tau > 0.f)) return make_float2(INFINITY, -INFINITY);
  const float det = c.x * c.z - c.y * c.y;
  if (!(det > 0.f) || !(c.x > 0.f)) return make_float2(-INFINITY, INFINITY);
  const float h = sqrtf(2.f * tau * c.x / det) * 1.001f + 1e-3f;
  return make_float2(y - h, y + h);
}

// A splat's projected record as loaded (loads only: a walk fetches the next
// batch's records into registers and waits on them only when it stages them,
// a whole batch later).
struct SplatRaw {
  float2 xy;
  float4 c;
  float r, g, b;
  int id;
};

__device__ __forceinline__ void fetch_splat(const RasterArgs& a, int id, SplatRaw& w) {
  w.id = id;
  w.xy = a.xy[id];
  w.c = a.conic_opac[id];
  w.r = a.rgb[3 * id];
  w.g = a.rgb[3 * id + 1];
  w.b = a.rgb[3 * id + 2];
}

__device__ __forceinline__ void finish_splat(const SplatRaw& w, Splat& sp) {
  sp.xy = w.xy;
  sp.yr = splat_rows(w.xy.y, w.c);
  sp.co = make_float4(__fmul_rn(w.c.x, kPow2A), __fmul_rn(w.c.y, kPow2B), __fmul_rn(w.c.z, kPow2A), w.c.w);
  sp.rgb = make_float4(w.r, w.g, w.b, __int_as_float(w.id));
}

__device__ __forceinline__ void load_splat(const RasterArgs& a, int k, Splat& sp) {
  SplatRaw w;
  fetch_splat(a, a.vals[k], w);
  finish_splat(w, sp);
}

// The rows [y0, y1] spanned by the sampled pixels of the calling warp
// (sampled pixels are in row-major order, so a warp's pixels form a band).
__device__ __forceinline__ float2 warp_rows(bool has, float py) {
  float lo = has ? py : INFINITY, hi = has ? py : -INFINITY;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  return make_float2(lo, hi);
}

// Checkpoints of the sampled forward for the split backward: slot c (c = 0
// .. n_slots - 1) of pixel s holds (T, C_r, C_g, C_b) in front of tile-list
// position (c + 1) kCkptEvery, at data[c * stride + s]; written by every
// pixel whose walk reaches that position.
struct Ckpt {
  float4* data;
  int n_slots;
  int64_t stride;
  const float* rgb;    // the forward's output (read by the backward)
  int32_t* tile_last;  // [active rank] longest blended run of the tile's pixels (nullable)
};

// Two fp32 values in one 64-bit register pair: each operation is the IEEE
// operation on both, in one issue slot.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float y;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// The rectangle (x0, y0, x1, y1) outside which a splat's alpha stays below
// 1/255: splat_rows along both axes (half-width sqrt(2 tau c / det)), with
// approximate functions and tau rounded up by 1e-6, well inside the margins.
__device__ __forceinline__ float4 splat_reach(float2 xy, const float4& c) {
  const float x = 255.f * c.w;
  if (!(x > 1.f)) return make_float4(INFINITY, INFINITY, -INFINITY, -INFINITY);
  const float det = c.x * c.z - c.y * c.y;
  if (!(det > 0.f) || !(c.x > 0.f)) return make_float4(-INFINITY, -INFINITY, INFINITY, INFINITY);
  const float k = __fdividef(2.f * (__logf(x) + 1e-6f), det);
  const float h = sqrt_approx(k * c.x) * 1.001f + 1e-3f, w = sqrt_approx(k * c.z) * 1.001f + 1e-3f;
  return make_float4(xy.x - w, xy.y - h, xy.x + w, xy.y + h);
}
__device__ __forceinline__ bool splat_reaches(float2 xy, const float4& c, float4 box) {
  const float4 r = splat_reach(xy, c);
  return r.w >= box.y && r.y <= box.w && r.z >= box.x && r.x <= box.z;
}

// ---------------------------------------------------------------------------
// The forward walk.  Every warp takes 32 PPL sampled pixels of a tile and
// walks the tile's list on its own, in chunks of 32 positions: one splat per
// lane is fetched (a chunk ahead) and tested against the rectangle of the
// warp's pixels, the ones that can reach it are kept in shared memory in pairs,
// and the pairs are evaluated in packed fp32 arithmetic, two splats an issue
// slot.  Only the blend goes through a pair one after the other, with the same
// operations in the same order as a walk of single splats, so the results are
// that walk's bits: a splat that a pixel skips has alpha 0 there, which leaves
// T and the colour as they are.
//
// Bound: instruction issue (every tile of 1M Gaussians at 1957x1091: 80 %
// issue); in sparse launches the chain of the longest list.  Against one thread
// per pixel over splats staged by the block, one splat at a time: that view
// 511 -> 313 us, the dense view of 500k Gaussians 279 -> 181, 720 tiles of 85
// pixels 56 -> 47, 3600 of 25 pixels 95 -> 67, eight views of 3M Gaussians 690 ->
// 541.  Two pixels a lane halve the per-chunk work (358 -> 313 and 194 -> 181 us
// for the whole tiles above) but lengthen the chains (20 whole tiles: 9.6 ->
// 12.2 us; 85 pixels a tile: 541 -> 646 us, half of the second warp idles).
// Staging the list once per block saves gathers (the L1 is 55-73 % busy with
// them) but its barriers cost more: 390 -> 421 us for the first view.
// ---------------------------------------------------------------------------
struct __align__(16) FwdPair {
  f32x2 nx, ny;  // minus the centre
  f32x2 ca, cb;  // the pre-scaled conic
  f32x2 cc, op;  // and the opacity
  f32x2 cr, cg;  // colour
  f32x2 cbl;
  int end[2];    // 1 + position in the tile's list
};
constexpr int kFwdPairs = 16;  // a chunk's splats

static size_t fwd_smem(int threads) { return (size_t)(threads / 32) * kFwdPairs * sizeof(FwdPair); }

__device__ __forceinline__ void fwd_stage(FwdPair* Q, int i, const SplatRaw& w, int end) {
  FwdPair& P = Q[i >> 1];
  const int e = i & 1;
  reinterpret_cast<float*>(&P.nx)[e] = -w.xy.x;
  reinterpret_cast<float*>(&P.ny)[e] = -w.xy.y;
  reinterpret_cast<float*>(&P.ca)[e] = __fmul_rn(w.c.x, kPow2A);
  reinterpret_cast<float*>(&P.cb)[e] = __fmul_rn(w.c.y, kPow2B);
  reinterpret_cast<float*>(&P.cc)[e] = __fmul_rn(w.c.z, kPow2A);
  reinterpret_cast<float*>(&P.op)[e] = w.c.w;
  reinterpret_cast<float*>(&P.cr)[e] = w.r;
  reinterpret_cast<float*>(&P.cg)[e] = w.g;
  reinterpret_cast<float*>(&P.cbl)[e] = w.b;
  P.end[e] = end;
}

// One pixel's state.
struct FwdPix {
  float T, C0, C1, C2;
  int last;
  bool done;
};

// A pair against one pixel.
__device__ __forceinline__ void fwd_pair(const FwdPair& P, f32x2 X, f32x2 Y, FwdPix& q) {
  const f32x2 dx = add2(X, P.nx), dy = add2(Y, P.ny);
  const f32x2 p = fma2(fma2(P.ca, dx, mul2(P.cb, dy)), dx, mul2(mul2(P.cc, dy), dy));  // splat_pow2 of both
  const float p0 = lo2(p), p1 = hi2(p);
  const f32x2 og = mul2(P.op, pk2(ex2_approx(p0), ex2_approx(p1)));
  const f32x2 over = add2(og, pk2(-kAlphaMin, -kAlphaMin));  // not negative where alpha >= 1/255
  const bool ok0 = fminf(-p0, lo2(over)) >= 0.f && !q.done, ok1 = fminf(-p1, hi2(over)) >= 0.f && !q.done;
  const float a0 = ok0 ? fminf(kAlphaMax, lo2(og)) : 0.f, a1 = ok1 ? fminf(kAlphaMax, hi2(og)) : 0.f;
  const float T1 = __fmul_rn(q.T, __fsub_rn(1.f, a0)), T2 = __fmul_rn(T1, __fsub_rn(1.f, a1));
  float w0 = __fmul_rn(a0, q.T), w1 = __fmul_rn(a1, T1), Tn = T2;
  int l = ok1 ? P.end[1] : ok0 ? P.end[0] : q.last;
  if (T2 < kTStop) {  // T itself is not below the stop: the walk ends in this pair, once a pixel
    q.done = true;
    w1 = 0.f;
    Tn = T1;
    l = ok0 ? P.end[0] : q.last;
    if (T1 < kTStop) {
      w0 = 0.f;
      Tn = q.T;
      l = q.last;
    }
  }
  q.C0 = __fmaf_rn(w1, hi2(P.cr), __fmaf_rn(w0, lo2(P.cr), q.C0));
  q.C1 = __fmaf_rn(w1, hi2(P.cg), __fmaf_rn(w0, lo2(P.cg), q.C1));
  q.C2 = __fmaf_rn(w1, hi2(P.cbl), __fmaf_rn(w0, lo2(P.cbl), q.C2));
  q.T = Tn;
  q.last = l;
}

// Entry i of the queue against one pixel (where a record is not finite).
__device__ __forceinline__ void fwd_single(const FwdPair* Q, int i, float px, float py, FwdPix& q) {
  const float* P = reinterpret_cast<const float*>(Q + (i >> 1)) + (i & 1);
  const float4 co = make_float4(P[4], P[6], P[8], P[10]);
  float al, G;
  if (q.done || !splat_alpha(co, __fadd_rn(px, P[0]), __fadd_rn(py, P[2]), al, G)) return;
  const float Tn = __fmul_rn(q.T, __fsub_rn(1.f, al));
  if (Tn < kTStop) {
    q.done = true;
    return;
  }
  const float wt = __fmul_rn(al, q.T);
  q.C0 = __fmaf_rn(wt, P[12], q.C0);
  q.C1 = __fmaf_rn(wt, P[14], q.C1);
  q.C2 = __fmaf_rn(wt, P[16], q.C2);
  q.T = Tn;
  q.last = Q[i >> 1].end[i & 1];
}

// Forward of active tile j by a block of one warp per 32 PPL sampled pixels.
template <int PPL>
__device__ __forceinline__ void render_tile_fwd(const RasterArgs& a, int j, FwdPair* sm, float* __restrict__ out_rgb,
                                                float* __restrict__ out_T, int32_t* __restrict__ out_last,
                                                const Ckpt& ck) {
  const unsigned full = 0xffffffffu;
  __shared__ int s_tl;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  FwdPair* Q = sm + warp * kFwdPairs;
  const int t = a.active_tiles ? a.active_tiles[j] : j;
  const int p0 = a.pix_off[j], p1 = a.pix_off[j + 1];
  int s[PPL];
  float px[PPL], py[PPL];
  f32x2 X[PPL], Y[PPL];
  FwdPix q[PPL];
  float4 box = make_float4(INFINITY, INFINITY, -INFINITY, -INFINITY);
#pragma unroll
  for (int u = 0; u < PPL; ++u) {
    s[u] = p0 + 32 * (PPL * warp + u) + lane;
    // a whole tile: the warps take 8 x 4 (8 x 8) blocks of it, which fewer splats reach than bands of rows
    if (p1 - p0 == TGS_TILE_PIX)
      s[u] = p0 + (4 * (PPL * (warp >> 1) + u) + (lane >> 3)) * TGS_TILE + 8 * (warp & 1) + (lane & 7);
    q[u] = FwdPix{1.f, 0.f, 0.f, 0.f, 0, s[u] >= p1};
    px[u] = py[u] = 0.f;
    if (s[u] < p1) {
      const int l = a.pix_idx[s[u]];
      px[u] = (float)((t % a.tiles_x) * TGS_TILE + (l & 15)) + 0.5f;
      py[u] = (float)((t / a.tiles_x) * TGS_TILE + (l >> 4)) + 0.5f;
      box = make_float4(fminf(box.x, px[u]), fminf(box.y, py[u]), fmaxf(box.z, px[u]), fmaxf(box.w, py[u]));
    }
    X[u] = pk2(px[u], px[u]);
    Y[u] = pk2(py[u], py[u]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    box.x = fminf(box.x, __shfl_xor_sync(full, box.x, o));
    box.y = fminf(box.y, __shfl_xor_sync(full, box.y, o));
    box.z = fmaxf(box.z, __shfl_xor_sync(full, box.z, o));
    box.w = fmaxf(box.w, __shfl_xor_sync(full, box.w, o));
  }
  if (ck.tile_last) {  // the tile's longest blended run, for the pieces of the backward
    if (threadIdx.x == 0) s_tl = 0;
    __syncthreads();
  }
  const int2 range = a.ranges[j];
  // a chunk's records are fetched while the chunk before is walked, and the
  // list entries (ids) of the chunk after it
  SplatRaw w;
  int idn = 0;
  if (range.x + lane < range.y) fetch_splat(a, a.vals[range.x + lane], w);
  if (range.x + 32 + lane < range.y) idn = a.vals[range.x + 32 + lane];
  for (int base = range.x; base < range.y; base += 32) {
    bool all = true;
#pragma unroll
    for (int u = 0; u < PPL; ++u) all = all && q[u].done;
    if (__all_sync(full, all)) break;
    if (ck.data) {
      const int c = (base - range.x) / kCkptEvery - 1;  // state in front of this chunk
      if (c >= 0 && c < ck.n_slots) {
#pragma unroll
        for (int u = 0; u < PPL; ++u)
          if (!q[u].done) ck.data[c * ck.stride + s[u]] = make_float4(q[u].T, q[u].C0, q[u].C1, q[u].C2);
      }
    }
    const bool keep = base + lane < range.y && splat_reaches(w.xy, w.c, box);
    const bool fin = !keep || fabsf(w.xy.x) + fabsf(w.xy.y) + fabsf(w.c.x) + fabsf(w.c.y) + fabsf(w.c.z) +
                                      fabsf(w.r) + fabsf(w.g) + fabsf(w.b) <
                                  INFINITY;
    const unsigned m = __ballot_sync(full, keep);
    const bool fast = __all_sync(full, fin);
    __syncwarp();  // the chunk before is no longer read
    const int n = __popc(m);
    if (keep) fwd_stage(Q, __popc(m & ((1u << lane) - 1u)), w, base + lane + 1 - range.x);
    if ((n & 1) && lane == 0) {  // the last pair's second half: a splat that blends nowhere
      SplatRaw z;
      z.xy = make_float2(0.f, 0.f);
      z.c = make_float4(0.f, 0.f, 0.f, 0.f);
      z.r = z.g = z.b = 0.f;
      fwd_stage(Q, n, z, 0);
    }
    __syncwarp();
    if (base + 32 + lane < range.y) fetch_splat(a, idn, w);
    if (base + 64 + lane < range.y) idn = a.vals[base + 64 + lane];
    if (fast) {
      const int pairs = (n + 1) >> 1;
#pragma unroll 2
      for (int i = 0; i < pairs; ++i) {
#pragma unroll
        for (int u = 0; u < PPL; ++u) fwd_pair(Q[i], X[u], Y[u], q[u]);
      }
    } else {  // an infinite or NaN record: splat by splat, so that it stays with the pixels that blend it
      for (int i = 0; i < n; ++i) {
#pragma unroll
        for (int u = 0; u < PPL; ++u) fwd_single(Q, i, px[u], py[u], q[u]);
      }
    }
  }
  int longest = 0;
#pragma unroll
  for (int u = 0; u < PPL; ++u) {
    if (s[u] < p1) {
      out_rgb[3 * s[u]] = q[u].C0 + q[u].T * a.bg[0];
      out_rgb[3 * s[u] + 1] = q[u].C1 + q[u].T * a.bg[1];
      out_rgb[3 * s[u] + 2] = q[u].C2 + q[u].T * a.bg[2];
      out_T[s[u]] = q[u].T;
      out_last[s[u]] = q[u].last;
    }
    longest = max(longest, q[u].last);
  }
  if (ck.tile_last) {
    if (longest > 0) atomicMax(&s_tl, longest);
    __syncthreads();
    if (threadIdx.x == 0) ck.tile_last[j] = s_tl;
  }
}

template <int PPL>
__global__ void __launch_bounds__(TGS_TILE_PIX / PPL) k_render_fwd(RasterArgs a, float* __restrict__ out_rgb,
                                                                   float* __restrict__ out_T,
                                                                   int32_t* __restrict__ out_last, Ckpt ck) {
  extern __shared__ __align__(16) FwdPair fwd_sm[];
  const int j = blockIdx.x;
  if (j >= *a.n_active) return;
  render_tile_fwd<PPL>(a, j, fwd_sm, out_rgb, out_T, out_last, ck);
}

// The same forward with two threads per sampled pixel: a warp holds 16
// pixels twice, and of every 32-position run the first half (lanes 0-15)
// walks positions 0-15 from the pixel's state, exactly as the walk above,
// while the second half (lanes 16-31) walks positions 16-31 at the same time
// from a local (T, C) = (1, 0), without stopping.  The halves then compose,
// (T, C) -> (T T_b, C + T C_b); where the product comes within 1e-5 of the
// stopping transmittance the second half walks its positions again from the
// composed entry state, with the stop, so every stop and n_last is the
// sequential walk's.  The walk of a run is half as long and the block has
// twice the warps; T and C differ from the sequential walk's by the rounding
// of the composition only.
constexpr float kTStopPairMargin = kTStop * (1.f + 1e-5f);

template <bool SELECT>
__device__ __forceinline__ void pair_walk(const Splat* sm, int q0, unsigned mask, float px, float py, int base_pos,
                                          bool can_stop, float& T, float& C0, float& C1, float& C2, int& last,
                                          bool& done) {
  while (mask && !done) {
    int qq[kUnroll];
    float al[kUnroll];
    bool ok[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const bool val = mask != 0u;
      qq[u] = val ? q0 + __ffs(mask) - 1 : q0;
      mask &= mask - 1u;
      const float2 xy = sm[qq[u]].xy;
      float G;
      ok[u] = (SELECT ? splat_alpha_nb(sm[qq[u]].co, __fsub_rn(px, xy.x), __fsub_rn(py, xy.y), al[u], G)
                      : splat_alpha(sm[qq[u]].co, __fsub_rn(px, xy.x), __fsub_rn(py, xy.y), al[u], G)) &&
              val;
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const float Tn = __fmul_rn(T, __fsub_rn(1.f, al[u]));
      const bool stop = ok[u] && !done && can_stop && Tn < kTStop;
      const bool take = ok[u] && !done && !stop;
      done = done || stop;
      const float4 rgb = sm[qq[u]].rgb;
      const float w = al[u] * T;
      C0 = take ? C0 + w * rgb.x : C0;
      C1 = take ? C1 + w * rgb.y : C1;
      C2 = take ? C2 + w * rgb.z : C2;
      T = take ? Tn : T;
      last = take ? base_pos + qq[u] + 1 : last;
    }
  }
}

template <bool SELECT>
__device__ __forceinline__ void render_tile_fwd_pair(const RasterArgs& a, int j, Splat* sm,
                                                     float* __restrict__ out_rgb, float* __restrict__ out_T,
                                                     int32_t* __restrict__ out_last, const Ckpt& ck) {
  const unsigned full = 0xffffffffu;
  const int t = a.active_tiles ? a.active_tiles[j] : j;
  const int p0 = a.pix_off[j], p1 = a.pix_off[j + 1];
  const int lane = threadIdx.x & 31, h = lane >> 4;
  const int s = p0 + 16 * (int)(threadIdx.x >> 5) + (lane & 15);
  const bool has_pix = s < p1;
  float px = 0.f, py = 0.f;
  if (has_pix) {
    const int l = a.pix_idx[s];
    px = (float)((t % a.tiles_x) * TGS_TILE + (l & 15)) + 0.5f;
    py = (float)((t / a.tiles_x) * TGS_TILE + (l >> 4)) + 0.5f;
  }
  const int2 range = a.ranges[j];
  float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
  int last = 0;
  bool done = !has_pix;
  const int B = blockDim.x;
  const float2 band = warp_rows(has_pix, py);
  SplatRaw nxt;
  int idn = 0;
  const int tid = threadIdx.x;
  if (range.x + tid < range.y) fetch_splat(a, a.vals[range.x + tid], nxt);
  if (range.x + B + tid < range.y) idn = a.vals[range.x + B + tid];
  for (int base = range.x; base < range.y; base += B) {
    if (__syncthreads_count(done) == B) break;
    if (base + tid < range.y) finish_splat(nxt, sm[tid]);
    __syncthreads();
    if (base + B + tid < range.y) fetch_splat(a, idn, nxt);
    if (base + 2 * B + tid < range.y) idn = a.vals[base + 2 * B + tid];
    const int cnt = min(B, range.y - base);
    const int base_pos = base - range.x;
    for (int q32 = 0; q32 < cnt; q32 += kCkptEvery) {
      if (ck.data && !done && h == 0) {
        const int c = (base_pos + q32) / kCkptEvery - 1;  // state in front of this run
        if (c >= 0 && c < ck.n_slots) ck.data[c * ck.stride + s] = make_float4(T, C0, C1, C2);
      }
      const int qe = min(cnt, q32 + kCkptEvery);
      bool in_l = false;
      if (q32 + lane < qe) {
        const float2 yr = sm[q32 + lane].yr;
        in_l = yr.y >= band.x && yr.x <= band.y;
      }
      const unsigned m32 = __ballot_sync(full, in_l);
      const unsigned hm = h ? (m32 >> 16) : (m32 & 0xFFFFu);
      const int q0 = q32 + 16 * h;
      // half 0: the pixel's state, with the stop; half 1: a local state from (1, 0)
      float Tw = h ? 1.f : T, W0 = h ? 0.f : C0, W1 = h ? 0.f : C1, W2 = h ? 0.f : C2;
      int lw = h ? 0 : last;
      bool dw = done;
      pair_walk<SELECT>(sm, q0, hm, px, py, base_pos, h == 0, Tw, W0, W1, W2, lw, dw);
      __syncwarp();
      const float oT = __shfl_xor_sync(full, Tw, 16), o0 = __shfl_xor_sync(full, W0, 16),
                  o1 = __shfl_xor_sync(full, W1, 16), o2 = __shfl_xor_sync(full, W2, 16);
      const int ol = __shfl_xor_sync(full, lw, 16);
      const bool od = __shfl_xor_sync(full, (int)dw, 16) != 0;
      // A: the first half's state (exact), Bh: the second half's local walk
      const float aT = h ? oT : Tw, a0 = h ? o0 : W0, a1 = h ? o1 : W1, a2 = h ? o2 : W2;
      const int al_ = h ? ol : lw;
      const bool ad = h ? od : dw;
      const float bT = h ? Tw : oT, b0 = h ? W0 : o0, b1 = h ? W1 : o1, b2 = h ? W2 : o2;
      const int bl = h ? lw : ol;
      // stopped in the first half, or nothing blended in the second: the first half's state
      const bool first = ad || bl == 0;
      const float Tc = __fmul_rn(aT, bT);
      // the stop may lie in the second half: it walks its positions again from the exact entry state
      const bool again = !first && Tc < kTStopPairMargin;
      if (__any_sync(full, again)) {  // warp-uniform, so that every lane takes part in the shuffles
        float rT = aT, r0 = a0, r1 = a1, r2 = a2;
        int rl = al_;
        bool rd = false;
        if (h && again) pair_walk<false>(sm, q0, hm, px, py, base_pos, true, rT, r0, r1, r2, rl, rd);
        __syncwarp();
        const int src = (lane & 15) + 16;
        rT = __shfl_sync(full, rT, src);
        r0 = __shfl_sync(full, r0, src);
        r1 = __shfl_sync(full, r1, src);
        r2 = __shfl_sync(full, r2, src);
        rl = __shfl_sync(full, rl, src);
        rd = __shfl_sync(full, (int)rd, src) != 0;
        if (again) {
          T = rT; C0 = r0; C1 = r1; C2 = r2; last = rl; done = rd;
          continue;
        }
      }
      if (first) {
        T = aT; C0 = a0; C1 = a1; C2 = a2; last = al_; done = ad;
      } else {
        T = Tc;
        C0 = a0 + aT * b0;
        C1 = a1 + aT * b1;
        C2 = a2 + aT * b2;
        last = bl;
      }
    }
  }
  if (has_pix && h == 0) {
    out_rgb[3 * s] = C0 + T * a.bg[0];
    out_rgb[3 * s + 1] = C1 + T * a.bg[1];
    out_rgb[3 * s + 2] = C2 + T * a.bg[2];
    out_T[s] = T;
    out_last[s] = last;
  }
  if (ck.tile_last) {
    __shared__ int s_tl;
    __syncthreads();
    if (threadIdx.x == 0) s_tl = 0;
    __syncthreads();
    if (last > 0 && h == 0) atomicMax(&s_tl, last);
    __syncthreads();
    if (threadIdx.x == 0) ck.tile_last[j] = s_tl;
  }
}

template <bool SELECT>
__global__ void k_render_fwd_pair(RasterArgs a, float* __restrict__ out_rgb, float* __restrict__ out_T,
                                  int32_t* __restrict__ out_last, Ckpt ck) {
  extern __shared__ Splat sm[];
  const int j = blockIdx.x;
  if (j >= *a.n_active) return;
  render_tile_fwd_pair<SELECT>(a, j, sm, out_rgb, out_T, out_last, ck);
}

// ---------------------------------------------------------------------------
// Split forward (few active tiles: a sparse step).  One block per active
// tile holds NW groups of G threads, one thread per sampled pixel in each
// group.  In round r, group g walks run r NW + g of the tile's list (the 32
// positions [32 (r NW + g), 32 (r NW + g + 1))) from a local transmittance of
// 1, so the NW runs of a round are walked at once and the tile's walk is NW
// times shorter.  A run walked from T = 1 to local transmittance T_l and
// local colour D_l turns the state (T, C) in front of it into
// (T T_l, C + T D_l); the groups' results are composed per pixel in list
// order through shared memory.  The walk stops in the first run where the
// composed product falls below the stopping transmittance, or whose local
// walk stopped by itself (T_l (1 - alpha) < 1e-4 implies the same for the
// global T <= T_l); that run is walked again by its group from its true entry
// state to find the exact stopping splat.  Checkpoints (the state at the end
// of each run) are written from the composed state, as the sequential walk
// writes them, so the backward is unchanged.  The composition rounds
// differently from the sequential product (one more rounding per run); when
// the product lands within rounding of the stopping value and the re-walk
// does not stop, the walk ends at the end of that run.  Rounds repeat until
// every pixel has stopped or the list ends, so work past the tile's last
// stopping point is bounded by one round.
// ---------------------------------------------------------------------------
constexpr int kLocalStop = 64;  // flag bit beside the run-local last position (0..32)

__device__ __forceinline__ void compose_run(float& T, float& C0, float& C1, float& C2, const float4& e) {
  C0 = __fmaf_rn(T, e.y, C0);
  C1 = __fmaf_rn(T, e.z, C1);
  C2 = __fmaf_rn(T, e.w, C2);
  T = __fmul_rn(T, e.x);
}

template <int NW>
__global__ void k_render_fwd_split(RasterArgs a, float* __restrict__ out_rgb, float* __restrict__ out_T,
                                   int32_t* __restrict__ out_last, Ckpt ck) {
  extern __shared__ float4 smem_f4[];
  __shared__ int s_tl;
  const int j = blockIdx.x;
  if (j >= *a.n_active) return;
  const int G = blockDim.x / NW;
  Splat* sp = reinterpret_cast<Splat*>(smem_f4);           // [NW][32]
  float4* loc = reinterpret_cast<float4*>(sp + NW * 32);   // [NW][G] (T_l, D_l)
  float4* rec = loc + NW * G;                              // [NW][G] state after a stopping run
  int* lastl = reinterpret_cast<int*>(rec + NW * G);       // [NW][G] local last | kLocalStop
  int* rec_last = lastl + NW * G;                          // [NW][G]
  const int g = threadIdx.x / G, i = threadIdx.x - g * G;
  const int t = a.active_tiles ? a.active_tiles[j] : j;
  const int p0 = a.pix_off[j], p1 = a.pix_off[j + 1];
  const bool has_pix = p0 + i < p1;
  const int s = p0 + i;
  float px = 0.f, py = 0.f;
  if (has_pix) {
    const int l = a.pix_idx[s];
    px = (float)((t % a.tiles_x) * TGS_TILE + (l & 15)) + 0.5f;
    py = (float)((t / a.tiles_x) * TGS_TILE + (l >> 4)) + 0.5f;
  }
  const int2 range = a.ranges[j];
  const int L = range.y - range.x;
  const int n_runs = (L + kCkptEvery - 1) / kCkptEvery;
  // the running state of pixel i in front of the current round (the same in every group)
  float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
  int last = 0;
  bool done = !has_pix;
  const Splat* S = sp + 32 * g;
  Splat nxt;
  if (i < 32 && 32 * g + i < L) load_splat(a, range.x + 32 * g + i, nxt);
  for (int r0 = 0; r0 < n_runs; r0 += NW) {
    const int run = r0 + g;
    // the previous round's reads of sp ended before its second barrier
    if (i < 32 && 32 * run + i < L) sp[32 * g + i] = nxt;
    if (__syncthreads_count(done) == (int)blockDim.x) break;
    if (i < 32 && 32 * (run + NW) + i < L) load_splat(a, range.x + 32 * (run + NW) + i, nxt);
    // 1. the group's run from a local T = 1 (alphas of kUnroll splats together, blend with selects)
    const int cnt = min(kCkptEvery, L - 32 * run);
    float Tl = 1.f, D0 = 0.f, D1 = 0.f, D2 = 0.f;
    int ll = 0;
    bool lstop = false;
    if (!done && cnt > 0) {
      for (int q0 = 0; q0 < cnt && !lstop; q0 += kUnroll) {
        float al[kUnroll];
        bool ok[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const float2 xy = S[q0 + u].xy;
          float Gv;
          ok[u] = splat_alpha_nb(S[q0 + u].co, __fsub_rn(px, xy.x), __fsub_rn(py, xy.y), al[u], Gv) &&
                  q0 + u < cnt;
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const float Tn = __fmul_rn(Tl, __fsub_rn(1.f, al[u]));
          const bool stop = ok[u] && !lstop && Tn < kTStop;
          const bool take = ok[u] && !lstop && !stop;
          lstop = lstop || stop;
          const float4 rgb = S[q0 + u].rgb;
          const float w = al[u] * Tl;
          D0 = take ? D0 + w * rgb.x : D0;
          D1 = take ? D1 + w * rgb.y : D1;
          D2 = take ? D2 + w * rgb.z : D2;
          Tl = take ? Tn : Tl;
          ll = take ? q0 + u + 1 : ll;
        }
      }
    }
    loc[g * G + i] = make_float4(Tl, D0, D1, D2);
    lastl[g * G + i] = ll | (lstop ? kLocalStop : 0);
    __syncthreads();
    // 2. the state in front of this group's run; its checkpoint, or the exact stop inside it
    if (!done && cnt > 0) {
      float T2 = T, E0 = C0, E1 = C1, E2 = C2;
      int l2 = last;
      bool before = false;
      for (int h = 0; h < g; ++h) {
        const float4 e = loc[h * G + i];
        const int lh = lastl[h * G + i];
        if ((lh & kLocalStop) || __fmul_rn(T2, e.x) < kTStop) {
          before = true;
          break;
        }
        compose_run(T2, E0, E1, E2, e);
        if (lh) l2 = 32 * (r0 + h) + lh;
      }
      if (!before) {
        if (lstop || __fmul_rn(T2, Tl) < kTStop) {
          for (int q = 0; q < cnt; ++q) {  // the stopping run again, from its entry state
            const Splat& sq = S[q];
            float al, Gv;
            if (!splat_alpha(sq.co, __fsub_rn(px, sq.xy.x), __fsub_rn(py, sq.xy.y), al, Gv)) continue;
            const float Tn = __fmul_rn(T2, __fsub_rn(1.f, al));
            if (Tn < kTStop) break;
            const float w = al * T2;
            E0 += w * sq.rgb.x;
            E1 += w * sq.rgb.y;
            E2 += w * sq.rgb.z;
            T2 = Tn;
            l2 = 32 * run + q + 1;
          }
          rec[g * G + i] = make_float4(T2, E0, E1, E2);
          rec_last[g * G + i] = l2;
        } else if (ck.data && run < ck.n_slots) {
          compose_run(T2, E0, E1, E2, make_float4(Tl, D0, D1, D2));
          ck.data[run * ck.stride + s] = make_float4(T2, E0, E1, E2);  // in front of position 32 (run + 1)
        }
      }
    }
    __syncthreads();
    // 3. the running state over the whole round (every group the same)
    if (!done) {
#pragma unroll
      for (int h = 0; h < NW; ++h) {
        if (r0 + h >= n_runs) break;
        const float4 e = loc[h * G + i];
        const int lh = lastl[h * G + i];
        if ((lh & kLocalStop) || __fmul_rn(T, e.x) < kTStop) {
          const float4 q = rec[h * G + i];
          T = q.x;
          C0 = q.y;
          C1 = q.z;
          C2 = q.w;
          last = rec_last[h * G + i];
          done = true;
          break;
        }
        compose_run(T, C0, C1, C2, e);
        if (lh) last = 32 * (r0 + h) + lh;
      }
    }
  }
  if (g == 0 && has_pix) {
    out_rgb[3 * s] = C0 + T * a.bg[0];
    out_rgb[3 * s + 1] = C1 + T * a.bg[1];
    out_rgb[3 * s + 2] = C2 + T * a.bg[2];
    out_T[s] = T;
    out_last[s] = last;
  }
  if (ck.tile_last) {
    __syncthreads();
    if (threadIdx.x == 0) s_tl = 0;
    __syncthreads();
    if (g == 0 && last > 0) atomicMax(&s_tl, last);
    __syncthreads();
    if (threadIdx.x == 0) ck.tile_last[j] = s_tl;
  }
}

template <int NW>
size_t split_smem_bytes(int G) {
  return NW * 32 * sizeof(Splat) + (size_t)NW * G * (2 * sizeof(float4) + 2 * sizeof(int));
}

// Where the backward also accumulates the error back-projection statistics of
// Sec. 3.8 (Eq. 12): the per-pixel error e (from the loss) and the per-
// Gaussian rows (E, W, D, 0) they are added to.
struct StatsK {
  const float* err;
  float4* stats;
};

// ---------------------------------------------------------------------------
// The compositing adjoint.  A warp takes one item: a group of at most 32 PPL
// sampled pixels of a tile (PPL per lane) and a piece of the tile's list.  It
// walks the piece from the back in chunks of 32 positions, keeps the splats
// that can reach the group's rectangle, and replays them two at a time, in
// packed fp32 arithmetic (the two splats of a pair in the halves of a
// register pair, one issue slot per operation): only a pixel's transmittance
// T and the light from behind it, R = sum_{j behind} w_j c_j . g + T_final
// bg . g, go through the two one after the other:
//   T_k = T / (1 - alpha),  dL/dalpha = T_k c . g - R / (1 - alpha),
//   R += w c . g  (w = alpha T_k).
// The lane sums a pair's adjoints over its pixels in registers; one warp
// reduction then serves both splats (22 shuffles and one atomic instruction
// a pair), so the work per splat and 32 pixels falls with PPL.  Warps never
// wait on each other.
//
// Where a piece ends: a pixel whose last blended splat lies in the piece
// starts from (T_final, T_final bg . g); one whose walk goes on past it from
// the forward's checkpoint at the piece's back edge, R = (out - C) . g.
// Without checkpoints a tile is one piece.
//
// Bound: instruction issue and the latency of the chain alpha -> T -> sums ->
// reduction (500k Gaussians, 1280x720: 54-68 % issue, 10-16 warps an SM).
// Against one splat at a time with scalar arithmetic and a reduction per
// splat and warp of pixels (and, without checkpoints, a block per tile with
// shared-memory atomics): 720 tiles of 85 pixels 67 -> 54 us, 3600 of 25
// pixels 155 -> 132, the dense view 728 -> 421, eight views of 3M Gaussians
// 1738 -> 1043.  Measured beside it and slower: pixels streamed through lanes
// that hold the splats (no reduction, but long serial chains): 98, 211 and 483
// us for the first three.
// Against 64 bits the nine columns are 1.4e-7 to 4.4e-7 of their norm off at 26 to
// 495 blended splats a pixel; the light behind as a sum, in place of a colour
// carried from splat to splat, costs up to 1.3 times in the first six.
//
// STATS: the same replay also sums, per splat, Eq. 12's e w, w and D w over
// the pixels (e the pixel's error, D the conic Mahalanobis distance of the
// pixel centre) into its statistics row.
// ---------------------------------------------------------------------------
constexpr int kBwdPpl = 4;      // most pixels a lane
// One warp a block: items differ in length (empty ones, long lists), and a
// block of four holds its slots until its longest is done (sparse step: 66 us
// with four warps a block, 57 with one).  20 blocks an SM: 96 registers.  Four
// pixels a lane spill 64 bytes a thread there, three none; with statistics 140
// and 104; in the batched kernel 152 and none, with statistics 228 and 88.
constexpr int kBwdBlocksPerSm = 20;

// Two kept splats as the replay reads them (element e in half e).
struct __align__(16) BwdPair {
  f32x2 nx, ny;      // minus the centre
  f32x2 ca, cb;      // the pre-scaled conic
  f32x2 cc, op;      // and the opacity
  f32x2 cr, cg;      // colour
  f32x2 cbl;
  f32x2 np;          // minus (position from the chunk's first + 1/2)
  float cf[2][8];    // factors of the reduced sums, in the gradient row's order
  float bo[2];       // cross factor of the centre's two sums
  int id[2];
};
constexpr int kBwdPairs = 17;  // a chunk's 32 splats and one left over

// Entry i of the warp's queue.
__device__ __forceinline__ void bwd_stage(BwdPair* Q, int i, const SplatRaw& w, float pos) {
  BwdPair& P = Q[i >> 1];
  const int e = i & 1;
  reinterpret_cast<float*>(&P.nx)[e] = -w.xy.x;
  reinterpret_cast<float*>(&P.ny)[e] = -w.xy.y;
  reinterpret_cast<float*>(&P.ca)[e] = __fmul_rn(w.c.x, kPow2A);
  reinterpret_cast<float*>(&P.cb)[e] = __fmul_rn(w.c.y, kPow2B);
  reinterpret_cast<float*>(&P.cc)[e] = __fmul_rn(w.c.z, kPow2A);
  reinterpret_cast<float*>(&P.op)[e] = w.c.w;
  reinterpret_cast<float*>(&P.cr)[e] = w.r;
  reinterpret_cast<float*>(&P.cg)[e] = w.g;
  reinterpret_cast<float*>(&P.cbl)[e] = w.b;
  reinterpret_cast<float*>(&P.np)[e] = -(pos + 0.5f);
  P.id[e] = w.id;
  // sums of dL/dpower times dx, dy, dx^2, dx dy, dy^2, 1 (power = -(a dx^2 +
  // c dy^2)/2 - b dx dy, dx = px - x): dL/dx = a m1 + b m2, dL/dy = c m2 + b m1,
  // dL/da = -m3 / 2, dL/db = -m4, dL/dc = -m5 / 2, dL/do = m0 / o, by the rounded
  // reciprocal: dL/do is then within 3 % of as near to 64 bits as the sum of
  // dL/dalpha G itself, for two selections less a pair and pixel (dense view 861
  // us a step against 867)
  const float o = w.c.w;
  float4* f = reinterpret_cast<float4*>(P.cf[e]);
  f[0] = make_float4(w.c.x, w.c.z, -0.5f, -1.f);
  f[1] = make_float4(-0.5f, o > 0.f ? __frcp_rn(o) : 0.f, 1.f, 1.f);
  P.bo[e] = w.c.y;
}

// One pair against the lane's pixels, and its sums into the gradient rows.
// CAPPED: an opacity reaches the cap on alpha.  Where a splat does not blend,
// sums and states change by zeros, so everything has to be finite; and T is
// multiplied by rcp_approx(-1) twice, which has to be exactly -1 (the PTX
// document promises it to one unit only; tested over thousands of skipped splats).
template <int PPL, bool CAPPED, bool STATS>
__device__ __forceinline__ void bwd_pair(const BwdPair& P, const f32x2 (&px)[PPL], const f32x2 (&py)[PPL],
                                         const f32x2 (&g0)[PPL], const f32x2 (&g1)[PPL], const f32x2 (&g2)[PPL],
                                         const float (&err)[STATS ? PPL : 1], const f32x2 (&last)[PPL],
                                         float (&T)[PPL], float (&R)[PPL], float* __restrict__ grad2d,
                                         float4* __restrict__ stats) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const f32x2 nx = P.nx, ny = P.ny, ca = P.ca, cb = P.cb, cc = P.cc, op = P.op, cr = P.cr, cg = P.cg, cbl = P.cbl;
  const f32x2 np = P.np;
  const f32x2 mone = pk2(-1.f, -1.f), namin = pk2(-kAlphaMin, -kAlphaMin);
  f32x2 v[9], sv[3];
#pragma unroll
  for (int u = 0; u < PPL; ++u) {
    const f32x2 dx = add2(px[u], nx), dy = add2(py[u], ny);
    const f32x2 p = fma2(fma2(ca, dx, mul2(cb, dy)), dx, mul2(mul2(cc, dy), dy));  // splat_pow2 of both
    const float p0 = lo2(p), p1 = hi2(p);
    const float G0 = ex2_approx(p0), G1 = ex2_approx(p1);
    const f32x2 og = mul2(op, pk2(G0, G1));
    // blends where power <= 0, alpha >= 1/255 and the pixel's walk came past the splat
    const f32x2 am_ = add2(og, namin), ahead = add2(last[u], np);
    const bool ok0 = min3(-p0, lo2(am_), lo2(ahead)) >= 0.f, ok1 = min3(-p1, hi2(am_), hi2(ahead)) >= 0.f;
    float a0 = ok0 ? lo2(og) : 0.f, a1 = ok1 ? hi2(og) : 0.f;
    if (CAPPED) {
      a0 = ok0 ? fminf(kAlphaMax, lo2(og)) : 0.f;
      a1 = ok1 ? fminf(kAlphaMax, hi2(og)) : 0.f;
    }
    const f32x2 am = pk2(a0, a1);
    const f32x2 cdg = fma2(cbl, g2[u], fma2(cg, g1[u], mul2(cr, g0[u])));  // c . g
    const f32x2 d = add2(am, mone);  // -(1 - alpha), at most -0.01
    const float i0 = rcp_approx(lo2(d)), i1 = rcp_approx(hi2(d));
    const float T0 = -T[u] * i0, T1 = -T0 * i1;  // transmittance in front of each
    const f32x2 Tv = pk2(T0, T1);
    const f32x2 w = mul2(am, Tv);
    const float R0 = R[u], R1 = __fmaf_rn(lo2(w), lo2(cdg), R0);
    const f32x2 da = fma2(pk2(R0, R1), pk2(i0, i1), mul2(Tv, cdg));  // dL/dalpha
    // alpha dL/dalpha, the gradient of the power and, over the opacity, of the
    // opacity; a capped alpha passes none
    const f32x2 t = mul2(da, CAPPED ? pk2(a0 < kAlphaMax ? a0 : 0.f, a1 < kAlphaMax ? a1 : 0.f) : am);
    T[u] = T1;
    R[u] = __fmaf_rn(hi2(w), hi2(cdg), R1);
    const f32x2 tx = mul2(t, dx), ty = mul2(t, dy);
    v[0] = u == 0 ? tx : add2(v[0], tx);
    v[1] = u == 0 ? ty : add2(v[1], ty);
    v[2] = u == 0 ? mul2(tx, dx) : fma2(tx, dx, v[2]);
    v[3] = u == 0 ? mul2(tx, dy) : fma2(tx, dy, v[3]);
    v[4] = u == 0 ? mul2(ty, dy) : fma2(ty, dy, v[4]);
    v[5] = u == 0 ? t : add2(v[5], t);
    v[6] = u == 0 ? mul2(w, g0[u]) : fma2(w, g0[u], v[6]);
    v[7] = u == 0 ? mul2(w, g1[u]) : fma2(w, g1[u], v[7]);
    v[8] = u == 0 ? mul2(w, g2[u]) : fma2(w, g2[u], v[8]);
    if (STATS) {
      // a dx^2 + 2 b dx dy + c dy^2 = -2 power = -2 ln(2) p
      const float D0 = sqrtf(fmaxf(p0 * kInvA, 0.f)), D1 = sqrtf(fmaxf(p1 * kInvA, 0.f));
      const f32x2 ee = pk2(err[u], err[u]);
      sv[0] = u == 0 ? mul2(w, ee) : fma2(w, ee, sv[0]);
      sv[1] = u == 0 ? w : add2(w, sv[1]);
      sv[2] = u == 0 ? mul2(w, pk2(D0, D1)) : fma2(w, pk2(D0, D1), sv[2]);
    }
  }
  // the sums over the warp: splat 0's to lanes 0-15, splat 1's to 16-31, then
  // component k to lanes 2 k and 2 k + 1 of the half, component 8 to all of it
  const bool up = lane & 16;
  float r[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const float keep = up ? hi2(v[k]) : lo2(v[k]), send = up ? lo2(v[k]) : hi2(v[k]);
    r[k] = keep + __shfl_xor_sync(full, send, 16);
  }
  float b4[4], b2[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool h = lane & 8;
    const float keep = h ? r[4 + k] : r[k], send = h ? r[k] : r[4 + k];
    b4[k] = keep + __shfl_xor_sync(full, send, 8);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool h = lane & 4;
    const float keep = h ? b4[2 + k] : b4[k], send = h ? b4[k] : b4[2 + k];
    b2[k] = keep + __shfl_xor_sync(full, send, 4);
  }
  const bool h2 = lane & 2;
  float s = (h2 ? b2[1] : b2[0]) + __shfl_xor_sync(full, h2 ? b2[0] : b2[1], 2);
  s += __shfl_xor_sync(full, s, 1);
  float s8 = r[8];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) s8 += __shfl_xor_sync(full, s8, o);
  const int e = lane >> 4, k = (lane >> 1) & 7;
  const float other = __shfl_xor_sync(full, s, 2);  // the other sum of the centre (k = 0, 1)
  float val = P.cf[e][k] * s;
  if (k < 2) val += P.bo[e] * other;
  float* gp = grad2d + 12 * (size_t)P.id[e] + k;
  if (lane & 1) {
    gp += 8;
    val = k == 0 ? s8 : 0.f;
  }
  if (val != 0.f) atomicAdd(gp, val);
  if (STATS) {
    float z[3];
#pragma unroll
    for (int k3 = 0; k3 < 3; ++k3) {
      const float keep = up ? hi2(sv[k3]) : lo2(sv[k3]), send = up ? lo2(sv[k3]) : hi2(sv[k3]);
      z[k3] = keep + __shfl_xor_sync(full, send, 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) z[k3] += __shfl_xor_sync(full, z[k3], o);
    }
    if ((lane & 15) == 0 && z[1] != 0.f)
      red_add_v4(reinterpret_cast<float*>(stats + P.id[e]), z[0], z[1], z[2], 0.f);
  }
}

// The rest of an item (list entries [first, top) from the back) where a
// gradient, a colour or a state is infinite or NaN: splat by splat, and only
// where a pixel blends one, so that such values stay with their own pixels
// and splats.  TR: T and R of the group's pixels.
template <bool STATS>
__device__ __noinline__ void bwd_rest_safe(const RasterArgs& a, int j, int p0, int p1, int lo_pos, int start, int first,
                                           int top, const float2* TR, const int32_t* __restrict__ n_last,
                                           const float* __restrict__ dL_drgb, float* __restrict__ grad2d,
                                           const StatsK& st) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, t = a.active_tiles ? a.active_tiles[j] : j;
  const float ox = (float)((t % a.tiles_x) * TGS_TILE) + 0.5f, oy = (float)((t / a.tiles_x) * TGS_TILE) + 0.5f;
  for (int s0 = p0; s0 < p1; s0 += 32) {
    const int s = s0 + lane;
    const bool has = s < p1;
    const int last = has ? n_last[s] : 0, l = has ? a.pix_idx[s] : 0;
    const float px = ox + (float)(l & 15), py = oy + (float)(l >> 4);
    const float g0 = has ? dL_drgb[3 * (size_t)s] : 0.f, g1 = has ? dL_drgb[3 * (size_t)s + 1] : 0.f,
                g2 = has ? dL_drgb[3 * (size_t)s + 2] : 0.f;
    const float err = STATS && has ? st.err[s] : 0.f;
    float T = TR[s - p0].x, R = TR[s - p0].y;
    for (int k = top - 1; k >= first; --k) {
      Splat sp;
      load_splat(a, k, sp);
      float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, z[3] = {0.f, 0.f, 0.f};
      const float dx = __fsub_rn(px, sp.xy.x), dy = __fsub_rn(py, sp.xy.y);
      float al, G;
      const bool ok = last > lo_pos && k - start < last && sp.yr.y >= py && sp.yr.x <= py &&
                      splat_alpha(sp.co, dx, dy, al, G);
      if (ok) {
        const float inv = rcp_approx(1.f - al), cdg = sp.rgb.x * g0 + sp.rgb.y * g1 + sp.rgb.z * g2;
        T *= inv;
        const float w = al * T, da = T * cdg - R * inv;
        R += w * cdg;
        v[6] = w * g0;
        v[7] = w * g1;
        v[8] = w * g2;
        if (al < kAlphaMax) {
          const float tt = da * al, tx = tt * dx, ty = tt * dy;
          v[0] = tx;
          v[1] = ty;
          v[2] = tx * dx;
          v[3] = tx * dy;
          v[4] = ty * dy;
          v[5] = da * G;
        }
        z[0] = err * w;
        z[1] = w;
        z[2] = w * sqrtf(fmaxf(splat_pow2(sp.co, dx, dy) * kInvA, 0.f));
      }
      if (!__any_sync(full, ok)) continue;
      for (int c = 0; c < 9; ++c) v[c] = warp_sum(v[c]);
      const int id = __float_as_int(sp.rgb.w);
      const float A = sp.co.x * kInvA, Bc = sp.co.y * kInvB, Cc = sp.co.z * kInvA;
      if (lane == 0) {
        float* gp = grad2d + 12 * (size_t)id;
        red_add_v4(gp, A * v[0] + Bc * v[1], Cc * v[1] + Bc * v[0], -0.5f * v[2], -v[3]);
        red_add_v4(gp + 4, -0.5f * v[4], v[5], v[6], v[7]);
        atomicAdd(gp + 8, v[8]);
      }
      if (STATS) {
        for (int c = 0; c < 3; ++c) z[c] = warp_sum(z[c]);
        if (lane == 0) red_add_v4(reinterpret_cast<float*>(st.stats + id), z[0], z[1], z[2], 0.f);
      }
    }
  }
}

// How a launch divides its tiles into items: `groups` of at most `gpx` pixels,
// and `pieces` of `span` checkpoint intervals (the last one open); one piece
// without checkpoints.
struct BwdSplit {
  int groups, gpx, pieces, span;
};

// Item (tile j, q = piece * groups + group); false where nothing blended in it.
template <int PPL, bool STATS>
__device__ __forceinline__ bool render_item_bwd(const RasterArgs& a, int j, int q, const BwdSplit& sp, BwdPair* Q,
                                                const float* __restrict__ T_final, const int32_t* __restrict__ n_last,
                                                const float* __restrict__ dL_drgb, float* __restrict__ grad2d,
                                                const Ckpt& ck, const StatsK& st) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int c = q / sp.groups, grp = q - c * sp.groups;
  const int lo_pos = c * sp.span * kCkptEvery;
  const bool open = c == sp.pieces - 1;
  const int hi_edge = open ? INT_MAX : lo_pos + sp.span * kCkptEvery;
  if (ck.tile_last && ck.tile_last[j] <= lo_pos) return false;  // warp-uniform
  const int p0 = a.pix_off[j] + grp * sp.gpx, p1 = min(a.pix_off[j + 1], p0 + sp.gpx);
  const int2 range = a.ranges[j];
  const int first = range.x + lo_pos;
  // the loads of the first chunk's list entries go out with the pixels' own
  int top = open ? 0 : range.x + hi_edge;
  int id = !open && top - 1 - lane < range.y ? a.vals[top - 1 - lane] : -1;
  const int t = a.active_tiles ? a.active_tiles[j] : j;
  const float ox = (float)((t % a.tiles_x) * TGS_TILE) + 0.5f, oy = (float)((t / a.tiles_x) * TGS_TILE) + 0.5f;
  int last[PPL], hi_pos = 0;
  f32x2 px[PPL], py[PPL], g0[PPL], g1[PPL], g2[PPL];
  float T[PPL], R[PPL], err[STATS ? PPL : 1];
  bool finite = true;
  float4 box = make_float4(INFINITY, INFINITY, -INFINITY, -INFINITY);
#pragma unroll
  for (int u = 0; u < PPL; ++u) {
    const int s = p0 + 32 * u + lane;
    const bool in = s < p1;
    last[u] = in ? n_last[s] : 0;
    const int l = in ? a.pix_idx[s] : 0;
    float d0 = in ? dL_drgb[3 * (size_t)s] : 0.f, d1 = in ? dL_drgb[3 * (size_t)s + 1] : 0.f,
          d2 = in ? dL_drgb[3 * (size_t)s + 2] : 0.f;
    T[u] = in ? T_final[s] : 1.f;
    if (STATS) err[u] = in ? st.err[s] : 0.f;
    const float x = ox + (float)(l & 15), y = oy + (float)(l >> 4);
    if (last[u] <= lo_pos) {  // this pixel blended nothing in the piece
      last[u] = 0;
      d0 = d1 = d2 = 0.f;
      T[u] = 1.f;
      if (STATS) err[u] = 0.f;
    } else {
      box = make_float4(fminf(box.x, x), fminf(box.y, y), fmaxf(box.z, x), fmaxf(box.w, y));
    }
    R[u] = T[u] * (a.bg[0] * d0 + a.bg[1] * d1 + a.bg[2] * d2);
    if (last[u] > hi_edge) {
      const float4 k4 = ck.data[((c + 1) * sp.span - 1) * ck.stride + s];  // in front of position hi_edge
      T[u] = k4.x;
      R[u] = (ck.rgb[3 * (size_t)s] - k4.y) * d0 + (ck.rgb[3 * (size_t)s + 1] - k4.z) * d1 +
             (ck.rgb[3 * (size_t)s + 2] - k4.w) * d2;
    }
    if (STATS) finite = finite && fabsf(err[u]) < INFINITY;
    finite = finite && fabsf(d0) + fabsf(d1) + fabsf(d2) + fabsf(R[u]) + fabsf(T[u]) < INFINITY;
    hi_pos = max(hi_pos, min(last[u], hi_edge));
    px[u] = pk2(x, x);
    py[u] = pk2(y, y);
    g0[u] = pk2(d0, d0);
    g1[u] = pk2(d1, d1);
    g2[u] = pk2(d2, d2);
  }
  hi_pos = __reduce_max_sync(full, hi_pos);
  if (hi_pos <= lo_pos) return false;
  if (open) {
    top = range.x + hi_pos;
    id = top - 1 - lane >= first ? a.vals[top - 1 - lane] : -1;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    box.x = fminf(box.x, __shfl_xor_sync(full, box.x, o));
    box.y = fminf(box.y, __shfl_xor_sync(full, box.y, o));
    box.z = fmaxf(box.z, __shfl_xor_sync(full, box.z, o));
    box.w = fmaxf(box.w, __shfl_xor_sync(full, box.w, o));
  }
  int qn = 0, left = 0;  // left: list entry of the splat left over in the queue
  for (; top > first; top -= 32) {
    // positions count from the chunk's first, so that they stay small in floats
    const int base = top - 32, k = top - 1 - lane;
    f32x2 lastf[PPL];
#pragma unroll
    for (int u = 0; u < PPL; ++u) {
      const float l = (float)max(min(last[u] - (base - range.x), 64), 0);
      lastf[u] = pk2(l, l);
    }
    SplatRaw w;
    bool keep = false;
    if (id >= 0 && k < range.x + hi_pos) {
      fetch_splat(a, id, w);
      keep = splat_reaches(w.xy, w.c, box);
      // a record that is not finite takes the item off the fast path
      finite = finite && (!keep || fabsf(w.xy.x) + fabsf(w.xy.y) + fabsf(w.c.x) + fabsf(w.c.y) + fabsf(w.c.z) +
                                           fabsf(w.c.w) + fabsf(w.r) + fabsf(w.g) + fabsf(w.b) <
                                       INFINITY);
    }
    // the next chunk's, ahead of this one's replay (a closed piece may begin past the list's end)
    id = k - 32 >= first && k - 32 < range.y ? a.vals[k - 32] : -1;
    if (!__all_sync(full, finite)) {
      float2* TR = reinterpret_cast<float2*>(Q);
      __syncwarp();
#pragma unroll
      for (int u = 0; u < PPL; ++u) TR[32 * u + lane] = make_float2(T[u], R[u]);
      __syncwarp();
      bwd_rest_safe<STATS>(a, j, p0, p1, lo_pos, range.x, first, qn ? left + 1 : min(top, range.y), TR, n_last, dL_drgb, grad2d, st);
      return true;
    }
    const unsigned m = __ballot_sync(full, keep);
    if (m) left = top - 1 - (31 - __clz(m));  // the front-most one kept
    if (keep) bwd_stage(Q, qn + __popc(m & ((1u << lane) - 1u)), w, (float)(k - base));
    qn += __popc(m);
    // the second half of the last pair, or of one left over for a whole chunk
    // (a position stays below 64): a splat that blends nowhere
    const bool end = top - 32 <= first || m == 0u;
    if (end && (qn & 1)) {
      if (lane == 0) {
        SplatRaw z;
        z.xy = make_float2(0.f, 0.f);
        z.c = make_float4(0.f, 0.f, 0.f, 0.f);
        z.r = z.g = z.b = 0.f;
        z.id = 0;
        bwd_stage(Q, qn, z, 1e9f);
      }
      ++qn;
    }
    __syncwarp();
    const int pairs = qn >> 1;
#pragma unroll 1
    for (int i = 0; i < pairs; ++i) {
      if (fmaxf(lo2(Q[i].op), hi2(Q[i].op)) < kAlphaMax)
        bwd_pair<PPL, false, STATS>(Q[i], px, py, g0, g1, g2, err, lastf, T, R, grad2d, st.stats);
      else
        bwd_pair<PPL, true, STATS>(Q[i], px, py, g0, g1, g2, err, lastf, T, R, grad2d, st.stats);
    }
    __syncwarp();
    if (qn & 1) {  // one splat left over: to the front
      const uint32_t* src = reinterpret_cast<const uint32_t*>(Q + pairs);
      uint32_t* dst = reinterpret_cast<uint32_t*>(Q);
      if (pairs > 0)
        for (int i = lane; i < (int)(sizeof(BwdPair) / 4); i += 32) dst[i] = src[i];
      __syncwarp();
      if (lane == 0) reinterpret_cast<float*>(&Q[0].np)[0] -= 32.f;  // from the next chunk's first
    }
    qn &= 1;
  }
  return true;
}

template <int PPL, bool STATS>
__global__ void __launch_bounds__(32, kBwdBlocksPerSm)
    k_render_bwd(RasterArgs a, const float* __restrict__ T_final, const int32_t* __restrict__ n_last,
                 const float* __restrict__ dL_drgb, float* __restrict__ grad2d, Ckpt ck, StatsK st, BwdSplit sp, int n_tiles) {
  __shared__ BwdPair Q[kBwdPairs];
  const int q = blockIdx.x / n_tiles, j = blockIdx.x - q * n_tiles;  // deeper pieces last: most of them are empty
  if (j >= *a.n_active) return;
  render_item_bwd<PPL, STATS>(a, j, q, sp, Q, T_final, n_last, dL_drgb, grad2d, ck, st);
}

// Error back-projection statistics (Sec. 3.8, Eq. 12): one
// block per active tile, one thread per sampled pixel, walking the tile's
// list front to back up to the pixel's n_last (the forward's stopping
// decision) and recomputing alpha and T as the forward does.  For each splat
// the warp sums (e w, w, D w) over its pixels (w = T alpha, D the conic
// Mahalanobis distance) and one lane adds them to the Gaussian's float4 row.
__global__ void k_error_stats(RasterArgs a, const int32_t* __restrict__ n_last, const float* __restrict__ err_pix,
                              float* __restrict__ stats) {
  extern __shared__ Splat sm[];
  __shared__ int s_max_last;
  const int j = blockIdx.x;
  if (j >= *a.n_active) return;
  const int t = a.active_tiles ? a.active_tiles[j] : j;
  const int p0 = a.pix_off[j], p1 = a.pix_off[j + 1];
  const bool has_pix = p0 + (int)threadIdx.x < p1;
  const int s = p0 + threadIdx.x;
  const int lane = threadIdx.x & 31;
  float px = 0.f, py = 0.f, e = 0.f, T = 1.f;
  int last = 0;
  if (has_pix) {
    const int l = a.pix_idx[s];
    px = (float)((t % a.tiles_x) * TGS_TILE + (l & 15)) + 0.5f;
    py = (float)((t / a.tiles_x) * TGS_TILE + (l >> 4)) + 0.5f;
    e = err_pix[s];
    last = n_last[s];
  }
  if (threadIdx.x == 0) s_max_last = 0;
  __syncthreads();
  if (last > 0) atomicMax(&s_max_last, last);
  __syncthreads();
  const int2 range = a.ranges[j];
  const int end = range.x + s_max_last;
  const int B = blockDim.x;
  const float2 band = warp_rows(last > 0, py);  // splats that cannot reach the warp's rows are skipped
  for (int base = range.x; base < end; base += B) {
    __syncthreads();  // the previous batch is no longer read
    if (base + (int)threadIdx.x < end) load_splat(a, base + threadIdx.x, sm[threadIdx.x]);
    __syncthreads();
    const int cnt = min(B, end - base);
    for (int q = 0; q < cnt; ++q) {
      const Splat sp = sm[q];
      if (sp.yr.y < band.x || sp.yr.x > band.y) continue;  // warp-uniform
      float v0 = 0.f, v1 = 0.f, v2 = 0.f;
      bool on = false;
      if (base + q - range.x < last) {
        const float dx = __fsub_rn(px, sp.xy.x), dy = __fsub_rn(py, sp.xy.y);
        float alpha, G;
        if (splat_alpha(sp.co, dx, dy, alpha, G)) {
          const float w = alpha * T;
          // a dx^2 + 2 b dx dy + c dy^2 = -2 power = -2 ln(2) p
          const float qf = splat_pow2(sp.co, dx, dy) * kInvA;
          const float D = sqrtf(fmaxf(qf, 0.f));
          v0 = e * w;
          v1 = w;
          v2 = D * w;
          T = __fmul_rn(T, __fsub_rn(1.f, alpha));  // the forward's transmittance sequence
          on = true;
        }
      }
      if (!__any_sync(0xffffffffu, on)) continue;
      v0 = warp_sum(v0);
      v1 = warp_sum(v1);
      v2 = warp_sum(v2);
      if (lane == 0) red_add_v4(stats + 4 * (size_t)__float_as_int(sp.rgb.w), v0, v1, v2, 0.f);
    }
  }
}

// ---------------------------------------------------------------------------
// Several views in one persistent launch: CTAs take (view, tile) items from
// an atomic counter (tiles of view v are [base[v], base[v+1]); the backward's
// items: below) until none are left.  There is no waiting on other CTAs, only
// one atomic per item.
// ---------------------------------------------------------------------------
constexpr int kMaxViews = 16;

struct BatchArgs {
  int n_views;
  BwdSplit split;  // the backward's items per tile
  int base[kMaxViews + 1];  // view v's tiles are [base[v], base[v + 1])
  RasterArgs a[kMaxViews];
  float* rgb[kMaxViews];
  float* T[kMaxViews];
  int32_t* last[kMaxViews];
  const float* dL[kMaxViews];
  float* grad2d[kMaxViews];
  Ckpt ck[kMaxViews];
  const float* err[kMaxViews];  // per-pixel errors, when the statistics are accumulated
  float4* stats;                // [N] (E, W, D, 0) rows shared by the views
};

__device__ __forceinline__ bool next_item(const BatchArgs& b, int* counter, int* s_item, int& v, int& j) {
  __syncthreads();  // the previous item's shared memory is no longer read
  if (threadIdx.x == 0) *s_item = atomicAdd(counter, 1);
  __syncthreads();
  const int item = *s_item;
  if (item >= b.base[b.n_views]) return false;
  v = 0;
  while (item >= b.base[v + 1]) ++v;
  j = item - b.base[v];
  return true;
}

__device__ __forceinline__ void item_view(const BatchArgs& b, int item, int& v, int& q) {
  v = 0;
  while (item >= b.base[v + 1]) ++v;
  q = item - b.base[v];
}

template <int PPL>
__global__ void __launch_bounds__(TGS_TILE_PIX / PPL) k_render_fwd_batched(BatchArgs b, int* __restrict__ counter) {
  extern __shared__ __align__(16) FwdPair fwd_sm[];
  __shared__ int s_item;
  int v, j;
  while (next_item(b, counter, &s_item, v, j)) {
    if (j < *b.a[v].n_active) render_tile_fwd<PPL>(b.a[v], j, fwd_sm, b.rgb[v], b.T[v], b.last[v], b.ck[v]);
  }
}

// The batched backward: a warp claims a group of a tile's pixels and one of Pm
// pieces, and replays that piece and every Pm-th after it as the one-view backward
// does, until one holds nothing (deeper ones do not either).  Pm is a quarter of the
// pieces, so a list of up to Pm pieces, most of them, is spread over as many warps,
// and the empty pieces take a quarter of the claims.  Claims go through the pieces at
// the fronts of all views' lists first.  Four neighbouring tiles at a time left the
// work to few warps, each of them four items to walk in turn: one view of 3600
// tiles, 100k Gaussians 235 -> 102 us; sixteen of 256x256 779 -> 368; 1080 whole lists
// of one view, a step 400 -> 227.  One at a time costs where most are empty (2000
// Gaussians, eight views of 3600 tiles: four at a time 169, one 349, here 134).
template <int PPL, bool STATS>
__global__ void __launch_bounds__(32, kBwdBlocksPerSm) k_render_bwd_batched(BatchArgs b, int* __restrict__ counter) {
  __shared__ BwdPair Q[kBwdPairs];
  const int n_tiles = b.base[b.n_views], per_tile = b.split.pieces * b.split.groups;
  const int step = (b.split.pieces + 3) / 4 * b.split.groups;  // Pm pieces
  for (;;) {
    int item = 0;
    if (threadIdx.x == 0) item = atomicAdd(counter, 1);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_tiles * step) return;
    int v, j, r = item / n_tiles;
    item_view(b, item - r * n_tiles, v, j);
    if (j >= *b.a[v].n_active) continue;
    const StatsK st{b.err[v], b.stats};
    for (; r < per_tile; r += step)
      if (!render_item_bwd<PPL, STATS>(b.a[v], j, r, b.split, Q, b.T[v], b.last[v], b.dL[v], b.grad2d[v], b.ck[v], st))
        break;
  }
}

// The kernels of a launch with at most 32 ppl pixels a group.
using BwdKernel = void (*)(RasterArgs, const float*, const int32_t*, const float*, float*, Ckpt, StatsK, BwdSplit,
                           int);
using BwdBatchedKernel = void (*)(BatchArgs, int*);
static BwdKernel bwd_kernel(int ppl, bool stats) {
  switch (2 * ppl + (stats ? 1 : 0)) {
    case 2: return k_render_bwd<1, false>;
    case 3: return k_render_bwd<1, true>;
    case 4: return k_render_bwd<2, false>;
    case 5: return k_render_bwd<2, true>;
    case 6: return k_render_bwd<3, false>;
    case 7: return k_render_bwd<3, true>;
    case 8: return k_render_bwd<4, false>;
    default: return k_render_bwd<4, true>;
  }
}
static BwdBatchedKernel bwd_batched_kernel(int ppl, bool stats) {
  switch (2 * ppl + (stats ? 1 : 0)) {
    case 2: return k_render_bwd_batched<1, false>;
    case 3: return k_render_bwd_batched<1, true>;
    case 4: return k_render_bwd_batched<2, false>;
    case 5: return k_render_bwd_batched<2, true>;
    case 6: return k_render_bwd_batched<3, false>;
    case 7: return k_render_bwd_batched<3, true>;
    case 8: return k_render_bwd_batched<4, false>;
    default: return k_render_bwd_batched<4, true>;
  }
}

static bool raster_args(const tgs_projected* proj, const int32_t* tile_ranges, const int32_t* vals,
                        const int32_t* active_tiles, const int32_t* n_active, const int32_t* pix_off,
                        const uint8_t* pix_idx, const tgs_camera* cam, const float* bg, RasterArgs& a) {
  if (!proj || !proj->xy || !proj->conic_opac || !proj->rgb || !tile_ranges || !vals || !n_active || !pix_off ||
      !pix_idx || !camera_ok(cam) || !bg)
    return false;
  if (!aligned8(proj->xy) || !aligned16(proj->conic_opac) || !aligned8(tile_ranges)) return false;
  a.xy = reinterpret_cast<const float2*>(proj->xy);
  a.conic_opac = reinterpret_cast<const float4*>(proj->conic_opac);
  a.rgb = proj->rgb;
  a.ranges = reinterpret_cast<const int2*>(tile_ranges);
  a.vals = vals;
  a.active_tiles = active_tiles;
  a.n_active = n_active;
  a.pix_off = pix_off;
  a.pix_idx = pix_idx;
  a.tiles_x = tiles_x(cam->width);
  a.bg[0] = bg[0];
  a.bg[1] = bg[1];
  a.bg[2] = bg[2];
  return true;
}

// The division of a backward launch over `tiles` tiles.  Groups of 32
// kBwdPpl pixels take the fewest instructions a pixel (one reduction serves
// them all), smaller ones shorten a warp's walk and give more of them.  With
// checkpoints the pieces give enough: groups are halved, down to one pixel a
// lane, while that leaves fewer than four items an SM (a tile's list counted as
// four pieces).  64 tiles of 85 pixels: 10.7 us in three groups, 12.1 in one.
// Without checkpoints a warp walks its tile's whole list: groups of 128 are
// halved below 32 items an SM and groups of 64 below 16.  Whole tiles of 1M
// Gaussians in groups of 128, 64, 32: 335 tiles 133, 98, 98 us; 670 tiles 150,
// 119, 152; 1005 tiles 186, 165, 202; 2010 tiles 262, 255, -; 201 tiles -, 87, 79.
// Pieces: short ones give more items, long ones read each pixel's state and
// run into half-filled chunks less often.  span 1 / 2 / 4: 64 tiles of 85
// pixels 12.1 / 17.6 / 28.9 us, 720 tiles 63.6 / 54.4 / 58.1 us, 3600 tiles of
// 25 pixels 218 / 160 / 132 us, eight views with 20000 tiles of 85 pixels
// 1334 / 1088 / 1043 us.
static BwdSplit bwd_split(int64_t tiles, int n_pix_max, const Ckpt& ck) {
  const int64_t sms = device_sm_count();
  BwdSplit sp;
  int most = 32 * kBwdPpl;
  auto groups = [&]() { return (n_pix_max + most - 1) / most; };
  const int64_t least = ck.data ? 1 : 16;  // items an SM below which groups of 64 are halved
  while (most > 32 && tiles * groups() < (ck.data || most <= 64 ? least : 2 * least) * sms) most /= 2;
  sp.groups = groups();
  sp.gpx = (n_pix_max + sp.groups - 1) / sp.groups;
  sp.span = tiles * sp.groups <= 2 * sms ? 1 : tiles * sp.groups <= 16 * sms ? 2 : 4;
  auto pieces = [&]() { return ck.data ? ck.n_slots / sp.span + 1 : 1; };
  while (pieces() > 1 && tiles * sp.groups * pieces() > INT_MAX / 2) sp.span *= 2;  // items are counted in 32 bits
  sp.pieces = pieces();
  return sp;
}

static int block_for(int n_pix_max) { return std::min(256, std::max(32, (n_pix_max + 31) / 32 * 32)); }

// Fewer than 16 warps per SM at one pixel a thread (B threads a tile).
static bool few_warps(int64_t n_tiles, int B) { return n_tiles * (B / 32) < 16 * (int64_t)device_sm_count(); }

// Pixels a lane of the forward walk: two for tiles of more than 128 pixels,
// where the launch has warps to spare.
static int fwd_ppl(int B, bool few) { return B > 128 && !few ? 2 : 1; }
static int fwd_threads(int B, int ppl) { return (B / 32 + ppl - 1) / ppl * 32; }


// Whether the automatic choice may pick the split walk: measured slower than
// the sequential walk at 500k Gaussians, 720 tiles of 85 pixels (0.085-0.089
// against 0.067 ms), so only an explicit setting selects it.
constexpr bool kSplitAuto = false;

// The split forward's group count: 0 = chosen per launch (below), or fixed
// at 1, 2 or 4 by tgs_set_forward_split (tuning and tests).
static int g_fwd_split = 0;

// The automatic choice of the walk with two threads per pixel: for tiles of
// at most 32 sampled pixels in a sparse launch, where one warp per tile
// leaves the GPU short of warps.  Elsewhere the composition and the second
// half's walk past the stop cost more than the shorter chains gain (at 85
// pixels per tile 0.068 ms against 0.047).
static bool pair_walk_auto(int B, bool sparse) { return B == 32 && sparse; }

// Groups per tile of the split forward for a launch of n_active tiles of B
// threads: the largest of 4 and 2 whose blocks all fit on the GPU at once
// (one wave), else 1 (the sequential walk).

static int split_groups(int n_active, int B) {
  const int wp = B / 32;  // 1..8
  const bool nw_ok[2] = {4 * B <= 1024, 2 * B <= 1024};
  if (g_fwd_split == 1 || g_fwd_split == 3 || g_fwd_split == 5) return 1;
  if (g_fwd_split) return (g_fwd_split == 4 && !nw_ok[0]) || (g_fwd_split == 2 && !nw_ok[1]) ? 1 : g_fwd_split;
  if (!kSplitAuto) return 1;
  static int per_sm[64][9][2] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  const int sms = device_sm_count();
  for (int k = 0; k < 2; ++k) {
    const int nw = k == 0 ? 4 : 2;
    if (!nw_ok[k]) continue;
    int& r = per_sm[dev][wp][k];
    if (r == 0) {
      int b = 0;
      if (nw == 4)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_render_fwd_split<4>, 4 * B, split_smem_bytes<4>(B));
      else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_render_fwd_split<2>, 2 * B, split_smem_bytes<2>(B));
      r = b > 0 ? b : -1;
    }
    if (r > 0 && (int64_t)n_active <= (int64_t)sms * r) return nw;
  }
  return 1;
}

}  // namespace tgs

using namespace tgs;

// Checkpoint buffer checks: stride covers every sampled pixel slot.
static bool ckpt_of(const tgs_checkpoints* c, int32_t n_active_max, int32_t n_pix_max, const float* rgb, Ckpt& k) {
  k = Ckpt{nullptr, 0, 0, nullptr, nullptr};
  if (!c || c->n_slots <= 0) return true;
  if (!c->data || !aligned16(c->data) || c->stride < (int64_t)n_active_max * n_pix_max) return false;
  k.data = reinterpret_cast<float4*>(c->data);
  k.n_slots = c->n_slots;
  k.stride = c->stride;
  k.rgb = rgb;
  k.tile_last = c->tile_last;
  return true;
}

extern "C" tgs_status tgs_set_forward_split(int32_t groups) {
  if (groups < 0 || groups > 5) return TGS_ERR_INVALID_ARG;
  g_fwd_split = groups;
  return TGS_OK;
}

extern "C" size_t tgs_checkpoint_bytes(int32_t n_active_max, int32_t n_pix_max, int32_t n_slots) {
  if (n_active_max <= 0 || n_pix_max <= 0 || n_slots <= 0) return 0;
  return sizeof(float4) * (size_t)n_slots * (size_t)n_active_max * (size_t)n_pix_max;
}

extern "C" tgs_status tgs_render_sampled(const tgs_projected* proj, const int32_t* tile_ranges, const int32_t* vals,
                                         const int32_t* active_tiles, const int32_t* n_active, int32_t n_active_max,
                                         const int32_t* pix_off, const uint8_t* pix_idx, int32_t n_pix_max,
                                         const tgs_camera* cam, const float* bg, float* rgb, float* T_final,
                                         int32_t* n_last, const tgs_checkpoints* ckpt, tgs_stream stream) {
  RasterArgs a;
  if (n_active_max < 0 || n_pix_max < 1 || n_pix_max > 256) return TGS_ERR_INVALID_ARG;
  if (!raster_args(proj, tile_ranges, vals, active_tiles, n_active, pix_off, pix_idx, cam, bg, a))
    return TGS_ERR_INVALID_ARG;
  if (!rgb || !T_final || !n_last) return TGS_ERR_INVALID_ARG;
  Ckpt ck;
  if (!ckpt_of(ckpt, n_active_max, n_pix_max, rgb, ck)) return TGS_ERR_INVALID_ARG;
  if (n_active_max == 0) return TGS_OK;
  const int B = block_for(n_pix_max);
  // sampled training (checkpoints) with few tiles: the split walk, NW groups per tile
  const int nw = ck.data ? split_groups(n_active_max, B) : 1;
  if (nw == 4) {
    k_render_fwd_split<4><<<n_active_max, 4 * B, split_smem_bytes<4>(B), (cudaStream_t)stream>>>(a, rgb, T_final,
                                                                                                 n_last, ck);
    return check_launch();
  }
  if (nw == 2) {
    k_render_fwd_split<2><<<n_active_max, 2 * B, split_smem_bytes<2>(B), (cudaStream_t)stream>>>(a, rgb, T_final,
                                                                                                 n_last, ck);
    return check_launch();
  }
  const bool few = few_warps(n_active_max, B);
  if (g_fwd_split == 5 || (g_fwd_split == 0 && pair_walk_auto(B, few))) {  // two threads per pixel
    const int B2 = 32 * ((n_pix_max + 15) / 16);
    if (few)
      k_render_fwd_pair<true><<<n_active_max, B2, B2 * sizeof(Splat), (cudaStream_t)stream>>>(a, rgb, T_final, n_last,
                                                                                              ck);
    else
      k_render_fwd_pair<false><<<n_active_max, B2, B2 * sizeof(Splat), (cudaStream_t)stream>>>(a, rgb, T_final,
                                                                                               n_last, ck);
    return check_launch();
  }
  const int ppl = fwd_ppl(B, few), threads = fwd_threads(B, ppl);
  (ppl == 2 ? k_render_fwd<2> : k_render_fwd<1>)<<<n_active_max, threads, fwd_smem(threads), (cudaStream_t)stream>>>(
      a, rgb, T_final, n_last, ck);
  return check_launch();
}

// Eq. 12's statistics of one view by the walk from the front.
static void launch_error_stats(const RasterArgs& a, int n_active_max, int n_pix_max, const int32_t* n_last,
                               const float* err, float* stats, cudaStream_t s) {
  if (n_active_max <= 0) return;
  const int B = block_for(n_pix_max);
  k_error_stats<<<n_active_max, B, B * sizeof(Splat), s>>>(a, n_last, err, stats);
}

// The one-view backward; with st.stats set, Eq. 12's statistics of the same
// pixels too: in the same replay where checkpoints are given, else by a walk of
// their own.  A replay from a checkpoint recovers T over at most a piece from the
// forward's own value, one without it over the whole list: at 500 blended splats a
// pixel its sums were 9.7e-8 of their norm off 64 bits, the walk's 5.9e-8.
static tgs_status render_backward_impl(const tgs_projected* proj, const int32_t* tile_ranges, const int32_t* vals,
                                       const int32_t* active_tiles, const int32_t* n_active, int32_t n_active_max,
                                       const int32_t* pix_off, const uint8_t* pix_idx, int32_t n_pix_max,
                                       const tgs_camera* cam, const float* bg, const float* T_final,
                                       const int32_t* n_last, const float* dL_drgb, float* grad2d,
                                       int64_t n_gaussians, const tgs_checkpoints* ckpt, StatsK st,
                                       int32_t accumulate_stats, tgs_stream stream) {
  RasterArgs a;
  if (n_gaussians < 0 || n_active_max < 0 || n_pix_max < 1 || n_pix_max > 256) return TGS_ERR_INVALID_ARG;
  if (!raster_args(proj, tile_ranges, vals, active_tiles, n_active, pix_off, pix_idx, cam, bg, a))
    return TGS_ERR_INVALID_ARG;
  if (!T_final || !n_last || !dL_drgb) return TGS_ERR_INVALID_ARG;
  if (n_gaussians > 0 && (!grad2d || !aligned16(grad2d))) return TGS_ERR_INVALID_ARG;
  const bool stats = st.stats != nullptr;
  Ckpt ck;
  if (!ckpt_of(ckpt, n_active_max, n_pix_max, ckpt ? ckpt->rgb : nullptr, ck)) return TGS_ERR_INVALID_ARG;
  if (ck.data && !ck.rgb) return TGS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_gaussians == 0) return TGS_OK;
  cudaMemsetAsync(grad2d, 0, sizeof(float) * 12 * (size_t)n_gaussians, s);
  if (stats && !accumulate_stats) cudaMemsetAsync(st.stats, 0, sizeof(float4) * (size_t)n_gaussians, s);
  if (n_active_max > 0) {
    const BwdSplit sp = bwd_split(n_active_max, n_pix_max, ck);
    const int64_t items = (int64_t)n_active_max * sp.groups * sp.pieces;
    const bool fused = stats && ck.data;
    bwd_kernel((sp.gpx + 31) / 32, fused)<<<(int)items, 32, 0, s>>>(a, T_final, n_last, dL_drgb, grad2d, ck, st,
                                                                          sp, n_active_max);
    if (stats && !fused)
      launch_error_stats(a, n_active_max, n_pix_max, n_last, st.err, reinterpret_cast<float*>(st.stats), s);
  }
  return check_launch();
}

extern "C" tgs_status tgs_render_backward_sampled(const tgs_projected* proj, const int32_t* tile_ranges,
                                                  const int32_t* vals, const int32_t* active_tiles,
                                                  const int32_t* n_active, int32_t n_active_max,
                                                  const int32_t* pix_off, const uint8_t* pix_idx, int32_t n_pix_max,
                                                  const tgs_camera* cam, const float* bg, const float* T_final,
                                                  const int32_t* n_last, const float* dL_drgb, float* grad2d,
                                                  int64_t n_gaussians, const tgs_checkpoints* ckpt,
                                                  tgs_stream stream) {
  return render_backward_impl(proj, tile_ranges, vals, active_tiles, n_active, n_active_max, pix_off, pix_idx,
                              n_pix_max, cam, bg, T_final, n_last, dL_drgb, grad2d, n_gaussians, ckpt,
                              StatsK{nullptr, nullptr}, 0, stream);
}

extern "C" tgs_status tgs_render_backward_sampled_stats(
    const tgs_projected* proj, const int32_t* tile_ranges, const int32_t* vals, const int32_t* active_tiles,
    const int32_t* n_active, int32_t n_active_max, const int32_t* pix_off, const uint8_t* pix_idx,
    int32_t n_pix_max, const tgs_camera* cam, const float* bg, const float* T_final, const int32_t* n_last,
    const float* dL_drgb, float* grad2d, int64_t n_gaussians, const tgs_checkpoints* ckpt, const float* err_pix,
    float* stats, int32_t accumulate_stats, tgs_stream stream) {
  if (!err_pix || (n_gaussians > 0 && (!stats || !aligned16(stats)))) return TGS_ERR_INVALID_ARG;
  return render_backward_impl(proj, tile_ranges, vals, active_tiles, n_active, n_active_max, pix_off, pix_idx,
                              n_pix_max, cam, bg, T_final, n_last, dL_drgb, grad2d, n_gaussians, ckpt,
                              StatsK{err_pix, reinterpret_cast<float4*>(stats)}, accumulate_stats, stream);
}

extern "C" tgs_status tgs_error_stats_sampled(const tgs_projected* proj, const int32_t* tile_ranges,
                                              const int32_t* vals, const int32_t* active_tiles,
                                              const int32_t* n_active, int32_t n_active_max, const int32_t* pix_off,
                                              const uint8_t* pix_idx, int32_t n_pix_max, const tgs_camera* cam,
                                              const int32_t* n_last, const float* err_pix, float* stats,
                                              int64_t n_gaussians, int32_t accumulate, tgs_stream stream) {
  RasterArgs a;
  const float bg[3] = {0.f, 0.f, 0.f};
  if (n_gaussians < 0 || n_active_max < 0 || n_pix_max < 1 || n_pix_max > 256) return TGS_ERR_INVALID_ARG;
  if (!raster_args(proj, tile_ranges, vals, active_tiles, n_active, pix_off, pix_idx, cam, bg, a))
    return TGS_ERR_INVALID_ARG;
  if (!n_last || !err_pix) return TGS_ERR_INVALID_ARG;
  if (n_gaussians > 0 && (!stats || !aligned16(stats))) return TGS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_gaussians == 0) return TGS_OK;
  if (!accumulate) cudaMemsetAsync(stats, 0, sizeof(float) * 4 * (size_t)n_gaussians, s);
  launch_error_stats(a, n_active_max, n_pix_max, n_last, err_pix, stats, s);
  return check_launch();
}

extern "C" tgs_status tgs_backward_sampled(const tgs_gaussians* g, const tgs_camera* cam, const tgs_projected* proj,
                                           const int32_t* tile_ranges, const int32_t* vals,
                                           const int32_t* active_tiles, const int32_t* n_active,
                                           int32_t n_active_max, const int32_t* pix_off, const uint8_t* pix_idx,
                                           int32_t n_pix_max, const float* bg, const float* T_final,
                                           const int32_t* n_last, const float* dL_drgb, float* grad2d,
                                           const tgs_param_ptrs* grads, uint8_t* touched, int32_t write_untouched,
                                           const tgs_checkpoints* ckpt, tgs_stream stream) {
  RasterArgs a;
  if (!gaussians_ok(g) || n_active_max < 0 || n_pix_max < 1 || n_pix_max > 256) return TGS_ERR_INVALID_ARG;
  if (!raster_args(proj, tile_ranges, vals, active_tiles, n_active, pix_off, pix_idx, cam, bg, a))
    return TGS_ERR_INVALID_ARG;
  if (!T_final || !n_last || !dL_drgb || !grads || !proj->radius) return TGS_ERR_INVALID_ARG;
  if (g->n > 0 && (!grad2d || !aligned16(grad2d) || !param_ptrs_ok(grads)))
    return TGS_ERR_INVALID_ARG;
  const tgs_status st = tgs_render_backward_sampled(proj, tile_ranges, vals, active_tiles, n_active, n_active_max,
                                                    pix_off, pix_idx, n_pix_max, cam, bg, T_final, n_last, dL_drgb,
                                                    grad2d, g->n, ckpt, stream);
  if (st != TGS_OK || g->n == 0) return st;
  launch_project_bwd(*g, *cam, proj->radius, grad2d, *grads, touched, write_untouched, 0, nullptr,
                     (cudaStream_t)stream);
  return check_launch();
}

static tgs_status batch_args(const tgs_view_batch* views, int32_t n_views, bool backward, BatchArgs& b, int& B) {
  if (!views || n_views < 1 || n_views > kMaxViews) return TGS_ERR_INVALID_ARG;
  b.n_views = n_views;
  b.stats = nullptr;
  for (int v = 0; v < kMaxViews; ++v) b.err[v] = nullptr;
  b.base[0] = 0;
  B = 32;
  // checkpoints: all views or none, with one slot count
  const int slots = views[0].ckpt.n_slots > 0 ? views[0].ckpt.n_slots : 0;
  for (int v = 0; v < n_views; ++v) {
    const tgs_view_batch& w = views[v];
    if (w.n_active_max < 0 || w.n_pix_max < 1 || w.n_pix_max > 256) return TGS_ERR_INVALID_ARG;
    if (!raster_args(&w.proj, w.tile_ranges, w.vals, w.active_tiles, w.n_active, w.pix_off, w.pix_idx, &w.cam,
                     w.bg, b.a[v]))
      return TGS_ERR_INVALID_ARG;
    if (!w.rgb || !w.T_final || !w.n_last) return TGS_ERR_INVALID_ARG;
    if (backward && (!w.dL_drgb || !w.grad2d || !aligned16(w.grad2d) || w.n_gaussians < 0))
      return TGS_ERR_INVALID_ARG;
    b.rgb[v] = w.rgb;
    b.T[v] = w.T_final;
    b.last[v] = w.n_last;
    b.dL[v] = w.dL_drgb;
    b.grad2d[v] = w.grad2d;
    if ((w.ckpt.n_slots > 0 ? w.ckpt.n_slots : 0) != slots) return TGS_ERR_INVALID_ARG;
    if (!ckpt_of(&w.ckpt, w.n_active_max, w.n_pix_max, w.rgb, b.ck[v])) return TGS_ERR_INVALID_ARG;
    if (b.ck[v].data && w.ckpt.rgb && w.ckpt.rgb != w.rgb) return TGS_ERR_INVALID_ARG;
    B = std::max(B, block_for(w.n_pix_max));
  }
  int64_t tiles = 0;
  int n_pix = 1;
  for (int v = 0; v < n_views; ++v) {
    tiles += views[v].n_active_max;
    n_pix = std::max(n_pix, (int)views[v].n_pix_max);
  }
  b.split = bwd_split(tiles, n_pix, b.ck[0]);
  for (int v = 0; v < n_views; ++v) b.base[v + 1] = b.base[v] + views[v].n_active_max;
  return TGS_OK;
}

// The backward's count is that of the kernel without statistics for whole groups
// of n_pix_max pixels (backward 1 and 2 alike); a launch whose groups bwd_split
// halves runs a kernel that fits more often, up to 23 blocks an SM for 20.
extern "C" tgs_status tgs_render_batched_resident(int32_t n_pix_max, int32_t backward, int32_t* ctas) {
  if (!ctas || n_pix_max < 1 || n_pix_max > 256 || backward < 0 || backward > 2) return TGS_ERR_INVALID_ARG;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return check_launch();
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int B = block_for(n_pix_max);
  if (backward)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bwd_batched_kernel(std::min(B / 32, kBwdPpl), false),
                                                  32, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fwd_ppl(B, false) == 2 ? k_render_fwd_batched<2> : k_render_fwd_batched<1>,
                                                  fwd_threads(B, fwd_ppl(B, false)),
                                                  fwd_smem(fwd_threads(B, fwd_ppl(B, false))));
  *ctas = sms * per_sm;
  return check_launch();
}

extern "C" tgs_status tgs_render_sampled_batched(const tgs_view_batch* views, int32_t n_views, int32_t grid_ctas,
                                                 int32_t* counter, tgs_stream stream) {
  BatchArgs b;
  int B = 32;
  tgs_status st = batch_args(views, n_views, false, b, B);
  if (st != TGS_OK) return st;
  if (grid_ctas < 1 || !counter) return TGS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  cudaMemsetAsync(counter, 0, sizeof(int32_t), s);
  if (b.base[n_views] == 0) return check_launch();
  const int ppl = fwd_ppl(B, false), threads = fwd_threads(B, ppl);
  (ppl == 2 ? k_render_fwd_batched<2> : k_render_fwd_batched<1>)<<<grid_ctas, threads, fwd_smem(threads), s>>>(b, counter);
  return check_launch();
}

static tgs_status render_backward_batched_impl(const tgs_view_batch* views, int32_t n_views, int32_t grid_ctas,
                                               int32_t* counter, const float* const* err_pix, float* stats,
                                               int64_t n_stats, int32_t accumulate_stats, tgs_stream stream) {
  BatchArgs b;
  int B = 32;
  tgs_status st = batch_args(views, n_views, true, b, B);
  if (st != TGS_OK) return st;
  if (grid_ctas < 1 || !counter) return TGS_ERR_INVALID_ARG;
  const bool with_stats = err_pix != nullptr;
  b.stats = reinterpret_cast<float4*>(stats);
  for (int v = 0; v < n_views; ++v) {
    b.err[v] = with_stats ? err_pix[v] : nullptr;
    if (with_stats && (!b.err[v] || views[v].n_gaussians > n_stats)) return TGS_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  for (int v = 0; v < n_views; ++v)
    if (views[v].n_gaussians > 0)
      cudaMemsetAsync(views[v].grad2d, 0, sizeof(float) * 12 * (size_t)views[v].n_gaussians, s);
  if (with_stats && !accumulate_stats && n_stats > 0) cudaMemsetAsync(stats, 0, sizeof(float4) * (size_t)n_stats, s);
  cudaMemsetAsync(counter, 0, sizeof(int32_t), s);
  if (b.base[n_views] == 0) return check_launch();
  const bool fused = with_stats && b.ck[0].data;
  bwd_batched_kernel((b.split.gpx + 31) / 32, fused)<<<grid_ctas, 32, 0, s>>>(b, counter);
  for (int v = 0; with_stats && !fused && v < n_views; ++v)  // without checkpoints: as in the one-view backward
    launch_error_stats(b.a[v], views[v].n_active_max, views[v].n_pix_max, b.last[v], b.err[v], stats, s);
  return check_launch();
}

extern "C" tgs_status tgs_render_backward_batched(const tgs_view_batch* views, int32_t n_views, int32_t grid_ctas,
                                                  int32_t* counter, tgs_stream stream) {
  return render_backward_batched_impl(views, n_views, grid_ctas, counter, nullptr, nullptr, 0, 0, stream);
}

extern "C" tgs_status tgs_render_backward_batched_stats(const tgs_view_batch* views, int32_t n_views,
                                                        int32_t grid_ctas, int32_t* counter,
                                                        const float* const* err_pix, float* stats,
                                                        int64_t n_gaussians, int32_t accumulate_stats,
                                                        tgs_stream stream) {
  if (!err_pix || n_gaussians < 0 || (n_gaussians > 0 && (!stats || !aligned16(stats)))) return TGS_ERR_INVALID_ARG;
  return render_backward_batched_impl(views, n_views, grid_ctas, counter, err_pix, stats, n_gaussians,
                                      accumulate_stats, stream);
}

extern "C" tgs_status tgs_project_backward(const tgs_gaussians* g, const tgs_camera* cam, const tgs_projected* proj,
                                           const float* grad2d, const tgs_param_ptrs* grads, uint8_t* touched,
                                           int32_t write_untouched, int32_t accumulate, float* view_row,
                                           tgs_stream stream) {
  if (!gaussians_ok(g) || !camera_ok(cam) || !proj || !grads) return TGS_ERR_INVALID_ARG;
  if (accumulate && !touched) return TGS_ERR_INVALID_ARG;
  if (view_row && !aligned8(view_row)) return TGS_ERR_INVALID_ARG;
  if (g->n == 0) return TGS_OK;
  if (!proj->radius || !grad2d || !aligned16(grad2d) || !param_ptrs_ok(grads))
    return TGS_ERR_INVALID_ARG;
  launch_project_bwd(*g, *cam, proj->radius, grad2d, *grads, touched, write_untouched, accumulate, view_row,
                     (cudaStream_t)stream);
  return check_launch();
}
