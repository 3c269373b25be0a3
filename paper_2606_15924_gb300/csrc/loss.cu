// Fused sparse supervision (Sec. 3.7, Eqs. 9-11; App. A): Charbonnier L1,
// tile-level sparse NCC (or, for Table 4's S-SSIM variant, SSIM) with the
// gradient-balanced weight, the per-pixel error
// of Eq. 2 and the error/age map updates of Eqs. 3-4.  One warp per active
// tile; tile moments are two-pass warp reductions.
#include "tgs_common.cuh"

namespace tgs {

struct LossArgs {
  const float* rgb;
  const float* target;
  int W, H, tiles_x;
  const int32_t* active_tiles;
  const int32_t* n_active;
  int n_active_max;
  const int32_t* pix_off;
  const uint8_t* pix_idx;
  float eps_c2, eps_n, beta, weight;
  uint16_t* err_map;
  uint16_t* age_map;
  float* dL;
  float* lambda;
  float* err_pix;
  double* loss;
};

// SSIM constants (Wang et al. 2004, dynamic range 1) of the S-SSIM variant.
constexpr float kC1 = 1e-4f, kC2 = 9e-4f;

// STRUCT 0: the sparse NCC term (Sec. 3.7); 1: the SSIM term of Table 4's
// S-SSIM variant, per channel from the same tile moments:
// SSIM = (2 mx my + C1)(2 cov + C2) / ((mx^2 + my^2 + C1)(var_x + var_y + C2)).
//
// A warp takes whole tiles in turn, PPL pixels a lane (pixel lane + 32 k), held in
// registers from the loads to the stores: a sum over the tile is a lane's own
// sum and one warp reduction, nothing waits at a barrier, and the loss leaves a
// block as one atomic at its end.  Bound by the chains of loads and reductions of
// the few warps that the registers leave.  With a block per tile and a thread
// per pixel every one of a tile's eight warps took all 18 reductions, three
// block sums of two barriers each, and one thread's FP64 divisions and atomic
// ended every tile: every pixel of 1957x1091 116 -> 42 us, of 1280x720 49 -> 20;
// 720 tiles of 85 pixels 10 -> 7.7, eight views of 1200 to 4500 such tiles 192 ->
// 105.
constexpr int kLossWarps = 4;
// Blocks on an SM, and launched per SM: 168 registers hold eight pixels a lane,
// without spills for NCC and with 64 bytes a thread for SSIM (four blocks of 128:
// 51 us for 42; 105 for 115 at three pixels).
__host__ __device__ constexpr int loss_blocks(int ppl) { return ppl > 4 ? 3 : 4; }

template <int STRUCT, int PPL>
__global__ void __launch_bounds__(32 * kLossWarps, loss_blocks(PPL)) k_loss(LossArgs a) {
  __shared__ double s_sum[kLossWarps][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int A = *a.n_active;
  const int P = A > 0 ? a.pix_off[A] : 0;
  double sum_l1 = 0.0, sum_lam = 0.0, sum_corr = 0.0;  // over the warp's tiles: L1, lambda, lambda times the structure sum
  for (int j = blockIdx.x * kLossWarps + warp; j < min(A, a.n_active_max); j += gridDim.x * kLossWarps) {
    const int t = a.active_tiles ? a.active_tiles[j] : j;
    const int p0 = a.pix_off[j], n = a.pix_off[j + 1] - p0;
    if (n <= 0) continue;
    const int tx0 = (t % a.tiles_x) * TGS_TILE, ty0 = (t / a.tiles_x) * TGS_TILE;
    float x[PPL][3], y[PPL][3];
    uint32_t pix[PPL];
    uint16_t old_err[PPL];
    int loc[PPL];
#pragma unroll
    for (int k = 0; k < PPL; ++k) loc[k] = lane + 32 * k < n ? a.pix_idx[p0 + lane + 32 * k] : -1;
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      const bool on = loc[k] >= 0;
      pix[k] = on ? (uint32_t)(ty0 + (loc[k] >> 4)) * (uint32_t)a.W + (uint32_t)(tx0 + (loc[k] & 15)) : 0u;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x[k][c] = on ? a.rgb[3 * (size_t)(p0 + lane + 32 * k) + c] : 0.f;
        y[k][c] = on ? a.target[3 * (size_t)pix[k] + c] : 0.f;
      }
      // the pixel's error-map entry, read now so that the load overlaps the reductions
      old_err[k] = on && a.err_map ? a.err_map[pix[k]] : (uint16_t)0;
    }
    const float inv_n = 1.f / (float)n;
    // pass 1: means
    float mx[3], my[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float sx = x[0][c], sy = y[0][c];
#pragma unroll
      for (int k = 1; k < PPL; ++k) {
        sx += x[k][c];
        sy += y[k][c];
      }
      mx[c] = warp_sum(sx) * inv_n;
      my[c] = warp_sum(sy) * inv_n;
    }
    // pass 2: variances and covariances
    float mom[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) mom[q] = 0.f;
#pragma unroll
    for (int k = 0; k < PPL; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float dx = loc[k] >= 0 ? x[k][c] - mx[c] : 0.f, dy = loc[k] >= 0 ? y[k][c] - my[c] : 0.f;
        mom[c] += dx * dx;
        mom[3 + c] += dy * dy;
        mom[6 + c] += dx * dy;
      }
#pragma unroll
    for (int q = 0; q < 9; ++q) mom[q] = warp_sum(mom[q]);
    // NCC: D = sqrt(var_x var_y + eps), ncc = cov / D.  SSIM: ncc holds SSIM,
    // q1 = 1 / (b1 b2), q2 = mx / b1, D = b2 (a1, a2, b1, b2 as in the SSIM formula)
    // cx = ncc var_y / D, what a pixel's dx weighs in the NCC gradient
    float D[3], ncc[3], cx[3], a1[3], a2[3], q1[3], q2[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float vx = mom[c] * inv_n;
      const float vy = mom[3 + c] * inv_n;
      const float cv = mom[6 + c] * inv_n;
      if (STRUCT == 0) {
        D[c] = sqrtf(vx * vy + a.eps_n);
        ncc[c] = cv / D[c];
        cx[c] = ncc[c] * vy / D[c];
      } else {
        a1[c] = 2.f * mx[c] * my[c] + kC1;
        a2[c] = 2.f * cv + kC2;
        const float b1 = mx[c] * mx[c] + my[c] * my[c] + kC1;
        D[c] = vx + vy + kC2;
        q1[c] = 1.f / (b1 * D[c]);
        q2[c] = mx[c] / b1;
        ncc[c] = a1[c] * a2[c] * q1[c];
      }
    }
    // per-pixel gradients of both terms (in x and y from here on) and the balancing weight
    float l1 = 0.f, g1 = 0.f, gn = 0.f, e[PPL];
#pragma unroll
    for (int k = 0; k < PPL; ++k) {
      e[k] = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float d = x[k][c] - y[k][c], dx = x[k][c] - mx[c], dy = y[k][c] - my[c];
        const float r = sqrtf(d * d + a.eps_c2);
        const float d1 = d / r;                               // dl1/dx
        float dn;
        if (STRUCT == 0)
          dn = (dy - cx[c] * dx) / D[c];                      // n dNCC_c/dx
        else                                                  // n dSSIM_c/dx
          dn = 2.f * ((my[c] * a2[c] + a1[c] * dy) * q1[c] - ncc[c] * (q2[c] + dx / D[c]));
        if (loc[k] >= 0) {
          l1 += r;
          e[k] += fabsf(d);
          g1 += fabsf(d1);
          gn += fabsf(dn);
        }
        x[k][c] = d1;
        y[k][c] = dn;
      }
    }
    l1 = warp_sum(l1);
    g1 = warp_sum(g1);
    gn = warp_sum(gn);
    const float lam = fminf(1.f, fmaxf(0.f, (g1 * inv_n) / (gn * inv_n + 1e-8f)));
    const float invP = 1.f / (float)P;
    const float cn = lam / (3.f * (float)A) * inv_n;
#pragma unroll
    for (int k = 0; k < PPL; ++k)
      if (loc[k] >= 0) {
        const size_t s = (size_t)(p0 + lane + 32 * k);
#pragma unroll
        for (int c = 0; c < 3; ++c) a.dL[3 * s + c] = (x[k][c] * invP - cn * y[k][c]) * a.weight;
        a.err_pix[s] = e[k];
        if (a.err_map) {
          const float old = __half2float(__ushort_as_half(old_err[k]));
          a.err_map[pix[k]] = __half_as_ushort(__float2half_rn(__fmaf_rn(a.beta, e[k], __fmul_rn(1.f - a.beta, old))));
        }
        if (a.age_map) a.age_map[pix[k]] = 0;
      }
    if (lane == 0) {
      a.lambda[j] = lam;
      sum_l1 += (double)l1;
      sum_lam += (double)lam;
      sum_corr += (double)lam * ((double)ncc[0] + (double)ncc[1] + (double)ncc[2]);
    }
  }
  if (lane == 0) {
    s_sum[warp][0] = sum_l1;
    s_sum[warp][1] = 3.0 * sum_lam - sum_corr;
  }
  __syncthreads();
  if (threadIdx.x == 0 && P > 0 && blockIdx.x * kLossWarps < A) {
    double l = 0.0, q = 0.0;
    for (int w = 0; w < kLossWarps; ++w) {
      l += s_sum[w][0];
      q += s_sum[w][1];
    }
    // l / P + q / (3 A), in one FP64 division
    const double a3 = 3.0 * (double)A;
    atomicAdd(a.loss, (l * a3 + q * (double)P) / (a3 * (double)P) * (double)a.weight);
  }
}

// A <- min(A + 1, 65535) on every pixel, eight at a time; the first thread
// also clears the loss accumulator the loss kernel adds to next.
__global__ void k_age_inc(uint16_t* __restrict__ age, int64_t n, double* __restrict__ loss) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *loss = 0.0;
  const int64_t n8 = n / 8;
  if (i < n8) {
    uint4 v = reinterpret_cast<uint4*>(age)[i];
    v.x = __vaddus2(v.x, 0x00010001u);
    v.y = __vaddus2(v.y, 0x00010001u);
    v.z = __vaddus2(v.z, 0x00010001u);
    v.w = __vaddus2(v.w, 0x00010001u);
    reinterpret_cast<uint4*>(age)[i] = v;
  } else {
    const int64_t k = n8 * 8 + (i - n8);
    if (i >= n8 && k < n) age[k] = (uint16_t)min(65535, (int)age[k] + 1);
  }
}

}  // namespace tgs

using namespace tgs;

static tgs_status loss_impl(int structure, const float* rgb, const float* target, int32_t width, int32_t height,
                            const int32_t* active_tiles, const int32_t* n_active, int32_t n_active_max,
                            const int32_t* pix_off, const uint8_t* pix_idx, int32_t n_pix_max,
                            const tgs_loss_params* params, uint16_t* err_map, uint16_t* age_map, float* dL_drgb,
                            float* lambda_tile, float* err_pix, double* loss, tgs_stream stream) {
  if (!rgb || !target || width <= 0 || height <= 0 || !n_active || n_active_max < 0 || !pix_off || !pix_idx ||
      n_pix_max < 1 || n_pix_max > 256 || !params || !dL_drgb || !lambda_tile || !err_pix || !loss)
    return TGS_ERR_INVALID_ARG;
  if (age_map && !aligned16(age_map)) return TGS_ERR_INVALID_ARG;
  if (!(params->eps_charbonnier >= 0.f) || !(params->eps_ncc >= 0.f) || !(params->beta >= 0.f) ||
      !(params->view_weight >= 0.f) ||
      !(params->beta <= 1.f))
    return TGS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (age_map) {
    const int64_t n = (int64_t)width * height;
    const int64_t threads = n / 8 + (n % 8);
    k_age_inc<<<(int)((threads + 255) / 256), 256, 0, s>>>(age_map, n, loss);
  } else {
    cudaMemsetAsync(loss, 0, sizeof(double), s);
  }
  if (n_active_max > 0) {
    LossArgs a;
    a.rgb = rgb; a.target = target; a.W = width; a.H = height; a.tiles_x = tiles_x(width);
    a.active_tiles = active_tiles; a.n_active = n_active; a.n_active_max = n_active_max; a.pix_off = pix_off; a.pix_idx = pix_idx;
    a.eps_c2 = params->eps_charbonnier * params->eps_charbonnier;
    a.eps_n = params->eps_ncc;
    a.beta = params->beta;
    a.weight = params->view_weight;
    a.err_map = err_map; a.age_map = age_map; a.dL = dL_drgb; a.lambda = lambda_tile; a.err_pix = err_pix;
    a.loss = loss;
    const int ppl = n_pix_max <= 128 ? (n_pix_max + 31) / 32 : 8;
    const int blocks = std::min((n_active_max + kLossWarps - 1) / kLossWarps,
                                loss_blocks(ppl) * std::max(1, device_sm_count()));
    auto launch = [&](auto ncc, auto ssim) { (structure == 0 ? ncc : ssim)<<<blocks, 32 * kLossWarps, 0, s>>>(a); };
    switch (ppl) {
      case 1: launch(k_loss<0, 1>, k_loss<1, 1>); break;
      case 2: launch(k_loss<0, 2>, k_loss<1, 2>); break;
      case 3: launch(k_loss<0, 3>, k_loss<1, 3>); break;
      case 4: launch(k_loss<0, 4>, k_loss<1, 4>); break;
      default: launch(k_loss<0, 8>, k_loss<1, 8>); break;
    }
  }
  return check_launch();
}

extern "C" tgs_status tgs_loss_sparse_ncc(const float* rgb, const float* target, int32_t width, int32_t height,
                                          const int32_t* active_tiles, const int32_t* n_active,
                                          int32_t n_active_max, const int32_t* pix_off, const uint8_t* pix_idx,
                                          int32_t n_pix_max, const tgs_loss_params* params, uint16_t* err_map,
                                          uint16_t* age_map, float* dL_drgb, float* lambda_tile, float* err_pix,
                                          double* loss, tgs_stream stream) {
  return loss_impl(0, rgb, target, width, height, active_tiles, n_active, n_active_max, pix_off, pix_idx,
                   n_pix_max, params, err_map, age_map, dL_drgb, lambda_tile, err_pix, loss, stream);
}

extern "C" tgs_status tgs_loss_sparse_ssim(const float* rgb, const float* target, int32_t width, int32_t height,
                                           const int32_t* active_tiles, const int32_t* n_active,
                                           int32_t n_active_max, const int32_t* pix_off, const uint8_t* pix_idx,
                                           int32_t n_pix_max, const tgs_loss_params* params, uint16_t* err_map,
                                           uint16_t* age_map, float* dL_drgb, float* lambda_tile, float* err_pix,
                                           double* loss, tgs_stream stream) {
  return loss_impl(1, rgb, target, width, height, active_tiles, n_active, n_active_max, pix_off, pix_idx,
                   n_pix_max, params, err_map, age_map, dL_drgb, lambda_tile, err_pix, loss, stream);
}
