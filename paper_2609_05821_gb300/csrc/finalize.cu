// Launches of the per-token and per-image reductions of the scoring pass
// (Conduit Eqs. 6-8; the block-level code is in token_reduce.cuh):
// finalize_tokens_kernel reduces 32 tokens per block over the layers (one
// warp per layer slot), finalize_warps_kernel 32 tokens per warp, and
// image_means_kernel takes one CTA per image.
#include "token_reduce.cuh"

namespace conduit {
namespace {

__global__ void __launch_bounds__(1024) finalize_tokens_kernel(TokenReduceArgs f,
                                                               const __grid_constant__ LayerList layers,
                                                               BatchDev b) {
  __shared__ float part_s[kLayerSlots][33];
  __shared__ float part_a[kLayerSlots][33];
  token_reduce_block(f, layers, b, int64_t(blockIdx.x) * kTokBlock, part_s, part_a);
}

// The same sums in the same order by one warp per 32 tokens, which walks the layers
// alone with all partials of a layer in flight: no barrier and no part of a warp's
// life without loads, where a block of the kernel above spends most of its time
// before its first and after its last load. It needs enough tokens for its warps to
// cover the loads' latency, and layers enough that they matter. With the scoring, us
// in blocks / warps: 28 layers, 28/4 heads 8 192 tokens 251 / 288, 32 768 870 / 890,
// 65 536 1 008 / 1 004, 98 304 1 511 / 1 498, 131 072 2 028 / 1 995, batched serving
// 4 752 / 4 645, where the blocks take 235 us for 411 MB of partials; 8 layers, 32/8
// heads 98 304 816 / 820, 131 072 972 / 974.
constexpr int kWarpsPerBlock = 4;

__global__ void __launch_bounds__(32 * kWarpsPerBlock, 8) finalize_warps_kernel(TokenReduceArgs f,
                                                                             const __grid_constant__ LayerList layers,
                                                                             BatchDev b) {
  const int64_t tg = (int64_t(blockIdx.x) * kWarpsPerBlock + threadIdx.x / 32) * kTokBlock + threadIdx.x % 32;
  if (tg >= f.n_tot) return;
  const int64_t n_tot = f.n_tot;
  const int r = request_of(b.tok_off, b.R, tg);
  const int nq = b.q_off[r + 1] - b.q_off[r];
  const float denom = float(nq * f.Hq);
  const int rows = (f.Hq / f.Hkv) * nq;
  const int n_sl = (f.group_rows ? (rows + f.group_rows - 1) / f.group_rows : 1) * f.parts;
  const int per_g = f.rg_max * f.parts, npa = f.Hkv * n_sl, nss = f.Hkv * f.parts;
  // partial q of a layer is row q + (q / n_sl) (per_g - n_sl) of its partials; q / n_sl
  // by the multiplier 2^32 / n_sl, exact for these sizes
  const uint32_t inv = n_sl == 1 ? 0u : 0xffffffffu / uint32_t(n_sl) + 1u;
  constexpr int kBatch = 24;
  auto load = [&](const float* base, int q0, float (&x)[kBatch]) {
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int q = q0 + k, g = n_sl == 1 ? q : int(__umulhi(uint32_t(q), inv));
      x[k] = q < npa ? __ldg(base + int64_t(q + g * (per_g - n_sl)) * n_tot) : 0.f;
    }
  };
  auto sum = [&](const float* base) {
    float total = 0.f;
    for (int q0 = 0; q0 < npa; q0 += kBatch) {
      float x[kBatch];
      load(base, q0, x);
#pragma unroll
      for (int k = 0; k < kBatch; ++k) total += x[k];
    }
    return total;
  };
  constexpr int kVals = 8;
  float ts = 0.f, ta = 0.f;
  for (int slot = 0; slot < min(kLayerSlots, f.n_layers); ++slot) {
    float acc_s = 0.f, acc_a = 0.f;
    for (int li = slot; li < f.n_layers; li += kLayerSlots) {
      const int64_t pa_l = int64_t(li) * f.Hkv * per_g * n_tot + tg;
      float xv[kVals];
      const float* ss_l = f.ss + int64_t(li) * nss * n_tot + tg;
      if (f.vmode == 0) {
#pragma unroll
        for (int k = 0; k < kVals; ++k) xv[k] = k < nss ? __ldg(ss_l + int64_t(k) * n_tot) : 0.f;
      }
      const float a = sum(f.pa + pa_l) / denom;
      const float stat = f.pa2 ? sqrtf(sum(f.pa2 + pa_l) / denom) : a;
      float vn = 1.f;
      if (f.vmode == 1) vn = f.vnorm[int64_t(layers.ids[li]) * n_tot + tg];
      if (f.vmode == 0) {
        float sq = 0.f;
#pragma unroll
        for (int k = 0; k < kVals; ++k) sq += xv[k];
        for (int k = kVals; k < nss; ++k) sq += __ldg(ss_l + int64_t(k) * n_tot);
        vn = sqrtf(sq);
      }
      acc_s = fmaf(stat, vn, acc_s);
      acc_a += a;
    }
    ts += acc_s;
    ta += acc_a;
  }
  const float sv = ts / float(f.n_layers);
  if (!isfinite(sv) || !isfinite(ta)) flag_status(f.status, CONDUIT_FLAG_NONFINITE);
  f.s[tg] = sv;
  f.attn_sum[tg] = ta;
}

// One CTA of 256 threads per image: g_j by a fixed-order tree reduction of A over its span.
__global__ void __launch_bounds__(kMeanThreads) image_means_kernel(const float* attn_sum, BatchDev b,
                                                                   int n_layers, float* g) {
  __shared__ float warp_s[kMeanThreads / 32];
  const int j = blockIdx.x;
  image_mean_group(attn_sum, b.img_off[j], b.img_off[j + 1], n_layers, int(threadIdx.x), warp_s, &g[j],
                   [] { __syncthreads(); });
}

// finalize_warps_kernel from so many tokens, and tokens times layers, on
constexpr int64_t kWarpTokens = 98304, kWarpWork = 1500000;

}  // namespace

cudaError_t launch_finalize(const float* pa, const float* pa2, const float* ss, const float* vnorm,
                            int vmode, const LayerList& layers, const BatchDev& b, int n_layers, int Hkv,
                            int Hq, int rg_max, int group_rows, int parts, int64_t n_tot, float* s,
                            float* attn_sum, float* g, int32_t* status, cudaStream_t stream) {
  if (n_tot == 0) return cudaSuccess;
  const TokenReduceArgs f{pa, pa2, ss, vnorm, vmode, n_layers, Hkv, Hq, rg_max, group_rows, parts,
                          n_tot, s, attn_sum, status};
  const unsigned groups = unsigned((n_tot + kTokBlock - 1) / kTokBlock);
  if (n_tot >= kWarpTokens && n_tot * n_layers >= kWarpWork)
    finalize_warps_kernel<<<(groups + kWarpsPerBlock - 1) / kWarpsPerBlock, 32 * kWarpsPerBlock, 0, stream>>>(f, layers,
                                                                                                             b);
  else
    finalize_tokens_kernel<<<groups, 32 * std::min(kLayerSlots, n_layers), 0, stream>>>(f, layers, b);
  cudaError_t err = cudaGetLastError();
  if (err) return err;
  image_means_kernel<<<b.K, kMeanThreads, 0, stream>>>(attn_sum, b, n_layers, g);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace conduit
