// CUDA-core scoring pass (any head_dim multiple of 8 up to 256, fp32 or bf16).
//
// Conduit Eq. 6 needs, per (request, layer, KV head g), the softmax over all
// N_r visual keys of every scoring row (query head h of group g, query q):
//   pass 1  row statistics over chunks of the keys: m = max_t x_t and Z = sum_t
//           2^(x_t - m), with x = <q, k_t> log2(e) / sqrt(d) (the log2 domain
//           keeps exp2 exact to the same softmax);
//   pass 2  column sums pa[l][g][t] = sum_rows 2^(x_t - lse), lse the rows'
//           log2-sum-exp merged over the chunks: the sum over the group's heads
//           and the span of alpha_{q,t}. The same blocks reduce their tokens' value
//           rows, ss[l][g][t] = sum_e V[l][g][t][e]^2 (Sec. 3.3, concatenated heads).
// Pass 1 splits the keys into chunks because a small call has few row blocks: on
// one layer, 2 KV heads, 32 rows and 256 keys two blocks walked all keys in 59 us
// (fp32, 64 dims); four chunks each take 7 us, and pass 2 with the norms
// 13.4 us (14 + 4.6 us in two launches before).
// All reductions run in a fixed order, so results are deterministic; the number of
// chunks goes by the whole launch, so the last bits of a request's results may differ
// with what else is in its batch.
#include <algorithm>

#include "simt_tile.cuh"

namespace conduit {
namespace {

using namespace simt;

// Scoring rows [row0, row0 + 32) of slab (l, g, r) as element offsets into q.
__device__ __forceinline__ void row_offsets(const KvDev& kv, int l, int g, int q0, int nq, int32_t q_tot, int row0,
                                            int64_t* off) {
  if (threadIdx.x < kRowTile) {
    const int rr = row0 + threadIdx.x;
    off[threadIdx.x] =
        rr < kv.G * nq ? ((int64_t(l) * kv.Hq + g * kv.G + rr / nq) * q_tot + q0 + rr % nq) * kv.d : -1;
  }
}

__device__ __forceinline__ void key_offsets(const KvDev& kv, int l, int g, int r, int t0, int N, int tt, int64_t* off) {
  if (threadIdx.x < kKeyTile) {
    const int t = tt + threadIdx.x;
    off[threadIdx.x] = t < N ? kv.row(l, g, r, int64_t(t0) + t, t) : -1;
  }
}

// Pass 1: one CTA per (row block x key chunk, layer * Hkv + g, request); writes
// (max, sum) of its rows over its chunk to stats[chunk][l][h][q].
template <typename T>
__global__ void __launch_bounds__(kThreads) rowstats_kernel(KvDev kv, BatchDev b, const T* q, int32_t q_tot,
                                                            const __grid_constant__ LayerList layers, int chunk_keys,
                                                            int chunks, float2* stats) {
  extern __shared__ __align__(16) float smem[];
  const int d = kv.d;
  float* q_s = smem;                                 // [32][d + 4]
  float* k_s = smem + kRowTile * row_stride(d);      // [64][d + 4]
  __shared__ int64_t q_off_s[kRowTile], k_off_s[kKeyTile];

  const int r = blockIdx.z;
  const int li = blockIdx.y / kv.Hkv, g = blockIdx.y % kv.Hkv, l = layers.ids[li];
  const int q0 = b.q_off[r], nq = b.q_off[r + 1] - q0, R = kv.G * nq;
  const int chunk = blockIdx.x % chunks, row0 = int(blockIdx.x / chunks) * kRowTile;
  if (row0 >= R) return;
  const int t0 = b.tok_off[r], N = b.tok_off[r + 1] - t0;
  const int t_end = min(N, (chunk + 1) * chunk_keys);

  row_offsets(kv, l, g, q0, nq, q_tot, row0, q_off_s);
  __syncthreads();
  load_rows(q_s, q, q_off_s, kRowTile, d, kLog2e * rsqrtf(float(d)));
  const int i = threadIdx.x / 16, j = threadIdx.x % 16;
  float m_run[2] = {-INFINITY, -INFINITY}, z_run[2] = {0.f, 0.f};
  for (int tt = chunk * chunk_keys; tt < t_end; tt += kKeyTile) {
    __syncthreads();
    key_offsets(kv, l, g, r, t0, N, tt, k_off_s);
    __syncthreads();
    load_rows(k_s, static_cast<const T*>(kv.k), k_off_s, kKeyTile, d, 1.f);
    __syncthreads();
    float x[2][4];
    dots(q_s, k_s, d, x);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      float tmax = -INFINITY;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (tt + j + 16 * m >= N) x[a][m] = -INFINITY;
        tmax = fmaxf(tmax, x[a][m]);
      }
      const float m_new = fmaxf(m_run[a], lanes_max(tmax));
      const float ref = m_new == -INFINITY ? 0.f : m_new;  // a chunk of masked keys: its sum is 0
      float psum = 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m) psum += exp2f(x[a][m] - ref);
      z_run[a] = z_run[a] * exp2f(m_run[a] - ref) + lanes_sum(psum);
      m_run[a] = m_new;
    }
  }
  if (j < 2) {
    const int rr = row0 + 2 * i + j;
    const int64_t rows_all = int64_t(gridDim.y) * kv.G * q_tot;  // of one chunk
    if (rr < R)
      stats[chunk * rows_all + int64_t(blockIdx.y) * kv.G * q_tot + int64_t(kv.G) * q0 + rr] =
          make_float2(j ? m_run[1] : m_run[0], j ? z_run[1] : z_run[0]);
  }
}

// Pass 2: one CTA per (64 tokens, layer * Hkv + g, request); loops over all row
// blocks of the slab and writes the complete column sums of its tokens, and their
// value sums of squares when ss is not NULL.
template <typename T>
__global__ void __launch_bounds__(kThreads) colsum_kernel(KvDev kv, BatchDev b, const T* q, int32_t q_tot,
                                                          const __grid_constant__ LayerList layers, int chunk_keys,
                                                          int chunks, const float2* stats, float* pa, float* pa2,
                                                          const float* extra_lse, float* ss) {
  extern __shared__ __align__(16) float smem[];
  const int d = kv.d;
  float* q_s = smem;
  float* k_s = smem + kRowTile * row_stride(d);
  __shared__ int64_t q_off_s[kRowTile], k_off_s[kKeyTile];
  __shared__ float lse_s[kRowTile];
  __shared__ float red_s[kRowTile / 2][kKeyTile + 1];

  const int r = blockIdx.z;
  const int li = blockIdx.y / kv.Hkv, g = blockIdx.y % kv.Hkv, l = layers.ids[li];
  const int t0 = b.tok_off[r], N = b.tok_off[r + 1] - t0;
  const int tt = blockIdx.x * kKeyTile;
  if (tt >= N) return;
  const int q0 = b.q_off[r], nq = b.q_off[r + 1] - q0, R = kv.G * nq;
  const int64_t rows_all = int64_t(gridDim.y) * kv.G * q_tot;
  const float2* st_slab = stats + int64_t(blockIdx.y) * kv.G * q_tot + int64_t(kv.G) * q0;
  const int64_t out0 = int64_t(blockIdx.y) * kv.n_tot + t0 + tt;

  key_offsets(kv, l, g, r, t0, N, tt, k_off_s);
  row_offsets(kv, l, g, q0, nq, q_tot, 0, q_off_s);
  __syncthreads();
  load_rows(k_s, static_cast<const T*>(kv.k), k_off_s, kKeyTile, d, 1.f);
  load_rows(q_s, q, q_off_s, kRowTile, d, kLog2e * rsqrtf(float(d)));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (ss != nullptr) {  // the eight rows of a warp are read before the first is written
    constexpr int kTok = kKeyTile / (kThreads / 32);
    float sq[kTok];
#pragma unroll
    for (int n = 0; n < kTok; ++n) {
      const int64_t o = k_off_s[warp + n * (kThreads / 32)];
      sq[n] = o >= 0 ? warp_row_sumsq(static_cast<const T*>(kv.v) + o, d, lane) : 0.f;
    }
#pragma unroll
    for (int n = 0; n < kTok; ++n) {
      const int t = warp + n * (kThreads / 32);
      if (lane == 0 && tt + t < N) ss[out0 + t] = sq[n];
    }
  }

  const int i = threadIdx.x / 16, j = threadIdx.x % 16;
  const int n_chunks = (N + chunk_keys - 1) / chunk_keys;
  float acc[4] = {0.f, 0.f, 0.f, 0.f}, acc2[4] = {0.f, 0.f, 0.f, 0.f};
  for (int row0 = 0; row0 < R; row0 += kRowTile) {
    if (row0 > 0) {
      __syncthreads();
      row_offsets(kv, l, g, q0, nq, q_tot, row0, q_off_s);
      __syncthreads();
      load_rows(q_s, q, q_off_s, kRowTile, d, kLog2e * rsqrtf(float(d)));
    }
    if (threadIdx.x < kRowTile) {
      const int rr = row0 + threadIdx.x;
      float lse = 0.f;
      if (rr < R) {
        float m = -INFINITY, z = 0.f;  // (max, sum) over the chunks, in order
        for (int c = 0; c < n_chunks; ++c) m = fmaxf(m, st_slab[c * rows_all + rr].x);
        for (int c = 0; c < n_chunks; ++c) {
          const float2 st = st_slab[c * rows_all + rr];
          z += n_chunks == 1 ? st.y : st.y * exp2f(st.x - m);
        }
        lse = m + log2f(z);
        if (extra_lse) {  // full-context softmax: keys outside the visual span join the denominator
          const int h = g * kv.G + rr / nq, qi = rr % nq;
          lse = log2_add(lse, extra_lse[(int64_t(l) * kv.Hq + h) * q_tot + q0 + qi] * kLog2e);
        }
      }
      lse_s[threadIdx.x] = lse;
    }
    __syncthreads();
    float x[2][4];
    dots(q_s, k_s, d, x);
    const float lse0 = lse_s[2 * i], lse1 = lse_s[2 * i + 1];
    const bool ok0 = row0 + 2 * i < R, ok1 = row0 + 2 * i + 1 < R;  // rows past the last add nothing
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float p0 = ok0 ? exp2f(x[0][m] - lse0) : 0.f, p1 = ok1 ? exp2f(x[1][m] - lse1) : 0.f;
      acc[m] += p0 + p1;
      if (pa2) acc2[m] += fmaf(p0, p0, p1 * p1);
    }
  }
  // sum over the 16 row pairs, in order
  auto reduce = [&](const float (&a)[4], float* out) {
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 4; ++m) red_s[i][j + 16 * m] = a[m];
    __syncthreads();
    if (threadIdx.x < kKeyTile && tt + threadIdx.x < N) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < kRowTile / 2; ++w) sum += red_s[w][threadIdx.x];
      out[out0 + threadIdx.x] = sum;
    }
  };
  reduce(acc, pa);
  if (pa2) reduce(acc2, pa2);
}

}  // namespace

// Chunks of keys pass 1 takes: enough that its blocks (32 rows of a slab by one
// chunk) fill the GPU about twice over, whole key tiles each.
constexpr int kFillBlocks = 320;
static int key_tiles(int max_tokens) { return std::max(1, (max_tokens + kKeyTile - 1) / kKeyTile); }

int score_simt_chunks(const KvDev& kv, int n_layers, int rows, int max_tokens) {
  const int64_t blocks = std::max<int64_t>(1, int64_t(n_layers) * kv.Hkv * ((rows + kRowTile - 1) / kRowTile));
  return int(std::min<int64_t>(key_tiles(max_tokens), (kFillBlocks + blocks - 1) / blocks));
}

// Entries that hold every row's chunks. A larger call has fewer chunks, so rows x
// chunks falls as often as it rises; a workspace must serve every call smaller than
// the one it was sized for, so this takes what bounds it and never falls. Rows x
// tiles is one bound. The other: with at least rows / 32 blocks, rows x ceil(320 /
// blocks) is at most rows + 32 x 320.
size_t score_simt_stats(int64_t rows, int max_tokens) {
  return size_t(std::min(rows * key_tiles(max_tokens), rows + int64_t(kRowTile) * kFillBlocks));
}

cudaError_t launch_score_simt(const KvDev& kv, const BatchDev& b, const void* q, int32_t q_tot,
                              const LayerList& layers, int max_rows, int max_tokens, int chunks, float2* stats,
                              float* pa, float* pa2, const float* extra_lse, float* ss, cudaStream_t stream) {
  if (layers.n == 0 || max_rows == 0 || max_tokens == 0) return cudaSuccess;
  const int smem = (kRowTile + kKeyTile) * row_stride(kv.d) * int(sizeof(float));
  const int tiles = (max_tokens + kKeyTile - 1) / kKeyTile;
  const int chunk_keys = (tiles + chunks - 1) / chunks * kKeyTile;
  chunks = (max_tokens + chunk_keys - 1) / chunk_keys;
  const dim3 g1(unsigned((max_rows + kRowTile - 1) / kRowTile) * chunks, layers.n * kv.Hkv, b.R);
  const dim3 g2(tiles, layers.n * kv.Hkv, b.R);
  auto go = [&](auto* f1, auto* f2, auto* qq) -> cudaError_t {
    cudaError_t err;
    if ((err = cudaFuncSetAttribute(f1, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return err;
    if ((err = cudaFuncSetAttribute(f2, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return err;
    f1<<<g1, kThreads, smem, stream>>>(kv, b, qq, q_tot, layers, chunk_keys, chunks, stats);
    if ((err = cudaGetLastError())) return err;
    f2<<<g2, kThreads, smem, stream>>>(kv, b, qq, q_tot, layers, chunk_keys, chunks, stats, pa, pa2, extra_lse, ss);
    return cudaGetLastError();
  };
  const cudaError_t err =
      kv.dtype == CONDUIT_BF16
          ? go(rowstats_kernel<__nv_bfloat16>, colsum_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16*>(q))
          : go(rowstats_kernel<float>, colsum_kernel<float>, static_cast<const float*>(q));
  if (err) return err;
  count_launches(2);
  return cudaSuccess;
}

}  // namespace conduit
