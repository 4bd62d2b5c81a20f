// CUDA-core causal refresh attention over the patched cache (selective
// recompute, Conduit Sec. 3.1 / 4.3):
//   out[l][i][h] = sum_{j <= p_i} softmax_j(<q[l][i][h], K'[l][h/G][j]> / sqrt(d)) V'[l][h/G][j]
// One CTA per (32 query rows, KV head, layer): the request's selected rows times
// the G query heads that share the KV head, in that order, cut into tiles of 32.
// Keys stream through shared memory in tiles of 64 with an online softmax
// (running max and sum per row) in the log2 domain, up to the tile's last
// position; every K and V row is read once per tile rather than once per row.
// What bounds it on the smallest calls is the chain of tiles, so where the row
// tiles leave SMs idle a cluster of up to eight CTAs takes the key tiles of one row
// tile in turn, and each then merges a part of the rows over the cluster's (max,
// sum, partial output) through distributed shared memory, in CTA order. fp32, 50
// rows of 25 selected tokens, 256 keys of 64 dims: 87 us with one warp per row, 40
// us with one CTA per row tile, 15.5 us with four.
#include <algorithm>

#include "simt_tile.cuh"

namespace conduit {
namespace {

using namespace simt;

constexpr int kMaxSplits = 8;  // CTAs of a cluster

// kDimVecs: float4 accumulators per row and thread, ceil(d / 64)
template <typename T, int kDimVecs>
__global__ void __launch_bounds__(kThreads) refresh_simt_kernel(KvDev kv, BatchDev b, const int32_t* idx,
                                                                const int32_t* idx_off, int32_t n_sel,
                                                                const T* q_rows, T* out, int splits) {
  extern __shared__ __align__(16) float sm[];
  const int d = kv.d, G = kv.G, ld = row_stride(d);
  float* q_s = sm;                         // [32][d + 4]
  float* k_s = q_s + kRowTile * ld;        // [64][d + 4]
  float* v_s = k_s + kKeyTile * ld;        // [64][d + 4]
  float* p_s = v_s + kKeyTile * ld;        // [64][32 + 2]: P transposed
  constexpr int kPStride = kRowTile + 2;
  __shared__ int64_t q_off_s[kRowTile], k_off_s[kKeyTile];
  __shared__ int pos_s[kRowTile];
  __shared__ float2 mz_s[kRowTile];        // (max, sum) of this CTA's keys, for its cluster

  const int part = blockIdx.x % splits;    // rank in the cluster
  int tile = blockIdx.x / splits, r = 0;  // the tile's request and first row
  for (; r < b.R; ++r) {
    const int tiles = int((int64_t(idx_off[r + 1] - idx_off[r]) * G + kRowTile - 1) / kRowTile);
    if (tile < tiles) break;
    tile -= tiles;
  }
  if (r == b.R) return;
  const int g = blockIdx.y, l = blockIdx.z;
  const int i0 = idx_off[r], rows = (idx_off[r + 1] - i0) * G, row0 = tile * kRowTile;
  const int t0 = b.tok_off[r], N = b.tok_off[r + 1] - t0;
  const float scale = kLog2e * rsqrtf(float(d));

  if (threadIdx.x < kRowTile) {
    const int row = row0 + threadIdx.x;
    int64_t off = -1;
    int p = -1;
    if (row < rows) {
      const int i = i0 + row / G, h = g * G + row % G;
      p = idx[i];
      if (p >= N) p = -1;  // rows without a position are not written
      if (p >= 0) off = ((int64_t(l) * n_sel + i) * kv.Hq + h) * d;
    }
    q_off_s[threadIdx.x] = off;
    pos_s[threadIdx.x] = p;
  }
  __syncthreads();
  load_rows(q_s, q_rows, q_off_s, kRowTile, d, scale, (reinterpret_cast<uintptr_t>(q_rows) & 15) == 0);
  const int i = threadIdx.x / 16, j = threadIdx.x % 16;
  const int p_row[2] = {pos_s[2 * i], pos_s[2 * i + 1]};
  int p_max = -1;
  for (int x = 0; x < kRowTile; ++x) p_max = max(p_max, pos_s[x]);

  float m_run[2] = {-INFINITY, -INFINITY}, z_run[2] = {0.f, 0.f};
  float4 acc[2][kDimVecs];  // dims 4 j + 64 v .. + 3 of the thread's two rows
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int v = 0; v < kDimVecs; ++v) acc[a][v] = make_float4(0.f, 0.f, 0.f, 0.f);
  const T* kb = static_cast<const T*>(kv.k);
  const T* vb = static_cast<const T*>(kv.v);

  for (int j0 = part * kKeyTile; j0 <= p_max; j0 += splits * kKeyTile) {
    __syncthreads();
    if (threadIdx.x < kKeyTile) {
      const int t = j0 + threadIdx.x;
      k_off_s[threadIdx.x] = t <= p_max ? kv.row(l, g, r, int64_t(t0) + t, t) : -1;
    }
    __syncthreads();
    load_rows(k_s, kb, k_off_s, kKeyTile, d, 1.f);
    load_rows(v_s, vb, k_off_s, kKeyTile, d, 1.f);
    __syncthreads();
    float x[2][4];
    dots(q_s, k_s, d, x);
    float f[2];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      float tmax = -INFINITY;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (j0 + j + 16 * m > p_row[a]) x[a][m] = -INFINITY;
        tmax = fmaxf(tmax, x[a][m]);
      }
      const float m_new = fmaxf(m_run[a], lanes_max(tmax));
      const float ref = m_new == -INFINITY ? 0.f : m_new;  // no visible key yet: P = 0
      f[a] = exp2f(m_run[a] - ref);
      float psum = 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        x[a][m] = exp2f(x[a][m] - ref);
        psum += x[a][m];
      }
      z_run[a] = z_run[a] * f[a] + lanes_sum(psum);
      m_run[a] = m_new;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
      *reinterpret_cast<float2*>(p_s + (j + 16 * m) * kPStride + 2 * i) = make_float2(x[0][m], x[1][m]);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int v = 0; v < kDimVecs; ++v) {
        acc[a][v].x *= f[a];
        acc[a][v].y *= f[a];
        acc[a][v].z *= f[a];
        acc[a][v].w *= f[a];
      }
    __syncwarp();  // a row pair's P is written and read by the same half warp
    // A key past a row's position adds nothing, whatever its V holds. Keys past both
    // rows' are not walked: most of a last tile is such keys, and small calls are last
    // tiles (fp32, 4 layers, 12/4 heads of 64 dims, five requests of 100 tokens 20.8 ->
    // 16.7 us; 2 layers of 1 024, 28/4 heads 155 -> 117).
    auto add_keys = [&](bool masked) {
      const int n_keys = masked ? min(kKeyTile, max(p_row[0], p_row[1]) + 1 - j0) : kKeyTile;
#pragma unroll 4
      for (int jj = 0; jj < n_keys; ++jj) {
        const float2 p = *reinterpret_cast<const float2*>(p_s + jj * kPStride + 2 * i);
        const bool see0 = !masked || j0 + jj <= p_row[0], see1 = !masked || j0 + jj <= p_row[1];
#pragma unroll
        for (int v = 0; v < kDimVecs; ++v) {
          const int e = 4 * j + 64 * v;
          if (e < d) {
            const float4 vv = *reinterpret_cast<const float4*>(v_s + jj * ld + e);
            if (see0)
              acc[0][v] = make_float4(fmaf(p.x, vv.x, acc[0][v].x), fmaf(p.x, vv.y, acc[0][v].y),
                                      fmaf(p.x, vv.z, acc[0][v].z), fmaf(p.x, vv.w, acc[0][v].w));
            if (see1)
              acc[1][v] = make_float4(fmaf(p.y, vv.x, acc[1][v].x), fmaf(p.y, vv.y, acc[1][v].y),
                                      fmaf(p.y, vv.z, acc[1][v].z), fmaf(p.y, vv.w, acc[1][v].w));
          }
        }
      }
    };
    if (j0 + kKeyTile - 1 <= min(p_row[0], p_row[1]))
      add_keys(false);
    else
      add_keys(true);
  }
  if (splits > 1) {
    __syncthreads();  // k_s is free
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      if (j == 0) mz_s[2 * i + a] = make_float2(m_run[a], z_run[a]);
#pragma unroll
      for (int v = 0; v < kDimVecs; ++v) {
        const int e = 4 * j + 64 * v;
        if (e < d) *reinterpret_cast<float4*>(k_s + (2 * i + a) * ld + e) = acc[a][v];
      }
    }
    cluster_barrier();
    const int rows_part = kRowTile / splits, vecs = d / 4;
    for (int x = threadIdx.x; x < rows_part * vecs; x += kThreads) {
      const int row = part * rows_part + x / vecs, e = x % vecs * 4;
      if (pos_s[row] < 0) continue;
      float m = -INFINITY, z = 0.f;
      for (int c = 0; c < splits; ++c) m = fmaxf(m, cluster_ld(&mz_s[row].x, c));
      const float ref = m == -INFINITY ? 0.f : m;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int c = 0; c < splits; ++c) {
        const float w = exp2f(cluster_ld(&mz_s[row].x, c) - ref);
        const float4 y = cluster_ld4(k_s + row * ld + e, c);
        z = fmaf(cluster_ld(&mz_s[row].y, c), w, z);
        o = make_float4(fmaf(y.x, w, o.x), fmaf(y.y, w, o.y), fmaf(y.z, w, o.z), fmaf(y.w, w, o.w));
      }
      T* dst = out + q_off_s[row] + e;
      dst[0] = from_float<T>(o.x / z);
      dst[1] = from_float<T>(o.y / z);
      dst[2] = from_float<T>(o.z / z);
      dst[3] = from_float<T>(o.w / z);
    }
    cluster_barrier();  // no CTA leaves while another may still read its part
    return;
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    if (p_row[a] < 0) continue;
    const int64_t off = q_off_s[2 * i + a];
#pragma unroll
    for (int v = 0; v < kDimVecs; ++v) {
      const int e = 4 * j + 64 * v;
      if (e < d) {
        T* o = out + off + e;
        o[0] = from_float<T>(acc[a][v].x / z_run[a]);
        o[1] = from_float<T>(acc[a][v].y / z_run[a]);
        o[2] = from_float<T>(acc[a][v].z / z_run[a]);
        o[3] = from_float<T>(acc[a][v].w / z_run[a]);
      }
    }
  }
}

template <typename T>
cudaError_t launch(const KvDev& kv, const BatchDev& b, const int32_t* idx, const int32_t* idx_off_dev,
                   unsigned tiles, int splits, int32_t n_sel, const void* q_rows, void* out, cudaStream_t stream) {
  const int ld = row_stride(kv.d);
  const int smem = int(sizeof(float)) * ((kRowTile + 2 * kKeyTile) * ld + kKeyTile * (kRowTile + 2));
  auto go = [&](auto* f) -> cudaError_t {
    cudaError_t err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err) return err;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = splits;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(tiles * splits, kv.Hkv, kv.L);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, kv, b, idx, idx_off_dev, n_sel, static_cast<const T*>(q_rows),
                              static_cast<T*>(out), splits);
  };
  return kv.d <= 64 ? go(refresh_simt_kernel<T, 1>)
         : kv.d <= 128 ? go(refresh_simt_kernel<T, 2>) : go(refresh_simt_kernel<T, 4>);
}

}  // namespace

cudaError_t launch_refresh_simt(const KvDev& kv, const BatchDev& b, const int32_t* idx, const int32_t* idx_off_dev,
                                const int32_t* idx_off_host, int32_t n_sel, const void* q_rows, void* out,
                                cudaStream_t stream) {
  if (n_sel == 0) return cudaSuccess;
  int64_t tiles = 0;
  for (int r = 0; r < b.R; ++r)
    tiles += (int64_t(idx_off_host[r + 1] - idx_off_host[r]) * kv.G + kRowTile - 1) / kRowTile;
  if (tiles == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t err;
  if ((err = cudaGetDevice(&dev))) return err;
  if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return err;
  // the largest split that keeps one CTA per SM and a key tile for each
  const int64_t ctas = tiles * kv.Hkv * kv.L, key_tiles = (kv.n_tot + kKeyTile - 1) / kKeyTile;
  int splits = kMaxSplits;
  while (splits > 1 && (ctas * splits > sms || key_tiles < splits)) splits /= 2;
  err = kv.dtype == CONDUIT_BF16
            ? launch<__nv_bfloat16>(kv, b, idx, idx_off_dev, unsigned(tiles), splits, n_sel, q_rows, out, stream)
            : launch<float>(kv, b, idx, idx_off_dev, unsigned(tiles), splits, n_sel, q_rows, out, stream);
  if (err) return err;
  count_launches(1);
  return cudaSuccess;
}

}  // namespace conduit
