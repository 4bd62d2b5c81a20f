// Tile code shared by the CUDA-core scoring and refresh kernels (fp32 caches,
// and bf16 ones the tensor-core kernels do not take): rows of d elements as fp32
// in shared memory, d + 4 floats apart (d is a multiple of 8, so the float4 reads
// of eight consecutive rows fall into different banks), and 32 x 64 products with
// 2 x 4 of them per thread: 32 FMAs for six 16-byte reads.
#pragma once

#include "internal.cuh"

namespace conduit {
namespace simt {

constexpr int kRowTile = 32;    // query rows of a tile
constexpr int kKeyTile = 64;    // keys of a tile
constexpr int kThreads = 256;   // 16 row pairs x 16 key lanes

__host__ __device__ constexpr int row_stride(int d) { return d + 4; }

// Rows off[0 .. nrows) (element offsets; negative: a row of zeros) of src into
// dst as fp32, scaled by `scale`; 16-byte loads unless src is not `aligned` to them.
template <typename T>
__device__ __forceinline__ void load_rows(float* dst, const T* src, const int64_t* off, int nrows, int d, float scale,
                                          bool aligned = true) {
  if (!aligned) {
    for (int x = threadIdx.x; x < nrows * d; x += kThreads) {
      const int64_t o = off[x / d];
      dst[x / d * row_stride(d) + x % d] = o >= 0 ? to_float(src[o + x % d]) * scale : 0.f;
    }
    return;
  }
  constexpr int kVec = 16 / sizeof(T);
  constexpr int kBatch = 4;  // loads in flight per thread
  const int cpr = d / kVec, ld = row_stride(d), n = nrows * cpr;
  for (int x0 = threadIdx.x; x0 < n; x0 += kBatch * kThreads) {
    uint4 raw[kBatch];
    int at[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int x = x0 + k * kThreads;
      raw[k] = make_uint4(0u, 0u, 0u, 0u);
      at[k] = -1;
      if (x < n) {
        const int row = x / cpr, c = x - row * cpr;
        const int64_t o = off[row];
        at[k] = row * ld + c * kVec;
        if (o >= 0) raw[k] = __ldg(reinterpret_cast<const uint4*>(src + o) + c);
      }
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      if (at[k] < 0) continue;
      const T* vals = reinterpret_cast<const T*>(&raw[k]);
      float4* out = reinterpret_cast<float4*>(dst + at[k]);
#pragma unroll
      for (int u = 0; u < kVec / 4; ++u)
        out[u] = make_float4(to_float(vals[4 * u]) * scale, to_float(vals[4 * u + 1]) * scale,
                             to_float(vals[4 * u + 2]) * scale, to_float(vals[4 * u + 3]) * scale);
    }
  }
}

// x[a][m] = <q row 2 i + a, k row j + 16 m> for thread (i, j) = (tid / 16, tid % 16).
__device__ __forceinline__ void dots(const float* q_s, const float* k_s, int d, float (&x)[2][4]) {
  const int i = threadIdx.x / 16, j = threadIdx.x % 16, ld = row_stride(d);
  const float* q0 = q_s + 2 * i * ld;
  const float* k0 = k_s + j * ld;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int m = 0; m < 4; ++m) x[a][m] = 0.f;
  for (int e = 0; e < d; e += 4) {
    float4 q[2], k[4];
#pragma unroll
    for (int a = 0; a < 2; ++a) q[a] = *reinterpret_cast<const float4*>(q0 + a * ld + e);
#pragma unroll
    for (int m = 0; m < 4; ++m) k[m] = *reinterpret_cast<const float4*>(k0 + 16 * m * ld + e);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int m = 0; m < 4; ++m)
        x[a][m] = fmaf(q[a].w, k[m].w, fmaf(q[a].z, k[m].z, fmaf(q[a].y, k[m].y, fmaf(q[a].x, k[m].x, x[a][m]))));
  }
}

// Maximum / sum over the 16 key lanes of a row pair (a half warp).
__device__ __forceinline__ float lanes_max(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float lanes_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Barrier over the cluster's CTAs, and reads of another CTA's shared memory at the
// offset of `local` in this one's.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void* local, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(local))), "r"(rank));
  return a;
}
__device__ __forceinline__ float cluster_ld(const float* local, int rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr(local, rank)) : "memory");
  return v;
}
__device__ __forceinline__ float4 cluster_ld4(const float* local, int rank) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(cluster_addr(local, rank))
               : "memory");
  return v;
}

}  // namespace simt
}  // namespace conduit
