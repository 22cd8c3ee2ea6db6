// Builds the tensor-core weight tiles on the device from the canonical packed arrays.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace rt3d {
namespace {

// Last group that starts at or before entry e (empty groups share a start).
__device__ __forceinline__ int group_of(const int32_t* group_ptr, int n_groups, long long e) {
  int lo = 0, hi = n_groups - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(group_ptr + mid) <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One warp per packed entry: the entry's group is found in group_ptr (all lanes search alike, so every probe is one
// transaction) and its g_m x g_n values go to their rows of the step's tile.  A few microseconds for a million values;
// what it saves is building zero-filled tiles on the host and copying them.
__global__ void __launch_bounds__(256)
fill_umma_tiles_kernel(const int32_t* __restrict__ group_ptr, const uint16_t* __restrict__ pos_idx,
                       const uint16_t* __restrict__ tiles, const int32_t* __restrict__ slots, int M, int N, int Ks,
                       int g_m, int g_n, int Q, int n_groups, int nnz, int n_tile, int chunk_bits, int n_chunks, uint16_t* __restrict__ wtiles) {
  const int lane = threadIdx.x & 31, size = g_m * g_n;
  for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < nnz; e += (long long)gridDim.x * (blockDim.x >> 5)) {
    const int lo = group_of(group_ptr, n_groups, e);
    const int p = lo / Q, q = lo - p * Q, k = __ldg(pos_idx + e);
    const uint16_t* src = tiles + e * size;
    for (int v = lane; v < size; v += 32) {
      const int i = v / g_n, m = p * g_m + i, c = q * g_n + (v - i * g_n);
      if (m >= M || c >= N) continue;
      const int b = m / n_tile;
      const long long s = __ldg(slots + ((long long)b * Ks + k) * n_chunks + (c >> chunk_bits));
      wtiles[((s * n_tile + (m - b * n_tile)) << chunk_bits) + (c & ((1 << chunk_bits) - 1))] = src[v];
    }
  }
}

// The same for fp32 weights in three bf16 parts.  A step's weights are one or two (for the CTAs of a pair) runs of rows, each
// [16 channels][8 channels][part][row][8 values]: operands without swizzle, core matrices of 8 rows x 8 values in 128 bytes,
// the rows of the three parts one after the other.
__global__ void __launch_bounds__(256)
fill_split_tiles_kernel(const int32_t* __restrict__ group_ptr, const uint16_t* __restrict__ pos_idx, const float* __restrict__ tiles,
                        const int32_t* __restrict__ slots, int M, int N, int Ks, int g_m, int g_n, int Q, int n_groups, int nnz,
                        int n_tile, int halves, int n_chunks, __nv_bfloat16* __restrict__ wtiles) {
  const int lane = threadIdx.x & 31, size = g_m * g_n, rows = n_tile / halves;
  for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < nnz; e += (long long)gridDim.x * (blockDim.x >> 5)) {
    const int lo = group_of(group_ptr, n_groups, e);
    const int p = lo / Q, q = lo - p * Q, k = __ldg(pos_idx + e);
    for (int v = lane; v < size; v += 32) {
      const int i = v / g_n, m = p * g_m + i, c = q * g_n + (v - i * g_n);
      if (m >= M || c >= N) continue;
      const int b = m / n_tile, row = m - b * n_tile, half = row / rows, r = row - half * rows, cc = c & 31;
      const long long s = __ldg(slots + ((long long)b * Ks + k) * n_chunks + (c >> 5));
      __nv_bfloat16* dst = wtiles + s * (n_tile * 96) + half * (rows * 96) + (cc >> 3) * (rows * 24) + r * 8 + (cc & 7);
      float w = tiles[e * size + v];
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        const __nv_bfloat16 h = __float2bfloat16_rn(w);
        dst[part * (rows * 8)] = h;
        w -= __bfloat162float(h);
      }
    }
  }
}

// Returns this launch's own error: the runtime's last one may be an earlier call's, a caller's among them.
template <typename... P, typename... A>
cudaError_t launch_fill(void (*kernel)(P...), int64_t blocks, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(blocks < 65536 ? blocks : 65536));
  cfg.blockDim = dim3(256);
  cfg.stream = cudaStreamLegacy;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace

cudaError_t launch_fill_split_tiles(const int32_t* group_ptr, const uint16_t* pos_idx, const float* tiles, const int32_t* slots,
                                    int M, int N, int Ks, int g_m, int g_n, int Q, int n_groups, int64_t nnz, int n_tile,
                                    int halves, int n_chunks, void* wtiles, size_t bytes) {
  cudaError_t e = cudaMemsetAsync(wtiles, 0, bytes, cudaStreamLegacy);
  if (e != cudaSuccess || nnz == 0) return e;
  const int64_t blocks = (nnz + 7) / 8;
  return launch_fill(fill_split_tiles_kernel, blocks, group_ptr, pos_idx, tiles, slots, M, N, Ks, g_m, g_n, Q, n_groups, int(nnz), n_tile, halves,
                     n_chunks, static_cast<__nv_bfloat16*>(wtiles));
}

cudaError_t launch_fill_umma_tiles(const int32_t* group_ptr, const uint16_t* pos_idx, const void* tiles, const int32_t* slots,
                                   int M, int N, int Ks, int g_m, int g_n, int Q, int n_groups, int64_t nnz, int n_tile,
                                   int chunk, int n_chunks, void* wtiles, size_t bytes) {
  cudaError_t e = cudaMemsetAsync(wtiles, 0, bytes, cudaStreamLegacy);
  if (e != cudaSuccess || nnz == 0) return e;
  const int64_t blocks = (nnz + 7) / 8;
  return launch_fill(fill_umma_tiles_kernel, blocks, group_ptr, pos_idx, static_cast<const uint16_t*>(tiles), slots, M, N, Ks, g_m, g_n, Q, n_groups,
                     int(nnz), n_tile, chunk == 32 ? 5 : 6, n_chunks, static_cast<uint16_t*>(wtiles));
}

}  // namespace rt3d
