// Builds the tensor-core weight tiles on the device from the canonical packed arrays.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace rt3d {
namespace {

// One warp per packed entry: the entry's group is found in group_ptr (all lanes search alike, so every probe is one
// transaction) and its g_m x g_n values go to their rows of the step's tile.  A few microseconds for a million values;
// what it saves is building zero-filled tiles on the host and copying them.
__global__ void __launch_bounds__(256)
fill_umma_tiles_kernel(const int32_t* __restrict__ group_ptr, const uint16_t* __restrict__ pos_idx,
                       const uint16_t* __restrict__ tiles, const int32_t* __restrict__ slots, int M, int N, int Ks,
                       int g_m, int g_n, int Q, int n_groups, int nnz, int n_tile, int n_chunks, uint16_t* __restrict__ wtiles) {
  const int lane = threadIdx.x & 31, size = g_m * g_n;
  for (long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < nnz; e += (long long)gridDim.x * (blockDim.x >> 5)) {
    int lo = 0, hi = n_groups - 1;                     // last group that starts at or before e (empty groups share a start)
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(group_ptr + mid) <= e) lo = mid;
      else hi = mid - 1;
    }
    const int p = lo / Q, q = lo - p * Q, k = __ldg(pos_idx + e);
    const uint16_t* src = tiles + e * size;
    for (int v = lane; v < size; v += 32) {
      const int i = v / g_n, m = p * g_m + i, c = q * g_n + (v - i * g_n);
      if (m >= M || c >= N) continue;
      const int b = m / n_tile;
      const long long s = __ldg(slots + ((long long)b * Ks + k) * n_chunks + (c >> 6));
      wtiles[(s * n_tile + (m - b * n_tile)) * 64 + (c & 63)] = src[v];
    }
  }
}

}  // namespace

cudaError_t launch_fill_umma_tiles(const int32_t* group_ptr, const uint16_t* pos_idx, const void* tiles, const int32_t* slots,
                                   int M, int N, int Ks, int g_m, int g_n, int Q, int n_groups, int64_t nnz, int n_tile,
                                   int n_chunks, void* wtiles, size_t bytes) {
  cudaError_t e = cudaMemsetAsync(wtiles, 0, bytes, cudaStreamLegacy);
  if (e != cudaSuccess || nnz == 0) return e;
  const int64_t blocks = (nnz + 7) / 8;
  fill_umma_tiles_kernel<<<unsigned(blocks < 65536 ? blocks : 65536), 256, 0, cudaStreamLegacy>>>(
      group_ptr, pos_idx, static_cast<const uint16_t*>(tiles), slots, M, N, Ks, g_m, g_n, Q, n_groups, int(nnz), n_tile, n_chunks,
      static_cast<uint16_t*>(wtiles));
  return cudaGetLastError();
}

}  // namespace rt3d
