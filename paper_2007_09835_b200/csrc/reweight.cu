// Data-free part of the paper's pruning step, run where the weights already are (Section 4):
// the group-lasso norm of every (kernel group, kernel location), the reweighted penalty
// 1 / (norm^2 + eps) of the update rule below Eq. 3, the keep / prune decision norm > threshold,
// and the expansion of that group-level decision to the per-weight mask rt3d_pack_kgs takes.
// All three are bound by memory: the weights are read once, the decisions and the mask written once.
#include <cuda_runtime.h>

#include <cstdint>

#include "pdl.cuh"
#include "rt3d.h"

namespace rt3d {
namespace {

constexpr int kNormThreads = 256;
constexpr int kNormChunk = 2048;      // floats of one weight row that a block can reduce at a time
constexpr int kNormRun = 1024;        // ... and that it takes where groups are short enough

// log2 of the lanes that share the Ks locations of a group: the next power of two, at most a warp.
int lanes_of(int Ks) {
  int lg = 0;
  while (lg < 5 && (1 << lg) < Ks) ++lg;
  return lg;
}

// One block takes a row p of kernel groups and a run of whole groups along the input channels, at most kNormChunk
// floats of each of its g_m weight rows.  A weight row [N][Ks] is contiguous, so
// every thread reads 16 bytes (VEC) or 4 of it and adds up the g_m rows at that place in registers, with the loads of
// four rows in flight; shared memory then holds one value per (input channel, location), of which each output sums g_n.
// The former kernel, one thread per output, read runs of Ks floats that began at odd addresses, one 4-byte load each.
// 1024 x 512 x 27 fp32, 4x4 groups, the three calls of a step one after the other: 88 -> 26.9 us, this one 12.7; with chunks
// of 1024 instead of 2048 floats, one load round per thread and twice the blocks to even out the last wave, 11.0 (57 MB at
// the measured copy rate: 8.7); straight code for four rows and no divisions: 10.7.
template <int G, bool VEC>
__global__ void __launch_bounds__(kNormThreads, 8)
group_norms_kernel(const float* __restrict__ w, int M, int N, int Ks, int g_m, int g_n, int Q, int q_run, int n_runs,
                   int lg, float* __restrict__ norms) {
  pdl_entry();
  __shared__ __align__(16) float part[kNormChunk];
  const int p = blockIdx.x / n_runs, q0 = (blockIdx.x - p * n_runs) * q_run;
  const int nq = min(q_run, Q - q0);
  const int m0 = p * g_m, rows = min(g_m, M - m0);
  const long long row_len = (long long)N * Ks;
  const float* base = w + (long long)m0 * row_len + (long long)q0 * g_n * Ks;
  const int len = int(min((long long)nq * g_n * Ks, row_len - (long long)q0 * g_n * Ks));   // missing channels add 0
  auto term = [](float v) { return G == 1 ? fabsf(v) : v * v; };
  if (VEC && rows == 4) {
    for (int o = threadIdx.x * 4; o < len; o += kNormThreads * 4) {
      const float* at = base + o;
      float4 v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r, at += row_len) v[r] = __ldg(reinterpret_cast<const float4*>(at));
      *reinterpret_cast<float4*>(part + o) =
          make_float4(((term(v[0].x) + term(v[1].x)) + term(v[2].x)) + term(v[3].x), ((term(v[0].y) + term(v[1].y)) + term(v[2].y)) + term(v[3].y),
                      ((term(v[0].z) + term(v[1].z)) + term(v[2].z)) + term(v[3].z), ((term(v[0].w) + term(v[1].w)) + term(v[2].w)) + term(v[3].w));
    }
  } else if (VEC) {
    for (int o = threadIdx.x * 4; o < len; o += kNormThreads * 4) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      int i = 0;
      for (; i + 4 <= rows; i += 4) {
        float4 v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = __ldg(reinterpret_cast<const float4*>(base + (i + r) * row_len + o));
#pragma unroll
        for (int r = 0; r < 4; ++r) { s.x += term(v[r].x); s.y += term(v[r].y); s.z += term(v[r].z); s.w += term(v[r].w); }
      }
      for (; i < rows; ++i) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(base + i * row_len + o));
        s.x += term(v.x); s.y += term(v.y); s.z += term(v.z); s.w += term(v.w);
      }
      *reinterpret_cast<float4*>(part + o) = s;
    }
  } else {
    for (int o = threadIdx.x; o < len; o += kNormThreads) {
      float s = 0.f;
      int i = 0;
      for (; i + 4 <= rows; i += 4) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = __ldg(base + (i + r) * row_len + o);
#pragma unroll
        for (int r = 0; r < 4; ++r) s += term(v[r]);
      }
      for (; i < rows; ++i) s += term(__ldg(base + i * row_len + o));
      part[o] = s;
    }
  }
  __syncthreads();
  float* out = norms + ((long long)p * Q + q0) * Ks;
  for (int q = threadIdx.x >> lg; q < nq; q += kNormThreads >> lg) {       // 2^lg lanes to a group: no division
    const int cols = min(g_n, N - (q0 + q) * g_n);
    for (int k = threadIdx.x & ((1 << lg) - 1); k < Ks; k += 1 << lg) {
      const float* src = part + q * g_n * Ks + k;
      float s = 0.f;
      if (cols == 4) s = ((src[0] + src[Ks]) + src[2 * Ks]) + src[3 * Ks];
      else
        for (int j = 0; j < cols; ++j) s += src[j * Ks];
      out[q * Ks + k] = G == 1 ? s : sqrtf(s);
    }
  }
}

// Groups longer than a chunk (g_n * Ks > kNormChunk): one thread per (group, location).
template <int G>
__global__ void group_norms_wide_kernel(const float* __restrict__ w, int M, int N, int Ks, int g_m, int g_n, int Q,
                                        float* __restrict__ norms, long long total) {
  pdl_entry();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int k = int(idx % Ks);
  const long long pq = idx / Ks;
  const int q = int(pq % Q), p = int(pq / Q);
  float s = 0.f;
  for (int m = p * g_m; m < min(M, (p + 1) * g_m); ++m)
    for (int c = q * g_n; c < min(N, (q + 1) * g_n); ++c) {
      const float v = fabsf(__ldg(w + ((long long)m * N + c) * Ks + k));
      s += G == 1 ? v : v * v;
    }
  norms[idx] = G == 1 ? s : sqrtf(s);
}

template <int G>
cudaError_t launch_group_norms(const float* w, int M, int N, int Ks, int g_m, int g_n, int Q, float* norms, cudaStream_t st) {
  const int P = (M + g_m - 1) / g_m;
  if ((long long)g_n * Ks > kNormChunk) {
    const long long total = (long long)P * Q * Ks;
    LaunchSetup ls(dim3(unsigned((total + 255) / 256)), dim3(256), 0, st);
    return cudaLaunchKernelEx(&ls.cfg, group_norms_wide_kernel<G>, w, M, N, Ks, g_m, g_n, Q, norms, total);
  }
  // groups per block: a whole run, in steps of four so that every run starts on a 16-byte boundary of its row; at
  // most a quarter of a run where fewer blocks than two per SM would run
  int q_run = g_n * Ks < kNormRun ? kNormRun / (g_n * Ks) : 1;
  if ((long long)P * ((Q + q_run - 1) / q_run) < 2 * current_device_sms()) q_run = (q_run + 3) / 4;
  if (q_run > 4) q_run &= ~3;
  const bool vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0 && ((long long)N * Ks) % 4 == 0 && (q_run * g_n * Ks) % 4 == 0;
  const int n_runs = (Q + q_run - 1) / q_run, lg = lanes_of(Ks);
  LaunchSetup ls(dim3(unsigned((long long)P * n_runs)), dim3(kNormThreads), 0, st);
  return vec ? cudaLaunchKernelEx(&ls.cfg, group_norms_kernel<G, true>, w, M, N, Ks, g_m, g_n, Q, q_run, n_runs, lg, norms)
             : cudaLaunchKernelEx(&ls.cfg, group_norms_kernel<G, false>, w, M, N, Ks, g_m, g_n, Q, q_run, n_runs, lg, norms);
}

// Four norms per thread where the arrays allow it (VEC: 16-byte aligned floats, 4-byte aligned decisions).
template <bool VEC>
__global__ void reweight_kernel(const float* __restrict__ norms, long long count, float eps, float threshold,
                                float* __restrict__ penalty, uint8_t* __restrict__ keep) {
  pdl_entry();
  const long long i0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * (VEC ? 4 : 1);
  if (VEC && i0 + 4 <= count) {
    const float4 n = __ldg(reinterpret_cast<const float4*>(norms + i0));
    if (penalty)
      *reinterpret_cast<float4*>(penalty + i0) = make_float4(1.f / (n.x * n.x + eps), 1.f / (n.y * n.y + eps),
                                                             1.f / (n.z * n.z + eps), 1.f / (n.w * n.w + eps));
    if (keep)
      *reinterpret_cast<uchar4*>(keep + i0) = make_uchar4(n.x > threshold, n.y > threshold, n.z > threshold, n.w > threshold);
    return;
  }
  for (long long i = i0; i < count && i < i0 + (VEC ? 4 : 1); ++i) {
    const float n = norms[i];
    if (penalty) penalty[i] = 1.f / (n * n + eps);
    if (keep) keep[i] = n > threshold ? 1 : 0;
  }
}

constexpr int kMaskThreads = 256;
constexpr int kMaskChunk = 4096;      // bytes of one mask row that a block expands at a time

// The g_m mask rows of a row of kernel groups are the same N * Ks bytes: a block expands a chunk of them once into
// shared memory (each decision goes to the g_n channels of its group) and writes it to every row in 16-byte stores.  Chunks
// are whole groups where a group fits one; 2^lg lanes take a group's locations, so that neither needs a division or a
// test.  A row may start at any byte, so the words of a row that does not start on a 16-byte boundary are cut out of the
// staged chunk at that row's shift (funnel shifts), and only a chunk's first and last partial word go out byte by byte;
// rows with the same shift (row length a multiple of 16) share the words in registers.  Bound by its instructions:
// 1024 x 512 x 27, 4x4: 9.7 us gathering the bytes of a word, 7.2 scattering with a division and a test per byte, 5.6 now.
__global__ void __launch_bounds__(kMaskThreads)
expand_mask_kernel(const uint8_t* __restrict__ gmask, int M, int N, int Ks, int g_m, int g_n, int Q, int chunk, int q_chunk,
                   int n_chunks, int lg, uint8_t* __restrict__ mask) {
  pdl_entry();
  __shared__ __align__(16) uint32_t row_s[kMaskChunk / 4 + 12];      // [4] words of slack in front: shifts read from there
  uint8_t* bytes = reinterpret_cast<uint8_t*>(row_s + 4);
  const int p = blockIdx.x / n_chunks;
  const long long row_len = (long long)N * Ks, c0 = (long long)(blockIdx.x - p * n_chunks) * chunk;
  const int len = int(min((long long)chunk, row_len - c0));
  // the groups that the chunk touches, their decisions a contiguous run; first: where the first of them starts
  const long long span = (long long)g_n * Ks;
  int q0 = int(blockIdx.x - p * n_chunks) * q_chunk, n_q, first = 0;    // q_chunk: whole groups in a chunk, or 0
  if (q_chunk > 0) {
    n_q = min(q_chunk, Q - q0);
  } else {
    q0 = int(c0 / span);
    n_q = int((c0 + len - 1) / span) + 1 - q0;
    first = int(q0 * span - c0);
  }
  const uint8_t* g = gmask + ((long long)p * Q + q0) * Ks;
  const int k0 = threadIdx.x & ((1 << lg) - 1);
  const bool whole = q_chunk > 0;                                       // bytes beyond len are not written out
#pragma unroll 4
  for (int q = threadIdx.x >> lg; q < n_q; q += kMaskThreads >> lg)
    for (int k = k0; k < Ks; k += 1 << lg) {
      const uint8_t bit = __ldg(g + q * Ks + k);
      int o = first + q * int(span) + k;
      if (whole) {
#pragma unroll 4
        for (int j = 0; j < g_n; ++j, o += Ks) bytes[o] = bit;
      } else {
        for (int j = 0; j < g_n; ++j, o += Ks)
          if (unsigned(o) < unsigned(len)) bytes[o] = bit;
      }
    }
  __syncthreads();
  const int rows = min(g_m, M - p * g_m);
  uint8_t* dst0 = mask + (long long)(p * g_m) * row_len + c0;
  const bool same_shift = (row_len & 15) == 0;
  for (int i0 = 0; i0 < rows; i0 += same_shift ? rows : 1) {
    uint8_t* dst = dst0 + i0 * row_len;
    const int n_rows = same_shift ? rows : 1;
    const int shift = int(reinterpret_cast<uintptr_t>(dst) & 15);    // dst is `shift` bytes into its first 16-byte word
    const int n_words = (shift + len + 15) / 16;
    for (int u = threadIdx.x; u < n_words; u += kMaskThreads) {
      const int o = u * 16 - shift;                                  // first byte of the word inside the chunk
      if (o >= 0 && o + 16 <= len) {
        uint4 v;
        if (shift == 0) {
          v = *reinterpret_cast<const uint4*>(bytes + o);
        } else {
          const int w0 = (o >> 2) + 4, sh = (o & 3) * 8;
          v.x = __funnelshift_r(row_s[w0], row_s[w0 + 1], sh);
          v.y = __funnelshift_r(row_s[w0 + 1], row_s[w0 + 2], sh);
          v.z = __funnelshift_r(row_s[w0 + 2], row_s[w0 + 3], sh);
          v.w = __funnelshift_r(row_s[w0 + 3], row_s[w0 + 4], sh);
        }
        uint8_t* at = dst + o;
#pragma unroll 4
        for (int i = 0; i < n_rows; ++i, at += row_len) *reinterpret_cast<uint4*>(at) = v;
      } else {
        for (int i = 0; i < n_rows; ++i)
          for (int b = max(o, 0); b < min(o + 16, len); ++b) dst[i * row_len + b] = bytes[b];
      }
    }
  }
}

}  // namespace
}  // namespace rt3d

using namespace rt3d;

extern "C" {

rt3d_status rt3d_kgs_group_norms(const float* w, int M, int N, int Kt, int Kh, int Kw, int g_m, int g_n, int norm,
                                 float* norms, void* stream) {
  if (!w || !norms || M <= 0 || N <= 0 || Kt <= 0 || Kh <= 0 || Kw <= 0 || g_m <= 0 || g_n <= 0) return RT3D_ERR_INVALID_ARG;
  if (norm != 1 && norm != 2) return RT3D_ERR_INVALID_ARG;
  const int Ks = Kt * Kh * Kw;
  const int Q = (N + g_n - 1) / g_n;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const cudaError_t e = norm == 1 ? launch_group_norms<1>(w, M, N, Ks, g_m, g_n, Q, norms, st)
                                  : launch_group_norms<2>(w, M, N, Ks, g_m, g_n, Q, norms, st);
  return e == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
}

rt3d_status rt3d_kgs_reweight(const float* norms, int64_t count, float eps, float threshold, float* penalty,
                              uint8_t* keep, void* stream) {
  if (!norms || count <= 0 || (!penalty && !keep) || !(eps > 0.f)) return RT3D_ERR_INVALID_ARG;
  const uintptr_t f = reinterpret_cast<uintptr_t>(norms) | reinterpret_cast<uintptr_t>(penalty);
  const bool vec = (f & 15) == 0 && (reinterpret_cast<uintptr_t>(keep) & 3) == 0;
  const long long threads = vec ? (count + 3) / 4 : count;
  LaunchSetup ls(dim3(unsigned((threads + 255) / 256)), dim3(256), 0, static_cast<cudaStream_t>(stream));
  const cudaError_t e = vec ? cudaLaunchKernelEx(&ls.cfg, reweight_kernel<true>, norms, (long long)count, eps, threshold, penalty, keep)
                            : cudaLaunchKernelEx(&ls.cfg, reweight_kernel<false>, norms, (long long)count, eps, threshold, penalty, keep);
  return e == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
}

rt3d_status rt3d_kgs_expand_mask(const uint8_t* group_mask, int M, int N, int Kt, int Kh, int Kw, int g_m, int g_n,
                                 uint8_t* mask, void* stream) {
  if (!group_mask || !mask || M <= 0 || N <= 0 || Kt <= 0 || Kh <= 0 || Kw <= 0 || g_m <= 0 || g_n <= 0) return RT3D_ERR_INVALID_ARG;
  const int Ks = Kt * Kh * Kw;
  const int Q = (N + g_n - 1) / g_n;
  // whole groups per chunk, sixteen of them at a time so that chunks start on 16-byte boundaries of the row
  const long long span = (long long)g_n * Ks;
  int chunk = kMaskChunk;
  if (span * 16 <= kMaskChunk) chunk = int(kMaskChunk / (span * 16) * (span * 16));
  else if (span <= kMaskChunk) chunk = int(kMaskChunk / span * span);
  const int P = (M + g_m - 1) / g_m, n_chunks = int(((long long)N * Ks + chunk - 1) / chunk);
  const int lg = lanes_of(Ks);
  LaunchSetup ls(dim3(unsigned((long long)P * n_chunks)), dim3(kMaskThreads), 0, static_cast<cudaStream_t>(stream));
  const cudaError_t e = cudaLaunchKernelEx(&ls.cfg, expand_mask_kernel, group_mask, M, N, Ks, g_m, g_n, Q, chunk, span <= kMaskChunk ? int(chunk / span) : 0, n_chunks, lg, mask);
  return e == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
}

}  // extern "C"
