// fp32 KGS convolution on the CUDA cores, register-blocked: exact fp32 FMAs, pruned (group, location) places skipped.
//
// A warp owns 16 * V output voxels and one set of two rows of four output channels; neighbouring lanes share their voxels
// and halve the four channels of a row.  The input block under the output box of a thread block is staged in shared
// memory, a few quads of input channels at a time ([quad][voxel][4 channels], zero outside the tensor), together with
// the stage's index entries and weight tiles.  Per entry, a (quad, location) place, a thread loads V input quads and
// multiplies them with the 4 x 4 tile of each row that keeps the place.  The entries come in three lists (kept by both
// rows, by the first, by the second), so the loops hold no test and nothing diverges.
//
// Bound: fp32 FMA issue.  The FMAs are the packed fma.rn.f32x2 (two independent, individually rounded FMAs), here an even
// and an odd input channel, added at the end: measured on B200, plain FFMA reaches 57 TFLOP/s of the 74 of the packed
// form, which leaves every second issue slot to the loads.  Beside that the shared-memory reads set the shape: a 16-byte
// load costs two cycles an SM whether all lanes read one address or pairs of lanes 16 voxels, a row's tile takes two
// loads a lane and a place V, against 8 V cycles of packed FMAs a row.  Two rows and V = 8 keep the reads at 0.85 of the
// FMA time (0.4 of the places kept) in 128 registers, i.e. with four warps a scheduler.  Tests on a mask of rows instead
// of the lists, with 4 or 8 rows a set, ran at 0.4 of the FMA rate: every test is a dependent branch.  A thread's voxels
// lie at distances that are the same for all lanes, so that one address register serves all V loads (a register each:
// 655 us instead of 524).  Measured, 0.4 of the places kept: 64 -> 128 channels, 3x3x3, 2 x 16 x 56 x 56 voxels 2475 ->
// 524 us (7.2 -> 34 TFLOP/s kept); 16 -> 32 channels, 8 x 28 x 28 voxels 27.4 -> 9.6 us, half of it launch and latency.
//
// Small calls leave an SM too few warps, each a serial chain of entries, or too few voxels a thread.  There `parts` warps
// share a set and its voxels, each takes its part of every list, and the first adds up the others' sums, in order, through
// shared memory: the call of 8 x 28 x 28 voxels 10.1 -> 9.2 us, 64 -> 128 channels on 4 x 14 x 14 26 -> 20 us.
//
// Two buffers; the copies of stage s + 1 (cp.async) run while stage s is multiplied.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "kernels.h"
#include "pdl.cuh"
#include "rt3d_internal.h"

namespace rt3d {
namespace {

constexpr int kThreadsF32 = 256;
constexpr int kKoffMax = 512;                        // kernel locations (the layout refuses more)

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void lds_pairs(uint32_t addr, f32x2& a, f32x2& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr));
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
// 16 bytes of which the first `bytes` are read and the rest zero-filled.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// Shared memory: two buffers of {weight tiles, staged input, entries}, then the tables.
struct F32Smem {
  int tile_bytes, x_bytes, entry_bytes, buffer_bytes, total;
};
__host__ __device__ inline F32Smem f32_smem(int max_tiles, int max_entries, int quads, int voxels, int sum_bytes = 0) {
  F32Smem s;
  s.tile_bytes = max_tiles * 64;
  s.x_bytes = quads * voxels * 16;
  s.entry_bytes = ((max_entries + 1) * 4 + 15) & ~15;              // one past the end is read ahead
  s.buffer_bytes = s.tile_bytes + s.x_bytes + s.entry_bytes;
  s.total = 2 * s.buffer_bytes + kKoffMax * 4 + voxels * 4;
  if (s.total < sum_bytes) s.total = sum_bytes;
  return s;
}

// The entries of one list: `first` .. `last` say which of the set's two rows they feed.  Entry and tile pointers advance.
template <int V, int first, int last>
__device__ __forceinline__ void run_list(int n, uint32_t& ep, uint32_t& wp, uint32_t x_lane, const uint32_t (&delta)[V],
                                         f32x2 (&acc)[2][V][2]) {
  if (n <= 0) return;
  uint32_t xp = x_lane + lds32(ep);
#pragma unroll 1
  for (int e = 0; e < n; ++e) {
    f32x2 x[V][2];
#pragma unroll
    for (int v = 0; v < V; ++v) lds_pairs(xp + delta[v], x[v][0], x[v][1]);
    ep += 4;
    xp = x_lane + lds32(ep);                         // the next entry's (past the last one: a word that is not used)
#pragma unroll
    for (int r = first; r <= last; ++r) {
      f32x2 w[2][2];
#pragma unroll
      for (int o = 0; o < 2; ++o) lds_pairs(wp + o * 16, w[o][0], w[o][1]);
      wp += 64;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int o = 0; o < 2; ++o) acc[r][v][o] = fma2(x[v][j], w[o][j], acc[r][v][o]);
    }
  }
}

template <int V, bool kParts>
__global__ void __launch_bounds__(kThreadsF32, 2)
conv3d_f32_kernel(const F32Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const ConvGeom& g = a.g;
  const int halo = a.ht * a.hh * a.hw;
  const F32Smem sm = f32_smem(a.max_tiles, a.max_entries, a.quads, halo);
  const uint32_t base = smem_addr(smem);
  int* koff_s = reinterpret_cast<int*>(smem + 2 * sm.buffer_bytes);        // kernel location -> byte offset in a plane
  int* vox_s = koff_s + kKoffMax;                                          // staged voxel -> input voxel, or -1
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int parts = kParts ? a.parts : 1, part = kParts ? warp % parts : 0;
  const int voxel_warps = (kThreadsF32 / 32) / a.sets / parts, slot = kParts ? warp / parts : warp;
  const int set_local = slot / voxel_warps, vw = slot - set_local * voxel_warps;
  const int set0 = blockIdx.y * a.sets, n_here = min(a.sets, a.n_sets - set0);

  int tile = blockIdx.x;
  const int w0 = (tile % a.tiles_w) * a.bw; tile /= a.tiles_w;
  const int h0 = (tile % a.tiles_h) * a.bh; tile /= a.tiles_h;
  const int t0 = (tile % a.tiles_t) * a.bt;
  const int nn = tile / a.tiles_t;

  for (int k = threadIdx.x; k < g.Kt * g.Kh * g.Kw; k += kThreadsF32) {
    const int kw = k % g.Kw, kh = (k / g.Kw) % g.Kh, kt = k / (g.Kw * g.Kh);
    koff_s[k] = ((kt * a.hh + kh) * a.hw + kw) * 16;
  }
  for (int i = threadIdx.x; i < halo; i += kThreadsF32) {
    const int w = i % a.hw, h = (i / a.hw) % a.hh, t = i / (a.hw * a.hh);
    const int ti = t0 * g.st - g.pt + t * a.ht_step, hi = h0 * g.sh - g.ph + h * a.hh_step, wi = w0 * g.sw - g.pw + w * a.hw_step;
    const bool in = unsigned(ti) < unsigned(g.t) && unsigned(hi) < unsigned(g.h) && unsigned(wi) < unsigned(g.w);
    vox_s[i] = in ? ((nn * g.t + ti) * g.h + hi) * g.w + wi : -1;
  }
  // this lane's first voxel, and the others at distances that are the same for all lanes
  const int lt = a.bt / a.vt, lh = a.bh / a.vh;
  const int pos = min(vw * 16 + (lane >> 1), lt * lh * a.bw - 1);
  const int lw_i = pos % a.bw, lh_i = (pos / a.bw) % lh, lt_i = pos / (a.bw * lh);
  const int st_s = a.ht_step > 1 ? 1 : g.st, sh_s = a.hh_step > 1 ? 1 : g.sh, sw_s = a.hw_step > 1 ? 1 : g.sw;
  const uint32_t vox_off = uint32_t(((lt_i * st_s * a.hh + lh_i * sh_s) * a.hw + lw_i * sw_s) * 16);
  uint32_t delta[V];
#pragma unroll
  for (int v = 0; v < V; ++v)
    delta[v] = uint32_t((((v / a.vh) * lt * st_s) * a.hh + (v % a.vh) * lh * sh_s) * a.hw * 16);

  auto issue_weights = [&](int st, int buf) {
    const int i0 = st * a.n_sets + set0;
    const int e0 = __ldg(a.entry_ptr + i0), n_e = __ldg(a.entry_ptr + i0 + n_here) - e0;
    const int w0_ = __ldg(a.tile_ptr + i0), n_w = __ldg(a.tile_ptr + i0 + n_here) - w0_;
    const uint32_t dst = base + buf * sm.buffer_bytes;
    for (int i = threadIdx.x; i < n_w * 4; i += kThreadsF32) cp_async16(dst + i * 16, a.tiles + (size_t(w0_) * 16 + size_t(i) * 4), 16);
    for (int i = threadIdx.x; i < n_e; i += kThreadsF32) cp_async4(dst + sm.tile_bytes + sm.x_bytes + i * 4, a.entries + e0 + i);
  };
  auto issue_input = [&](int st, int buf) {
    const uint32_t dst = base + buf * sm.buffer_bytes + sm.tile_bytes;
    const int lg = a.quads == 2 ? 1 : a.quads == 4 ? 2 : 3;
    const int c_base = st * a.quads * 4;
    for (int i = threadIdx.x; i < halo << lg; i += kThreadsF32) {
      const int voxel = i >> lg, quad = i & (a.quads - 1), c0 = c_base + quad * 4;
      const int src = vox_s[voxel];
      const int bytes = src < 0 ? 0 : max(0, min(16, (g.c - c0) * 4));      // channels beyond the last are not read
      const float* p = bytes > 0 ? a.x + (long long)src * g.xcs + c0 : a.x;
      cp_async16(dst + (quad * halo + voxel) * 16, p, bytes);
    }
  };

  f32x2 acc[2][V][2];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int v = 0; v < V; ++v) acc[r][v][0] = acc[r][v][1] = 0ull;

  issue_weights(0, 0);                               // the handle's arrays: no kernel writes them
  pdl_entry();
  __syncthreads();                                   // tables
  issue_input(0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int st = 0; st < a.n_stages; ++st) {
    const int buf = st & 1;
    if (st + 1 < a.n_stages) {
      issue_weights(st + 1, buf ^ 1);
      issue_input(st + 1, buf ^ 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    {                                                // entries become byte offsets, each by the thread that copied it
      const int i0 = st * a.n_sets + set0, n_e = __ldg(a.entry_ptr + i0 + n_here) - __ldg(a.entry_ptr + i0);
      uint32_t* ent = reinterpret_cast<uint32_t*>(smem + buf * sm.buffer_bytes + sm.tile_bytes + sm.x_bytes);
      for (int i = threadIdx.x; i < n_e; i += kThreadsF32) ent[i] = uint32_t(koff_s[ent[i] & 0xffffu]) + (ent[i] >> 16) * (halo * 16u);
    }
    __syncthreads();
    if (set_local < n_here) {
      const int i0 = st * a.n_sets + set0;
      const int e0 = __ldg(a.entry_ptr + i0), es = __ldg(a.entry_ptr + i0 + set_local), n_e = __ldg(a.entry_ptr + i0 + set_local + 1) - es;
      const int t0_ = __ldg(a.tile_ptr + i0), counts = __ldg(a.counts + i0 + set_local);
      const int n_both = counts & 0xffff, n_first = counts >> 16;
      const uint32_t b0 = base + buf * sm.buffer_bytes;
      uint32_t wp = b0 + uint32_t(__ldg(a.tile_ptr + i0 + set_local) - t0_) * 64u + (lane & 1) * 32;   // this lane's two outputs
      uint32_t ep = b0 + sm.tile_bytes + sm.x_bytes + (es - e0) * 4;
      const uint32_t x_lane = b0 + sm.tile_bytes + vox_off;
      if constexpr (!kParts) {
        run_list<V, 0, 1>(n_both, ep, wp, x_lane, delta, acc);
        run_list<V, 0, 0>(n_first, ep, wp, x_lane, delta, acc);
        run_list<V, 1, 1>(n_e - n_both - n_first, ep, wp, x_lane, delta, acc);
      } else {
        const auto mine = [&](int n, int rows, auto run) {             // this warp's part of the next list
          const int from = n * part / parts, to = n * (part + 1) / parts;
          uint32_t ep_at = ep + from * 4, wp_at = wp + from * rows * 64;
          run(to - from, ep_at, wp_at);
          ep += n * 4;
          wp += n * rows * 64;
        };
        mine(n_both, 2, [&](int n, uint32_t& e, uint32_t& w) { run_list<V, 0, 1>(n, e, w, x_lane, delta, acc); });
        mine(n_first, 1, [&](int n, uint32_t& e, uint32_t& w) { run_list<V, 0, 0>(n, e, w, x_lane, delta, acc); });
        mine(n_e - n_both - n_first, 1, [&](int n, uint32_t& e, uint32_t& w) { run_list<V, 1, 1>(n, e, w, x_lane, delta, acc); });
      }
    }
    __syncthreads();
  }

  if (kParts) {                                      // the buffers are free: the other parts' sums, [part][register][lane]
    f32x2* sums = reinterpret_cast<f32x2*>(smem) + (set_local * voxel_warps + vw) * (parts - 1) * (V * 128) + lane;
    if (part > 0)
#pragma unroll
      for (int i = 0; i < 4 * V; ++i) sums[(part - 1) * (V * 128) + i * 32] = acc[i / (2 * V)][(i / 2) % V][i & 1];
    __syncthreads();
    if (part > 0) return;
    for (int p = 0; p < parts - 1; ++p)
#pragma unroll
      for (int i = 0; i < 4 * V; ++i) acc[i / (2 * V)][(i / 2) % V][i & 1] = add2(acc[i / (2 * V)][(i / 2) % V][i & 1], sums[p * (V * 128) + i * 32]);
  }

  // bias, residual, ReLU; a pair of lanes writes the 16 bytes of a (voxel, row)
  if (set_local >= n_here || vw * 16 + (lane >> 1) >= lt * lh * a.bw) return;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int w = w0 + lw_i, h = h0 + lh_i + (v % a.vh) * lh, t = t0 + lt_i + (v / a.vh) * lt;
    if (t >= g.To || h >= g.Ho || w >= g.Wo) continue;
    const long long vox = (((long long)nn * g.To + t) * g.Ho + h) * g.Wo + w;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int m = ((set0 + set_local) * 2 + r) * 4 + (lane & 1) * 2;
      if (m >= g.M) break;
      const float2 a0 = unpack2(acc[r][v][0]), a1 = unpack2(acc[r][v][1]);
      float2 o = make_float2(a0.x + a0.y, a1.x + a1.y);
      float* yp = a.y + vox * g.ycs + m;
      const float* rp = a.residual ? a.residual + vox * a.rcs + m : nullptr;
      const bool both = m + 1 < g.M;
      if (a.bias) { o.x += __ldg(a.bias + m); if (both) o.y += __ldg(a.bias + m + 1); }
      if (rp) { o.x += rp[0]; if (both) o.y += rp[1]; }
      if (g.relu) { o.x = fmaxf(o.x, 0.f); o.y = fmaxf(o.y, 0.f); }
      if (both) *reinterpret_cast<float2*>(yp) = o;
      else yp[0] = o.x;
    }
  }
}

template <int V, bool kParts>
cudaError_t launch_t(const F32Args& a, dim3 grid, size_t smem, cudaStream_t stream) {
  static bool attr_done[kMaxDevices] = {};             // the attribute is per device
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(conv3d_f32_kernel<V, kParts>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  LaunchSetup ls(grid, dim3(kThreadsF32), smem, stream);
  return cudaLaunchKernelEx(&ls.cfg, conv3d_f32_kernel<V, kParts>, a);
}

int f32_sum_bytes(int voxels, int parts) { return (kThreadsF32 / 32) / parts * (parts - 1) * voxels * 1024; }

int staged(int out, int kernel, int stride) { return kernel == 1 ? out : (out - 1) * stride + kernel; }

// Output box of at most `lanes` positions times `voxels` = vt * vh of them along t and h, inside one clip: fewest boxes, a
// staged voxel counted as `weight` of an output.
double choose_box_f32(const ConvGeom& g, int lanes, int voxels, double weight, F32Plan* p) {
  double best = -1.0;
  for (int vh = 1; vh <= voxels; vh *= 2) {
    const int vt = voxels / vh;
    for (int bw = 1; bw <= g.Wo && bw <= lanes; ++bw) {
      if (bw < g.Wo && bw % 8 && bw != 4) continue;    // whole rows, or runs of 64 bytes and more
      for (int lh = 1; lh <= ceil_div(g.Ho, vh) && bw * lh <= lanes; ++lh) {
        const int most_t = ceil_div(g.To, vt), lt = lanes / (bw * lh) < most_t ? lanes / (bw * lh) : most_t;
        const int bt = lt * vt, bh = lh * vh;
        const double boxes = double(ceil_div(g.To, bt)) * ceil_div(g.Ho, bh) * ceil_div(g.Wo, bw);
        const double halo = double(staged(bt, g.Kt, g.st)) * staged(bh, g.Kh, g.sh) * staged(bw, g.Kw, g.sw);
        // eight lanes' quads pass at a time: rows of 8 or more voxels keep their banks apart, narrower ones collide
        const double banks = bw % 8 == 0 ? 1.0 : bw > 8 ? 1.0 + 1.0 / bw : 1.3;
        const double cost = boxes * (lanes * voxels * banks + weight * halo);
        if (best < 0 || cost < best) { best = cost; p->bt = bt; p->bh = bh; p->bw = bw; p->vt = vt; p->vh = vh; }
      }
    }
  }
  return best;
}

}  // namespace

// Cycles of the busiest SM for every variant, fitted to timings on B200: an entry costs a scheduler 25 + V (4 + 10 h) with
// four warps at work (h = tiles per entry) and a warp by itself 45 + V (12 + 30 h); a stage costs its copies and barriers, adding up the parts 220 V for each and 800.
static int search_plans(const ConvGeom& g, double density, int sm_count, F32Plan plans[kF32MaxPlans], double* cycles) {
  const int Ks = g.Kt * g.Kh * g.Kw, n_rows = ceil_div(g.M, 4), n_quads = ceil_div(g.c, 4), quads = f32_stage_quads(Ks);
  const int n_stages = ceil_div(n_quads, quads);
  double cost[kF32MaxPlans];
  int n = 0;
  const int n_sets = ceil_div(n_rows, 2);
  const double places = double(n_quads) * Ks, rows = n_rows > 1 ? 2.0 : 1.0;
  const double entries = places * (rows > 1.0 ? density * (2.0 - density) : density), hits = places * density * rows;
  const double warps = double(g.n) * g.To * g.Ho * g.Wo * n_sets / 16.0;
  for (int V = 1; V <= 8; V *= 2)
    for (int lg = 0; lg < 16; ++lg) {
      const int sets = 1 << (lg & 3), parts = 1 << (lg >> 2);
      if (sets >= 2 * n_sets || sets * parts > 8) continue;
      if (parts > 1 && (V == 8 || warps / V > 32.0 * sm_count)) continue;      // enough warps as it is
      F32Plan p{V, sets, parts, 1, 1, 1, 1, 1};
      if (choose_box_f32(g, 8 / (sets * parts) * 16, V, 0.1, &p) < 0) continue;
      const double boxes = double(g.n) * ceil_div(g.To, p.bt) * ceil_div(g.Ho, p.bh) * ceil_div(g.Wo, p.bw);
      const int halo = staged(p.bt, g.Kt, g.st) * staged(p.bh, g.Kh, g.sh) * staged(p.bw, g.Kw, g.sw);
      const double mean = double(quads) * Ks * density * 2 * sets;         // tiles of a stage
      const F32Smem sm = f32_smem(int(mean * 1.2) + 1, quads * Ks * sets, quads, halo, f32_sum_bytes(V, parts));
      if (sm.total > 227 * 1024) continue;
      const int occ = 226 * 1024 / (sm.total + 1024) > 1 ? 2 : 1;
      const double per_sm = double(ceil_div64(int64_t(boxes) * ceil_div(n_sets, sets), sm_count));
      const double h = hits / entries, staging = double(n_stages) * (halo * quads * 32.0 + mean * 4 * 12.0) / 128.0;
      const double own = parts > 1 ? entries / parts + 1.5 * n_stages : entries, sum = parts > 1 ? 800.0 + 220.0 * V * (parts - 1) : 0.0;
      const double busy = 2.0 * own * (25.0 + V * (4.0 + 10.0 * h)) + staging + sum;      // two warps a scheduler
      const double lone = own * (45.0 + V * (12.0 + 30.0 * h)) + staging + sum + n_stages * 900.0 + 2500.0;
      double t = per_sm * busy;
      if (std::ceil(per_sm / occ) * lone > t) t = std::ceil(per_sm / occ) * lone;
      int at = n;
      while (at > 0 && cost[at - 1] > t) { cost[at] = cost[at - 1]; plans[at] = plans[at - 1]; --at; }
      cost[at] = t; plans[at] = p;
      ++n;
    }
  *cycles = n > 0 ? cost[0] : 0.0;
  return n;
}

int conv_f32_plans(const ConvGeom& g, double density, int sm_count, F32Plan plans[kF32MaxPlans], double* cycles) {
  // The search takes 0.1 ms; a call in chunks asks for the same shape for every chunk.
  struct Entry { ConvGeom g; double density, cycles; int n; F32Plan plans[kF32MaxPlans]; };
  thread_local Entry cache[4];
  thread_local int next = 0;
  for (const Entry& e : cache)
    if (e.n > 0 && memcmp(&e.g, &g, sizeof(g)) == 0 && e.density == density) {
      std::copy(e.plans, e.plans + e.n, plans);
      *cycles = e.cycles;
      return e.n;
    }
  Entry& e = cache[next];
  next = (next + 1) % 4;
  e.g = g; e.density = density;
  e.n = search_plans(g, density, sm_count, e.plans, &e.cycles);
  *cycles = e.cycles;
  std::copy(e.plans, e.plans + e.n, plans);
  return e.n;
}

bool conv_f32_fill(const F32Plan& p, const F32Layout& L, F32Args* a) {
  const ConvGeom& g = a->g;
  a->bt = p.bt; a->bh = p.bh; a->bw = p.bw; a->vt = p.vt; a->vh = p.vh;
  a->tiles_t = ceil_div(g.To, p.bt); a->tiles_h = ceil_div(g.Ho, p.bh); a->tiles_w = ceil_div(g.Wo, p.bw);
  a->ht = staged(p.bt, g.Kt, g.st); a->hh = staged(p.bh, g.Kh, g.sh); a->hw = staged(p.bw, g.Kw, g.sw);
  a->ht_step = g.Kt == 1 ? g.st : 1; a->hh_step = g.Kh == 1 ? g.sh : 1; a->hw_step = g.Kw == 1 ? g.sw : 1;
  a->n_sets = L.n_sets; a->n_stages = L.n_stages; a->quads = L.quads;
  a->sets = p.sets; a->parts = p.parts;
  const int lg = p.sets == 1 ? 0 : p.sets == 2 ? 1 : p.sets == 4 ? 2 : 3;
  a->max_entries = L.max_entries[lg]; a->max_tiles = L.max_tiles[lg];
  return f32_smem(a->max_tiles, a->max_entries, a->quads, a->ht * a->hh * a->hw, f32_sum_bytes(p.voxels, p.parts)).total <= 227 * 1024 &&
         (long long)g.n * a->tiles_t * a->tiles_h * a->tiles_w < (1ll << 31) && ceil_div(L.n_sets, p.sets) <= 65535;
}

cudaError_t launch_conv_f32(const F32Args& a, const F32Plan& p, cudaStream_t stream) {
  const dim3 grid(unsigned(a.g.n * a.tiles_t * a.tiles_h * a.tiles_w), unsigned(ceil_div(a.n_sets, p.sets)));
  const size_t smem = size_t(f32_smem(a.max_tiles, a.max_entries, a.quads, a.ht * a.hh * a.hw, f32_sum_bytes(p.voxels, p.parts)).total);
  switch (p.voxels) {
    case 1: return p.parts > 1 ? launch_t<1, true>(a, grid, smem, stream) : launch_t<1, false>(a, grid, smem, stream);
    case 2: return p.parts > 1 ? launch_t<2, true>(a, grid, smem, stream) : launch_t<2, false>(a, grid, smem, stream);
    case 4: return p.parts > 1 ? launch_t<4, true>(a, grid, smem, stream) : launch_t<4, false>(a, grid, smem, stream);
    case 8: return launch_t<8, false>(a, grid, smem, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace rt3d
