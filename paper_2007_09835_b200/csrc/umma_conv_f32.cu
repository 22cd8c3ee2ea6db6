// fp32 KGS convolution on the tensor cores: every fp32 value as the sum of three bf16 ones.
//
// x = xh + xm + xl with xh = bf16(x), xm = bf16(x - xh), xl = bf16(x - xh - xm): three significands of 8 bits hold all 24, and
// a product of two such sums needs six of the nine bf16 products, each exact in fp32: xh wh, xh wm, xm wh, xm wm, xh wl and
// xl wh (the other three are below 2^-25 of the product).  Per K step, one kernel location and one chunk of 32 input channels
// that a kernel group keeps:  D[128 output voxels x n_tile output channels] += A[128 x 32] B[n_tile x 32]^T
// or, on CTA pairs (two tiles, each CTA with half of the weights), 256 voxels.
//
// Sums: the tensor core adds into its fp32 accumulator with less care than an fp32 add (the addends are aligned and cut off),
// so no long sum is left to it.  xh wh goes into one of two accumulators for `period` steps, then the other takes over while
// the drain warps add the finished one, rounded to nearest, to sums that they hold in registers.  The small products, 2^-8
// and less of the first, have accumulators of their own.
//
// Roles (640 threads): warp 0 loads, warp 1 issues the MMAs, warps 4..11 split the staged fp32 voxels and put them into tensor
// memory, which is where the MMAs read A from, warps 12..19 drain.  From shared memory the MMAs would read A three times beside
// the weights and the split would be written there as well, and shared memory moves 128 bytes a clock.
//
// Bound: at 128 columns the tensor pipe (64 -> 128 channels 3x3x3 on 2 x 16 x 56 x 56: 266 GFLOP of bf16 products in 168 us,
// 1.58 of the 1.64 PFLOP/s that cuBLAS reaches; the register-blocked FMAs of 0.4 of the places take 528), below that the hand-shakes
// and the arithmetic of a step, 0.31 us each.  Errors against 64 bits, relative, CUDA cores and here: 3.3e-7 and 1.2e-7 for
// that layer, 6.0e-8 and 4.3e-8 for 44 channels 1x1x1; at most 0.81 of the CUDA cores' in 300 random layers that the dispatch sends
// here, with weights of both signs.  Layers whose weights lean to one side do not come here (pack.cpp: splits_well).
//
// Range: x is split as 2^24 x, which leaves the parts of the smallest denormal (2^-149) normal bf16 numbers; the sums are
// scaled back, exactly, as they are stored.  Weights are split as they are; handles with magnitudes outside of [2^-100, 2^64)
// stay on the CUDA cores, so all parts are exact, and what a product of parts loses to underflow is below 2^-172.  What is too
// large is found in the result: an infinity or NaN in x, or |x| from 2^103 on, makes the parts infinite or NaN and with them the
// voxel's whole row (NaN times a pruned weight's zero is NaN too), and so do sums from 2^103 on.  Rows with such results are
// computed again with fp32 FMAs from the packed arrays, skipping what is pruned, by the threads that drain them.
#include <algorithm>

#include "f32_split_plan.h"
#include "kernels.h"
#include "pdl.cuh"
#include "rt3d_internal.h"
#include "umma_pair.cuh"

namespace rt3d {
namespace {

constexpr int kThreadsSplit = 640;
constexpr int kDrainThreads = 256;
constexpr uint32_t kSlotCols = kSplitSlotCols;
constexpr long long kAgainClocks = 2048;                // allowed to a drain warp for each of the products in F32SplitArgs::again
constexpr int kSplitSegment = 64;                       // steps after which a shared accumulator of small products is drained
constexpr uint32_t kDrainStage = kSplitDrainStage;

struct __align__(8) SplitBars {
  Barriers b;                                           // full: weights; empty: MMAs done; tmem_*: the two xh wh accumulators
  unsigned long long x_full[kSplitInputs], x_empty[kSplitInputs];
  // of a pair, the leader's:
  unsigned long long a_full[kSplitSlots];               // A operands (of a pair: and the weights) of both CTAs
  unsigned long long small_empty;                       // the small products' accumulator, where it is shared
};
static_assert(sizeof(SplitBars) == kSplitBarBytes && kABytes == kSplitInputBytes, "f32_split_plan.h");

struct SplitItem { int bundle, n0, t0, h0, w0; };
// `ctas`: tiles of an item, `rank`: which of them.
__device__ __forceinline__ SplitItem decode_split_item(const F32SplitArgs& a, int item, int ctas, int rank) {
  const int n_mtiles = a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w, per_bundle = (n_mtiles + ctas - 1) / ctas;
  SplitItem c;
  c.bundle = item / per_bundle;
  int mt = (item - c.bundle * per_bundle) * ctas + rank;
  if (mt >= n_mtiles) {                                 // odd tile count: the last pair's second tile does not exist
    c.n0 = a.g.n; c.t0 = 0; c.h0 = 0; c.w0 = 0;
    return c;
  }
  const int iw = mt % a.tiles_w; mt /= a.tiles_w;
  const int ih = mt % a.tiles_h; mt /= a.tiles_h;
  const int it = mt % a.tiles_t; mt /= a.tiles_t;
  c.w0 = iw * a.box.bw; c.h0 = ih * a.box.bh; c.t0 = it * a.box.bt; c.n0 = mt * a.box.bn;
  return c;
}

// D[tmem] (+)= A[tmem] * B[smem] where `go` holds.
template <bool kPair>
__device__ __forceinline__ void mma_ta(bool go, uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, int acc) {
  if constexpr (kPair)
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc), "r"(int(go))
        : "memory");
  else
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc), "r"(int(go))
        : "memory");
}
template <bool kPair>
__device__ __forceinline__ void commit_to(uint32_t bar) {
  if constexpr (kPair) umma_commit_pair(bar);
  else umma_commit(bar);
}
// Arrival on a barrier of the CTA, of a pair: of its leader.
template <bool kPair>
__device__ __forceinline__ void arrive_at(uint32_t bar) {
  if constexpr (kPair) mbar_arrive_cluster(mapa_shared(bar, 0));
  else mbar_arrive(bar);
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_st16_words(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
constexpr float kUp = 16777216.f, kDown = 1.f / 16777216.f;             // 2^24: see the head of the file
struct Float2 { unsigned long long bits; };              // two floats for the instructions that work on both
__device__ __forceinline__ Float2 float2_of(float a, float b) {
  Float2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d.bits) : "f"(a), "f"(b));
  return d;
}
// Two values rounded to bf16, and what is left of them (exact).
__device__ __forceinline__ uint32_t take_bf16x2(Float2& x) {
  float x0, x1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x0), "=f"(x1) : "l"(x.bits));
  const uint32_t h = pack_bf16x2(x0, x1);
  const Float2 taken = float2_of(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u)), minus = float2_of(-1.f, -1.f);
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(x.bits) : "l"(taken.bits), "l"(minus.bits), "l"(x.bits));
  return h;
}
// The three parts of two neighbouring channels.  Instructions on pairs: the splitting warps' arithmetic is what up to 48 columns
// wait for (64 -> 32 channels 3x3x3 on 2 x 16 x 56 x 56 111.7 us, one value at a time 114.2).
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& h, uint32_t& m, uint32_t& l) {
  Float2 x = float2_of(x0, x1);
  const Float2 up = float2_of(kUp, kUp);
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(x.bits) : "l"(x.bits), "l"(up.bits));
  h = take_bf16x2(x);
  m = take_bf16x2(x);
  l = take_bf16x2(x);
}

// J consecutive values: one; four at a multiple of 16 bytes; or (kRagged) four of which `left`, at least one, exist, and zeros.
constexpr int kOne = 1, kFour = 4, kRagged = 0;
template <int J>
__device__ __forceinline__ float4 load_some(const float* p, int left) {
  if (J == kFour) return __ldg(reinterpret_cast<const float4*>(p));
  if (J == kOne) return make_float4(__ldg(p), 0.f, 0.f, 0.f);
  const float v[4] = {__ldg(p), __ldg(p + min(1, left - 1)), __ldg(p + min(2, left - 1)), __ldg(p + min(3, left - 1))};
  return make_float4(v[0], left > 1 ? v[1] : 0.f, left > 2 ? v[2] : 0.f, left > 3 ? v[3] : 0.f);
}
// Adds two packed entries' products over J input channels to the sums of C output channels (of which n exist).  x: where an entry
// meets the input, nullptr: nowhere.  No branches, so that the loads are on their way together: entries that meet nothing add
// zeros, channels that do not exist repeat the last one.
template <int C, int J>
__device__ __forceinline__ void add_entries(float (&s)[4], const float* const (&x)[2], const float* somewhere, const float* const (&w)[2], int g_n, int n, int left) {
  float4 v[2], t[2][C];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    v[u] = load_some<J>(x[u] != nullptr ? x[u] : somewhere, left);
#pragma unroll
    for (int c = 0; c < C; ++c) t[u][c] = load_some<J>(w[u] + min(c, n - 1) * g_n, left);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const bool there = x[u] != nullptr;
    const float4 f = make_float4(there ? v[u].x : 0.f, there ? v[u].y : 0.f, there ? v[u].z : 0.f, there ? v[u].w : 0.f);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      s[c] = fmaf(t[u][c].x, f.x, s[c]);
      if (J != kOne) s[c] = fmaf(t[u][c].w, f.w, fmaf(t[u][c].z, f.z, fmaf(t[u][c].y, f.y, s[c])));
    }
  }
}
// n <= C output channels of one voxel from channel m on, all in one kernel group, in fp32 from the packed arrays.
template <int C>
__device__ __forceinline__ void exact_outputs(float (&s)[4], const F32SplitArgs& a, int m, int n, int nn, int ti0, int hi0, int wi0) {
  const ConvGeom& g = a.g;
  const int p = m / a.g_m, i = m - p * a.g_m;
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c] = 0.f;
  int e = __ldg(a.group_ptr + p * a.Q);
  for (int q = 0; q < a.Q; ++q) {
    const int e1 = __ldg(a.group_ptr + p * a.Q + q + 1), real = min(a.g_n, g.c - q * a.g_n);         // padding channels hold anything
    for (; e < e1; e += 2) {
      const float *x[2], *w[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int at = min(e + u, e1 - 1), k = __ldg(a.pos_idx + at), row = k / g.Kw, kt = row / g.Kh;
        const int ti = ti0 + kt, hi = hi0 + row - kt * g.Kh, wi = wi0 + k - row * g.Kw;
        const bool there = e + u < e1 && unsigned(ti) < unsigned(g.t) && unsigned(hi) < unsigned(g.h) && unsigned(wi) < unsigned(g.w);
        x[u] = there ? a.x + ((((long long)nn * g.t + ti) * g.h + hi) * g.w + wi) * g.xcs + q * a.g_n : nullptr;
        w[u] = a.tiles + ((long long)at * a.g_m + i) * a.g_n;
      }
      for (int j = 0; j < real; j += 4) {
        if (real - j == 1) add_entries<C, kOne>(s, x, a.x, w, a.g_n, n, 1);
        else if (a.g_n % 4 == 0 && real - j >= 4) add_entries<C, kFour>(s, x, a.x, w, a.g_n, n, 4);
        else add_entries<C, kRagged>(s, x, a.x, w, a.g_n, n, real - j);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (x[u] != nullptr) x[u] += 4;
          w[u] += 4;
        }
      }
    }
    e = e1;
  }
}
// The output channels [m0, m0 + n) of the voxels (one a lane) that `odd` names, shared out over the warp in fours: a single odd
// voxel takes as long as one of its channel quads, a warp of them as long as all of its quads after one another.  Bound by the
// latency of the loads: 700 to 1000 clocks for each entry and quad.  64 -> 128 channels 3x3x3 on 2 x 16 x 56 x 56, 0.4 kept: 0.57 ms
// with one NaN in the input, 10.5 ms with nothing else (a voxel's channels one after the other on one lane: 8.5 and 70 ms; the CUDA
// cores take 0.57 for any input).  Four entries at a time were no faster, and their registers cost finite inputs 1 %.  The other roles wait meanwhile: their limit grows by F32SplitArgs::again.
__device__ __noinline__ void exact_rows(const F32SplitArgs& a, const float* bias_s, int m0, int n, uint32_t odd, int lane, int vox) {
  const ConvGeom& g = a.g;
  const int n_odd = __popc(odd), items = n_odd * ((n + 3) / 4);
  for (int first = 0; first < items; first += 32) {
    const int item = min(first + lane, items - 1), quad = item / n_odd, from = __fns(odd, 0, item - quad * n_odd + 1);
    const int at = __shfl_sync(0xffffffffu, vox, from), line = at / g.Wo, frame = line / g.Ho, nn = frame / g.To;
    const int wi = (at - line * g.Wo) * g.sw - g.pw, hi = (line - frame * g.Ho) * g.sh - g.ph, ti = (frame - nn * g.To) * g.st - g.pt;
    const int m1 = m0 + min(n, 4 * quad + 4);
    for (int m = m0 + 4 * quad; m < m1 && first + lane < items;) {
      const int here = min(m1, (m / a.g_m + 1) * a.g_m) - m;             // that lie in one group
      float r[4];
      if (here == 1) exact_outputs<1>(r, a, m, here, nn, ti, hi, wi);
      else exact_outputs<4>(r, a, m, here, nn, ti, hi, wi);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (c >= here) break;
        float s = r[c] + bias_s[m + c];
        if (a.residual) s += a.residual[(long long)at * a.rcs + m + c];
        a.y[(long long)at * g.ycs + m + c] = g.relu ? fmaxf(s, 0.f) : s;
      }
      m += here;
    }
    __syncwarp();
  }
}

// NH: columns that one thread of the drain warps holds (the first set of warps takes columns [0, NH), the second the rest).
// kSub: steps per hand-shake of the pipeline.  kMode: a narrow MMA takes 46 clocks whatever its width, so the products of one
// part of x with neighbouring parts of w are one MMA where tensor memory has room for their accumulators:
//   kAll: a buffer holds [xh wh | order 2^-8 | order 2^-16], three MMAs a K = 16 slice, all of it drained at once
//   kSmall: two buffers for xh wh, one [order 2^-8 | order 2^-16], four MMAs
//   kNone: two buffers for xh wh, one for all small products, six MMAs
// kPair: CTA pairs.
constexpr int kNone = kSplitNone, kSmall = kSplitSmall, kAll = kSplitAll;
template <int NH, int kSub, int kMode, bool kPair>
__global__ void __launch_bounds__(kThreadsSplit, 1)
conv3d_umma_f32_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ F32SplitArgs a) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  constexpr int kCtas = kPair ? 2 : 1;
  const uint32_t w_rows = uint32_t(a.n_tile) / kCtas, w_step = w_rows * 192u, w_stage = kSub * w_step;       // this CTA's weights
  const uint32_t w_smem = base + uint32_t(a.inputs) * (kSub * kABytes);
  const uint32_t turn = w_smem + uint32_t(a.stages) * w_stage;           // the drain warps' 2 KB each
  SplitBars* sb = reinterpret_cast<SplitBars*>(smem_raw + (turn - raw) + 8 * kDrainStage);
  Barriers* bars = &sb->b;
  float* bias_s = align16_f32(sb + 1);
  int32_t* err = a.sched + 2;

  const int warp = uniform(int(threadIdx.x >> 5)), lane = threadIdx.x & 31;
  const int rank = kPair ? int(blockIdx.x & 1u) : 0;
  const int first_item = int(blockIdx.x) / kCtas, item_step = int(gridDim.x) / kCtas;
  const int n_items = (a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w + kCtas - 1) / kCtas * a.n_bundles;
  const int box_rows = a.box.bn * a.box.bt * a.box.bh * a.box.bw;
  const int slots = a.slots;

  if (threadIdx.x == 32) tma_prefetch_map(&xmap);
  if (threadIdx.x == 0) {
    for (int s = 0; s < a.stages; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int s = 0; s < a.inputs; ++s) {
      mbar_init(smem_u32(&sb->x_full[s]), 1);
      mbar_init(smem_u32(&sb->x_empty[s]), 4);                                       // the splitting warps of a team
    }
    for (int s = 0; s < slots; ++s) mbar_init(smem_u32(&sb->a_full[s]), 4 * kCtas);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bars->tmem_full[b]), 1);
      mbar_init(smem_u32(&bars->tmem_empty[b]), 8 * kCtas);                          // drain warps
    }
    mbar_init(smem_u32(&sb->small_empty), 8 * kCtas);
    bars->abort_flag = 0;
    bars->wait_limit = kWaitCycles + a.again * kAgainClocks;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = 0;                          // all 512 columns are this CTA's
  const uint32_t buf_cols = (kMode == kAll ? 3u : 1u) * uint32_t(a.n_tile);
  const uint32_t small_tmem = tmem_base + 2u * uint32_t(a.n_tile);                   // not kAll
  const uint32_t a_tmem = tmem_base + 512u - uint32_t(slots) * (kSub * kSlotCols);

  pdl_launch();
  pdl_wait();
  if (warp >= 12) {
    for (int i = threadIdx.x - 384; i < a.n_bundles * a.n_tile; i += kDrainThreads)
      bias_s[i] = (a.bias != nullptr && i < a.g.M) ? __ldg(a.bias + i) : 0.f;
    epilogue_bar_sync(kDrainThreads);
  }

  if (warp == 0) {
    // ------------------------------------------------------------------ loads
    if (lane == 0) {
      int stage = 0, xb = 0;
      uint32_t phase = 0, x_phase = 0;
      bool ok = true;
      for (int item = first_item; item < n_items && ok; item += item_step) {
        const SplitItem c = decode_split_item(a, item, kCtas, rank);
        const int s0 = __ldg(a.step_ptr + c.bundle), s1 = __ldg(a.step_ptr + c.bundle + 1);
        const int wq = c.w0 * a.g.sw - a.g.pw, hq = c.h0 * a.g.sh - a.g.ph, tq = c.t0 * a.g.st - a.g.pt;
        int enc[kSub];
#pragma unroll
        for (int q = 0; q < kSub; ++q) enc[q] = s0 + q < s1 ? __ldg(a.steps + s0 + q) : 0;
        for (int s = s0; s < s1; s += kSub) {
          const int n_sub = min(kSub, s1 - s);
          int now[kSub];
#pragma unroll
          for (int q = 0; q < kSub; ++q) {
            now[q] = enc[q];
            if (s + kSub + q < s1) enc[q] = __ldg(a.steps + s + kSub + q);
          }
          const uint32_t x_full = smem_u32(&sb->x_full[xb]), x_dst = base + uint32_t(xb) * (kSub * kABytes);
          if (!mbar_wait(smem_u32(&sb->x_empty[xb]), x_phase ^ 1u, bars, err, 72)) { ok = false; break; }
          mbar_expect_tx(x_full, uint32_t(box_rows) * 128u * uint32_t(n_sub));
#pragma unroll
          for (int q = 0; q < kSub; ++q)
            if (q < n_sub)
              tma_load_5d(x_dst + q * kABytes, &xmap, x_full, (now[q] & 4095) * 32, wq + ((now[q] >> 12) & 63), hq + ((now[q] >> 18) & 63),
                          tq + ((now[q] >> 24) & 63), c.n0);
          if (++xb == a.inputs) { xb = 0; x_phase ^= 1u; }
          const uint32_t full = smem_u32(&bars->full[stage]);
          if (!mbar_wait(smem_u32(&bars->empty[stage]), phase ^ 1u, bars, err, 71)) { ok = false; break; }
          mbar_expect_tx(full, w_step * uint32_t(n_sub));
          for (int q = 0; q < n_sub; ++q)
            bulk_load(w_smem + uint32_t(stage) * w_stage + uint32_t(q) * w_step, a.wtiles + (size_t(s + q) * kCtas + rank) * w_step, w_step, full);
          if (++stage == a.stages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (of a pair: the leader)
    // The whole warp walks the loop, one lane's MMAs take effect.  No branch and no address arithmetic on vector registers
    // between the MMAs: with both, an MMA left every 82 clocks.
    const bool elected = elect_one();
    const uint32_t n = uint32_t(a.n_tile);
    const uint32_t idesc1 = kPair ? instr_desc_bf16_pair(a.n_tile) : instr_desc_bf16(a.n_tile);
    const uint32_t idesc2 = instr_desc_bf16(2 * a.n_tile), idesc3 = instr_desc_bf16(3 * a.n_tile);      // single CTAs only
    // low descriptor word of the first stage's weights: [16 channels][8 channels][part][row][8]; core matrices 48 bytes a row
    // apart along K, 128 bytes along the rows
    const uint32_t w_lo0 = (w_smem >> 4) | ((3u * w_rows) << 16);
    const uint64_t w_hi = uint64_t((128u >> 4) | (1u << 14)) << 32;
    int stage = 0, slot = 0;
    uint32_t phase = 0, slot_phase = 0, n_periods = 0, n_segments = 0;
    bool ok = true, ready = false;
    for (int item = rank == 0 ? first_item : n_items; item < n_items && ok; item += item_step) {
      const int bundle = decode_split_item(a, item, kCtas, 0).bundle;
      const int s0 = uniform(__ldg(a.step_ptr + bundle)), s1 = uniform(__ldg(a.step_ptr + bundle + 1));
      int in_period = 0, in_segment = 0;
      int enc[kSub];                                       // read where the last chunk is half a chunk
#pragma unroll
      for (int q = 0; q < kSub; ++q) enc[q] = (a.last_k16 != 2 && s0 + q < s1) ? __ldg(a.steps + s0 + q) : -1;
      for (int s = s0; s < s1; s += kSub) {
        bool both[kSub];
#pragma unroll
        for (int q = 0; q < kSub; ++q) {
          both[q] = a.last_k16 == 2 || uniform(enc[q] & 4095) != a.last_chunk;
          if (a.last_k16 != 2 && s + kSub + q < s1) enc[q] = __ldg(a.steps + s + kSub + q);
        }
        const uint32_t buf = n_periods & 1u;
        if (kMode != kAll && in_segment == 0 && !mbar_wait_warp(smem_u32(&sb->small_empty), (n_segments & 1u) ^ 1u, bars, err, 73)) { ok = false; break; }
        if (in_period == 0 && !mbar_wait_warp(smem_u32(&bars->tmem_empty[buf]), ((n_periods >> 1) & 1u) ^ 1u, bars, err, 74)) { ok = false; break; }
        if (!kPair && !mbar_wait_warp(smem_u32(&bars->full[stage]), phase, bars, err, 75)) { ok = false; break; }
        if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(smem_u32(&sb->a_full[slot]), slot_phase, bars, err, 76)) { ok = false; break; }
        const int slot_n = slot + 1 == slots ? 0 : slot + 1;
        const uint32_t slot_phase_n = slot + 1 == slots ? slot_phase ^ 1u : slot_phase;
        ready = mbar_try_wait(smem_u32(&sb->a_full[slot_n]), slot_phase_n);       // its answer arrives while these MMAs leave
        tc_fence_after();
        const uint32_t big = tmem_base + buf * buf_cols;
#pragma unroll
        for (int q = 0; q < kSub; ++q) {
          if (s + q >= s1) break;
          const uint32_t ah = a_tmem + uint32_t(slot * kSub + q) * kSlotCols;
          const uint32_t w_lo = w_lo0 + (uint32_t(stage) * w_stage + uint32_t(q) * w_step) / 16u;
#pragma unroll
          for (uint32_t kk = 0; kk < 2; ++kk) {
            if (kk == 1 && !both[q]) break;
            const uint64_t bh = w_hi | (w_lo + 6u * kk * w_rows), bm = w_hi | (w_lo + (6u * kk + 1u) * w_rows),
                           bl = w_hi | (w_lo + (6u * kk + 2u) * w_rows);
            const uint32_t xh = ah + 8u * kk;
            if constexpr (kMode == kAll) {
              mma_ta<kPair>(elected, big, xh, bh, idesc3, in_period | q | int(kk));
              mma_ta<kPair>(elected, big + n, xh + 16, bh, idesc2, 1);
              mma_ta<kPair>(elected, big + 2 * n, xh + 32, bh, idesc1, 1);
            } else if constexpr (kMode == kSmall) {
              mma_ta<kPair>(elected, big, xh, bh, idesc1, in_period | q | int(kk));
              mma_ta<kPair>(elected, small_tmem, xh, bm, idesc2, in_segment | q | int(kk));
              mma_ta<kPair>(elected, small_tmem, xh + 16, bh, idesc2, 1);
              mma_ta<kPair>(elected, small_tmem + n, xh + 32, bh, idesc1, 1);
            } else {
              mma_ta<kPair>(elected, big, xh, bh, idesc1, in_period | q | int(kk));
              mma_ta<kPair>(elected, small_tmem, xh, bm, idesc1, in_segment | q | int(kk));
              mma_ta<kPair>(elected, small_tmem, xh + 16, bh, idesc1, 1);
              mma_ta<kPair>(elected, small_tmem, xh + 16, bm, idesc1, 1);
              mma_ta<kPair>(elected, small_tmem, xh, bl, idesc1, 1);
              mma_ta<kPair>(elected, small_tmem, xh + 32, bh, idesc1, 1);
            }
          }
        }
        if (elected) commit_to<kPair>(smem_u32(&bars->empty[stage]));
        in_segment += kSub;
        in_period += kSub;
        const bool last = s + kSub >= s1 || in_segment == kSplitSegment;
        if (in_period == a.period || last) {
          if (elected) commit_to<kPair>(smem_u32(&bars->tmem_full[buf]));
          in_period = 0;
          ++n_periods;
        }
        if (last) { in_segment = 0; ++n_segments; }
        if (++stage == a.stages) { stage = 0; phase ^= 1u; }
        slot = slot_n; slot_phase = slot_phase_n;
      }
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 12) {
    // ------------------------------------------------------------------ fp32 voxels -> three bf16 parts in tensor memory
    // Two teams of four warps, a warp to a lane quadrant, take turns: what a hand-shake costs a team is the latency of its
    // waits, loads, arithmetic and stores, one after the other (eight warps on each: 620 clocks for two steps).
    const int team = (warp - 4) >> 2;
    const uint32_t row = uint32_t((warp & 3) * 32 + lane), sw = row & 7u;
    const uint32_t lanes = uint32_t((warp & 3) * 32) << 16;
    int slot = 0, xb = 0, stage = 0, stage_b = 0;          // stage_b: of the steps whose MMAs free this slot
    uint32_t x_phase = 0, phase = 0, phase_b = 0;
    int count = 0;
    bool ok = true;
    for (int item = first_item; item < n_items && ok; item += item_step) {
      const int bundle = decode_split_item(a, item, kCtas, 0).bundle;
      const int n_steps = __ldg(a.step_ptr + bundle + 1) - __ldg(a.step_ptr + bundle);
      for (int s = 0; s < n_steps; s += kSub, ++count) {
        if ((count & 1) == team) {
          if (!mbar_wait_warp(smem_u32(&sb->x_full[xb]), x_phase, bars, err, 77)) { ok = false; break; }
          const uint32_t src = base + uint32_t(xb) * (kSub * kABytes) + row * 128u;
#pragma unroll
          for (int u = 0; u < kSub; ++u) {
            if (s + u >= n_steps) break;
            float v[32];
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k)
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[4 * k]), "=f"(v[4 * k + 1]), "=f"(v[4 * k + 2]), "=f"(v[4 * k + 3])
                           : "r"(src + u * kABytes + ((k ^ sw) << 4)));
            uint32_t h[16], m[16], l[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) split2(v[2 * q], v[2 * q + 1], h[q], m[q], l[q]);
            if (u == 0) {
              if (count >= slots && !mbar_wait_warp(smem_u32(&bars->empty[stage_b]), phase_b, bars, err, 78)) { ok = false; break; }
              tc_fence_after();
            }
            const uint32_t dst = a_tmem + lanes + uint32_t(slot * kSub + u) * kSlotCols;
            tmem_st16_words(dst, h);
            tmem_st16_words(dst + 16, m);
            tmem_st16_words(dst + 32, l);
          }
          if (!ok) break;
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&sb->x_empty[xb]));
          // of a pair, the arrival stands for this CTA's weights too
          if (kPair && !mbar_wait_warp(smem_u32(&bars->full[stage]), phase, bars, err, 75)) { ok = false; break; }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_at<kPair>(smem_u32(&sb->a_full[slot]));
        }
        if (count >= slots && ++stage_b == a.stages) { stage_b = 0; phase_b ^= 1u; }
        if (++xb == a.inputs) { xb = 0; x_phase ^= 1u; }
        if (++stage == a.stages) { stage = 0; phase ^= 1u; }
        if (++slot == slots) slot = 0;
      }
    }
  } else if (warp >= 12) {
    // ------------------------------------------------------------------ accumulators -> sums -> y
    const int quad = warp & 3, set = (warp - 12) >> 2;
    const int col0 = set * NH, n_cols = min(NH, a.n_tile - col0);      // a multiple of 16; 0 or less: only the hand-shakes
    const int row = quad * 32 + lane;
    int r = row;
    const int bw_i = r % a.box.bw; r /= a.box.bw;
    const int bh_i = r % a.box.bh; r /= a.box.bh;
    const int bt_i = r % a.box.bt; r /= a.box.bt;
    const int bn_i = r;
    const uint32_t lane_tmem = tmem_base + (uint32_t(quad * 32) << 16) + uint32_t(col0);
    const uint32_t small_lane = lane_tmem + 2u * uint32_t(a.n_tile);
    const uint32_t mine = turn + uint32_t(warp - 12) * kDrainStage;
    uint32_t n_periods = 0;
    bool ok = true;
    for (int item = first_item; item < n_items && ok; item += item_step) {
      const SplitItem c = decode_split_item(a, item, kCtas, rank);
      const int n_steps = __ldg(a.step_ptr + c.bundle + 1) - __ldg(a.step_ptr + c.bundle);
      const int nn = c.n0 + bn_i, to = c.t0 + bt_i, ho = c.h0 + bh_i, wo = c.w0 + bw_i;
      const bool in_range = row < box_rows && nn < a.g.n && to < a.g.To && ho < a.g.Ho && wo < a.g.Wo;
      const int vox = in_range ? ((nn * a.g.To + to) * a.g.Ho + ho) * a.g.Wo + wo : -1;
      const int m0 = c.bundle * a.n_tile + col0, n_here = min(n_cols, a.g.M - m0);
      if (a.residual != nullptr && in_range)               // on its way from memory while the accumulators are waited for
        for (int b = 0; b < n_here * 4; b += 128)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(a.residual + (long long)vox * a.rcs + m0) + b));
      float sum[NH];
#pragma unroll
      for (int q = 0; q < NH; ++q) sum[q] = 0.f;
      const auto add = [&](uint32_t taddr) {
#pragma unroll
        for (int k = 0; k < NH / 16; ++k)
          if (k * 16 < n_cols) {
            uint32_t v[16];
            tmem_ld16(taddr + k * 16, v);
#pragma unroll
            for (int q = 0; q < 16; ++q) sum[k * 16 + q] += __uint_as_float(v[q]);
          }
      };
      int left = n_steps;
      while (left > 0) {
        int seg = left < kSplitSegment ? left : kSplitSegment;
        left -= seg;
        while (seg > 0) {
          const uint32_t buf = n_periods & 1u, big = lane_tmem + buf * buf_cols;
          if (!mbar_wait_warp(smem_u32(&bars->tmem_full[buf]), (n_periods >> 1) & 1u, bars, err, 79)) { ok = false; break; }
          tc_fence_after();
          seg -= a.period;
          if (kMode == kAll) {
            add(big + 2u * uint32_t(a.n_tile));
            add(big + uint32_t(a.n_tile));
          } else if (seg <= 0) {                           // the segment's last: the small products are complete too
            if (kMode == kSmall) add(small_lane + uint32_t(a.n_tile));
            add(small_lane);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_at<kPair>(smem_u32(&sb->small_empty));
          }
          add(big);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_at<kPair>(smem_u32(&bars->tmem_empty[buf]));
          ++n_periods;
        }
        if (!ok) break;
      }
      if (!ok) break;
      int at[4];                                           // the voxels whose channels this lane stores
#pragma unroll
      for (int it = 0; it < 4; ++it) at[it] = __shfl_sync(0xffffffffu, vox, it * 8 + (lane >> 2));
      uint32_t high[4] = {0u, 0u, 0u, 0u};                 // largest magnitude, in four chains
#pragma unroll
      for (int k = 0; k < NH / 16; ++k) {
        if (16 * k >= n_here) break;
        // 16 channels of the warp's 32 voxels turn in shared memory, so that four lanes store the 64 bytes of a voxel (each
        // lane its own voxel's: 32 lines to an instruction, and the MMAs waited 15 % of their time for accumulators)
        __syncwarp();
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
          const float* v = sum + 16 * k + 4 * q;
#pragma unroll
          for (int e = 0; e < 4; ++e) high[e] = max(high[e], __float_as_uint(v[e]) & 0x7fffffffu);
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                       ::"r"(mine + uint32_t(lane) * 64u + ((q ^ ((uint32_t(lane) >> 1) & 3u)) << 4)), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
        }
        __syncwarp();
        const int m = m0 + 16 * k + (lane & 3) * 4, valid = a.g.M - m;
        const float4 b = *reinterpret_cast<const float4*>(bias_s + m);
        float o[4][4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
          const uint32_t r8 = uint32_t(it) * 8u + (uint32_t(lane) >> 2);
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o[it][0]), "=f"(o[it][1]), "=f"(o[it][2]), "=f"(o[it][3])
                       : "r"(mine + r8 * 64u + (((uint32_t(lane) & 3u) ^ ((r8 >> 1) & 3u)) << 4)));
          o[it][0] = fmaf(o[it][0], kDown, b.x); o[it][1] = fmaf(o[it][1], kDown, b.y);
          o[it][2] = fmaf(o[it][2], kDown, b.z); o[it][3] = fmaf(o[it][3], kDown, b.w);
        }
        if (a.residual != nullptr) {
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            const float* rp = a.residual + (long long)at[it] * a.rcs + m;
            if (at[it] >= 0 && valid >= 4) {
              const float4 t = *reinterpret_cast<const float4*>(rp);
              o[it][0] += t.x; o[it][1] += t.y; o[it][2] += t.z; o[it][3] += t.w;
            } else if (at[it] >= 0) {
#pragma unroll
              for (int q = 0; q < 3; ++q)
                if (q < valid) o[it][q] += rp[q];
            }
          }
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
          if (a.g.relu)
#pragma unroll
            for (int q = 0; q < 4; ++q) o[it][q] = fmaxf(o[it][q], 0.f);
          float* yp = a.y + (long long)at[it] * a.g.ycs + m;
          if (at[it] >= 0 && valid >= 4) {
            *reinterpret_cast<float4*>(yp) = make_float4(o[it][0], o[it][1], o[it][2], o[it][3]);
          } else if (at[it] >= 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q)
              if (q < valid) yp[q] = o[it][q];
          }
        }
      }
      __syncwarp();
      // infinite, NaN or close to it: see the head of the file
      const uint32_t odd = __ballot_sync(0xffffffffu, in_range && max(max(high[0], high[1]), max(high[2], high[3])) >= 0x7f000000u);
      if (odd) exact_rows(a, bias_s, m0, n_here, odd, lane, vox);
    }
  }

  // ---------------------------------------------------------------------- teardown
  if (bars->abort_flag) {
    // error path: copies and MMAs still in flight get time to land before shared and tensor memory go away
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) { }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

template <int NH, int kSub, int kMode, bool kPair>
cudaError_t launch_split_t(const F32SplitArgs& a, const CUtensorMap& xm, int grid, size_t smem, cudaStream_t stream) {
  static bool attr_done[kMaxDevices] = {};             // the attribute is per device
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(conv3d_umma_f32_kernel<NH, kSub, kMode, kPair>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  LaunchSetup ls(dim3(unsigned(grid)), dim3(kThreadsSplit), smem, stream, kPair ? 2 : 1);
  return cudaLaunchKernelEx(&ls.cfg, conv3d_umma_f32_kernel<NH, kSub, kMode, kPair>, xm, a);
}

}  // namespace

bool umma_f32_plan(F32SplitArgs* a) {
  SplitRing r;
  if (!split_ring(a->n_tile, a->n_bundles, &r)) return false;
  a->pair = split_variant(a->n_tile).pair ? 1 : 0;
  a->inputs = r.inputs; a->stages = r.stages; a->slots = r.slots;
  return true;
}

cudaError_t launch_conv_umma_f32(const F32SplitArgs& a, const void* xmap, int sm_count, cudaStream_t stream) {
  const SplitVariant v = split_variant(a.n_tile);
  const SplitRing ring = {a.inputs, a.stages, a.slots};
  const size_t smem = split_smem_bytes(a.n_tile, a.n_bundles, ring);
  if (smem > kSplitSmem || a.inputs < 2 || a.inputs > kSplitInputs || a.stages > kMaxStages || !split_inputs_ordered(ring)) return cudaErrorInvalidValue;
  if (a.stages <= a.slots || a.slots < 2 || a.slots > kSplitSlots || a.period < 2 || a.period % 2 || kSplitSegment % a.period) return cudaErrorInvalidValue;
  const int ctas = v.pair ? 2 : 1;
  const long long items = ((long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w + ctas - 1) / ctas * a.n_bundles;
  if (items <= 0) return cudaSuccess;
  if (items > (1ll << 29) || (long long)a.g.n * a.g.To * a.g.Ho * a.g.Wo > 0x7fffffffll) return cudaErrorInvalidValue;
  const int most = sm_count / ctas, grid = ctas * int(items < most ? items : most);
  CUtensorMap xm;
  memcpy(&xm, xmap, sizeof(CUtensorMap));
  if (v.nh == 16) return launch_split_t<16, 2, kAll, false>(a, xm, grid, smem, stream);
  if (v.nh == 32 && v.mode == kAll) return launch_split_t<32, 2, kAll, false>(a, xm, grid, smem, stream);
  if (v.nh == 32) return launch_split_t<32, 2, kSmall, false>(a, xm, grid, smem, stream);
  if (v.nh == 48) return launch_split_t<48, 2, kNone, true>(a, xm, grid, smem, stream);
  return launch_split_t<64, 1, kNone, true>(a, xm, grid, smem, stream);
}

}  // namespace rt3d
