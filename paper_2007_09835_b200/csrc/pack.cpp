// Host-side weight reorganisation: the KGS pack (Section 3 / Section 5.2 of the paper), its
// inverse, and the derivation of the tensor-core weight layout from the canonical arrays.
// Pure host code: no CUDA calls, usable without a GPU.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <exception>
#include <memory>
#include <new>
#include <system_error>
#include <thread>
#include <utility>

#include "kept_blocks.h"
#include "rt3d_internal.h"

namespace rt3d {

float bf16_bits_to_f32(uint16_t b) {
  uint32_t u = uint32_t(b) << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

int default_n_tile(int M) {
  const int bundles = ceil_div(round_up(M, 16), 256);
  return round_up(ceil_div(M, bundles), 16);
}

bool umma_layout_possible(const rt3d_packed* p) {
  return p->dtype == RT3D_BF16 && p->Kt <= 63 && p->Kh <= 63 && p->Kw <= 63 && ceil_div(p->N, kChunk) <= 4095;
}

// Never destroyed: handles may be freed while the process exits.
static KeptBlocks& host_blocks() {
  static KeptBlocks* kept = new KeptBlocks([](void* p) { delete[] static_cast<unsigned char*>(p); });
  return *kept;
}
unsigned char* host_block(size_t bytes) {
  if (void* p = host_blocks().take(bytes, -1)) return static_cast<unsigned char*>(p);
  unsigned char* p = new (std::nothrow) unsigned char[bytes];
  if (!p) {
    host_blocks().release_all();
    p = new unsigned char[bytes];
  }
  host_blocks().note(p, bytes, -1);
  return p;
}
void host_block_free(unsigned char* p) { host_blocks().give(p); }
void host_blocks_release() { host_blocks().release_all(); }

static float tile_value(const rt3d_packed* p, int64_t e, int i, int j) {
  const int64_t o = (e * p->g_m + i) * p->g_n + j;
  if (p->dtype == RT3D_BF16) return bf16_bits_to_f32(reinterpret_cast<const uint16_t*>(p->tiles.data())[o]);
  return reinterpret_cast<const float*>(p->tiles.data())[o];
}

// Runs first(i) for i in [0, n), then between() once, then, unless that said no, second(i) for i in [0, n): on up to eight
// threads if each gets at least `grain` units of work in all.  The threads are started once for both passes (starting and
// joining seven costs 0.25 ms).  What is thrown on any of them ends both passes early and is thrown again on this one.
template <typename F, typename G, typename H>
static void two_passes(int n, int64_t work, int64_t grain, const F& first, const G& between, const H& second) {
  const int threads = int(std::min<int64_t>(std::min<int64_t>(work / grain, n), std::min(8u, std::thread::hardware_concurrency())));
  if (threads <= 1) {
    for (int i = 0; i < n; ++i) first(i);
    if (!between()) return;
    for (int i = 0; i < n; ++i) second(i);
    return;
  }
  std::atomic<int> next[2] = {{0}, {0}}, done{0}, go{0};
  std::atomic<bool> failed{false};
  std::exception_ptr error;                              // of the thread that set `failed`; read after the join
  const int step = std::max(1, n / (threads * 8));       // pieces small enough to even out, large enough to be few
  const auto guarded = [&](const auto& fn) {
    try {
      fn();
    } catch (...) {
      if (!failed.exchange(true)) error = std::current_exception();
    }
  };
  const auto pass = [&](std::atomic<int>& at, const auto& fn) {
    guarded([&] {
      for (int i0 = at.fetch_add(step); i0 < n && !failed.load(std::memory_order_relaxed); i0 = at.fetch_add(step))
        for (int i = i0; i < std::min(n, i0 + step); ++i) fn(i);
    });
  };
  std::vector<std::thread> pool;
  pool.reserve(size_t(threads));
  try {
    for (int t = 1; t < threads; ++t)
      pool.emplace_back([&] {
        pass(next[0], first);
        done.fetch_add(1);
        while (go.load() == 0) std::this_thread::yield();
        if (go.load() == 1) pass(next[1], second);
      });
  } catch (const std::system_error&) {                   // no more threads to be had: the others do the work
  } catch (const std::bad_alloc&) {
  }
  pass(next[0], first);
  while (done.load() < int(pool.size())) std::this_thread::yield();
  bool on = false;
  if (!failed) guarded([&] { on = between(); });
  go = on ? 1 : 2;
  if (on) pass(next[1], second);
  for (std::thread& t : pool) t.join();
  if (error) std::rethrow_exception(error);
}

// For each bundle of n_tile output channels, list the (kernel location, 64-channel chunk)
// steps in which at least one kernel group of the bundle keeps that location; each step has an [n_tile][64]
// weight tile (zeros where a group prunes the location), which the device fills in (fill_umma_tiles does it
// here, for checks).  Steps are ordered by location, then chunk.
// `t_groups`: the order is (kh, kw), chunk, kt instead, and the steps that differ only in kt form a
// group (grp_ptr / grp_first): the CTA-pair kernel stages one input tile, Kt - 1 frames deeper, per group.
static const UmmaLayout* step_layout(rt3d_packed* p, int n_tile, bool t_groups, int chunk) {
  std::lock_guard<std::mutex> lock(p->mu);
  const int key = umma_key(n_tile, t_groups, p->dtype == RT3D_BF16 && chunk != kChunk);
  auto it = p->umma_layouts.find(key);
  if (it != p->umma_layouts.end()) return &it->second;

  UmmaLayout L;
  L.n_tile = n_tile;
  L.t_groups = t_groups;
  L.chunk = chunk;
  if (t_groups) L.grp_ptr.assign(1, 0);
  L.n_bundles = ceil_div(p->M, n_tile);
  L.n_chunks = ceil_div(p->N, chunk);
  L.step_ptr.assign(L.n_bundles + 1, 0);
  const int Ks = p->Ks;
  std::vector<int32_t> slot(size_t(Ks) * L.n_chunks);
  for (int b = 0; b < L.n_bundles; ++b) {
    const int m_lo = b * n_tile, m_hi = std::min(p->M, m_lo + n_tile);
    const int p_lo = m_lo / p->g_m, p_hi = ceil_div(m_hi, p->g_m);
    // pass 1: which steps are non-empty
    std::fill(slot.begin(), slot.end(), -1);
    for (int pr = p_lo; pr < p_hi; ++pr)
      for (int q = 0; q < p->Q; ++q) {
        const int c_lo = q * p->g_n, c_hi = std::min(p->N, c_lo + p->g_n), n_chunks = L.n_chunks;
        const uint16_t* const end = p->pos_idx.data() + p->group_ptr[size_t(pr) * p->Q + q + 1];
        for (int ch = c_lo / chunk; ch <= (c_hi - 1) / chunk; ++ch) {
          int32_t* const mark = slot.data() + ch;
          for (const uint16_t* e = p->pos_idx.data() + p->group_ptr[size_t(pr) * p->Q + q]; e < end; ++e) mark[size_t(*e) * n_chunks] = 0;
        }
      }
    const int32_t base = L.step_ptr[b];
    int32_t cnt = 0;
    if (!t_groups) {
      for (int kpos = 0; kpos < Ks; ++kpos)
        for (int ch = 0; ch < L.n_chunks; ++ch)
          if (slot[size_t(kpos) * L.n_chunks + ch] == 0) {
            slot[size_t(kpos) * L.n_chunks + ch] = base + cnt++;
            const int kw = kpos % p->Kw, kh = (kpos / p->Kw) % p->Kh, kt = kpos / (p->Kw * p->Kh);
            L.steps.push_back(encode_step(kt, kh, kw, ch));
          }
    } else {
      for (int hw = 0; hw < p->Kh * p->Kw; ++hw)
        for (int ch = 0; ch < L.n_chunks; ++ch) {
          bool open = false;
          for (int kt = 0; kt < p->Kt; ++kt) {
            const int kpos = kt * p->Kh * p->Kw + hw;
            if (slot[size_t(kpos) * L.n_chunks + ch] != 0) continue;
            if (!open) { L.grp_first.push_back(base + cnt); open = true; }
            slot[size_t(kpos) * L.n_chunks + ch] = base + cnt++;
            L.steps.push_back(encode_step(kt, hw / p->Kw, hw % p->Kw, ch));
          }
        }
      L.grp_ptr.push_back(int32_t(L.grp_first.size()));
    }
    L.step_ptr[b + 1] = base + cnt;
    L.max_steps = std::max(L.max_steps, int(cnt));
    L.slots.insert(L.slots.end(), slot.begin(), slot.end());
  }
  if (t_groups) L.grp_first.push_back(int32_t(L.steps.size()));     // sentinel: end of the last group
  auto res = p->umma_layouts.emplace(key, std::move(L));
  return &res.first->second;
}

const UmmaLayout* get_umma_layout(rt3d_packed* p, int n_tile, bool t_groups, bool narrow) {
  if (!umma_layout_possible(p) || (narrow && ceil_div(p->N, kNarrowChunk) > 4095)) return nullptr;
  if (n_tile <= 0) n_tile = default_n_tile(p->M);
  if (n_tile % 16 || n_tile > 256) return nullptr;
  return step_layout(p, n_tile, t_groups, narrow ? kNarrowChunk : kChunk);
}

// Whether the fp32 tensor-core kernel suits the weights:
//  - Each is zero or lies in [2^-100, 2^64): three bf16 parts hold it to the last bit then, and with the inputs' scale of 2^24 inputs
//    below 2^24 in magnitude keep every sum in range.
//  - No output channel's weights lean to one side: their sum more than half of the sum of their magnitudes, and more than weights of
//    both signs would show by chance.  The tensor core cuts addends off, always towards zero, which averages out in sums of both
//    signs and adds up in sums of one.  Errors against 64 bits over the CUDA cores', inputs of one sign: at most 0.81 on 300 random
//    layers with weights N(0, s^2), at most 1.1 on nine layers with N(s / 4, s^2), and up to 4.4 with weights of one sign.
static bool splits_well(const rt3d_packed* p) {
  const float* tiles = reinterpret_cast<const float*>(p->tiles.data());
  const int g_m = p->g_m, g_n = p->g_n, size = g_m * g_n;
  std::vector<float> sums(2 * size_t(size));
  for (int pr = 0; pr < p->P; ++pr) {
    const int64_t first = p->group_ptr[size_t(pr) * p->Q], end = p->group_ptr[size_t(pr + 1) * p->Q];
    float *const sum = sums.data(), *const mag = sum + size;       // of every place of a group, over the row's entries
    std::fill(sums.begin(), sums.end(), 0.f);
    int outside = 0;
    for (int64_t e = first; e < end; ++e) {
      const float* w = tiles + e * size;
      for (int v = 0; v < size; ++v) {
        const float m = std::fabs(w[v]);
        sum[v] += w[v];
        mag[v] += m;
        outside |= (int(m < 0x1p-100f) & int(m > 0.f)) | int(!(m < 0x1p64f));          // (NaNs are)
      }
    }
    if (outside) return false;
    const double chance = 25.0 / double(std::max<int64_t>(1, (end - first) * g_n));            // (five standard deviations)^2
    for (int i = 0; i < g_m; ++i) {
      double s = 0.0, m = 0.0;
      for (int k = 0; k < g_n; ++k) { s += sum[i * g_n + k]; m += mag[i * g_n + k]; }
      if (std::fabs(s) > 0.5 * m && s * s > chance * m * m) return false;
    }
  }
  return true;
}

const UmmaLayout* get_split_layout(rt3d_packed* p, int n_tile) {
  if (p->dtype != RT3D_F32 || p->Kt > 63 || p->Kh > 63 || p->Kw > 63 || ceil_div(p->N, kSplitChunk) > 4095) return nullptr;
  if (n_tile % 16 || n_tile < 16 || n_tile > 128) return nullptr;
  {
    std::lock_guard<std::mutex> lock(p->mu);
    if (p->splits_well < 0)
      p->splits_well = splits_well(p) ? 1 : 0;
    if (!p->splits_well) return nullptr;
  }
  return step_layout(p, n_tile, false, kSplitChunk);
}

// The weight tiles of a layout, as the device kernel builds them.
std::vector<uint16_t> fill_umma_tiles(const rt3d_packed* p, const UmmaLayout& L) {
  std::vector<uint16_t> wtiles(L.steps.size() * size_t(L.n_tile) * kChunk, 0);
  for (int pr = 0; pr < p->P; ++pr)
    for (int q = 0; q < p->Q; ++q)
      for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e)
        for (int i = 0; i < p->g_m && pr * p->g_m + i < p->M; ++i)
          for (int j = 0; j < p->g_n && q * p->g_n + j < p->N; ++j) {
            const int m = pr * p->g_m + i, c = q * p->g_n + j, b = m / L.n_tile;
            const int32_t s = L.slots[(size_t(b) * p->Ks + p->pos_idx[e]) * L.n_chunks + c / kChunk];
            wtiles[(size_t(s) * L.n_tile + (m - b * L.n_tile)) * kChunk + c % kChunk] =
                reinterpret_cast<const uint16_t*>(p->tiles.data())[(int64_t(e) * p->g_m + i) * p->g_n + j];
          }
  return wtiles;
}

// Layout of the sub-tile kernel (see SubLayout and SubStep).
const SubLayout* get_sub_layout(rt3d_packed* p, int n_tile) {
  if (!umma_layout_possible(p)) return nullptr;
  if (n_tile <= 0) n_tile = default_n_tile(p->M);
  if (n_tile % 16 || n_tile > 256) return nullptr;
  std::lock_guard<std::mutex> lock(p->mu);
  auto it = p->sub_layouts.find(n_tile);
  if (it != p->sub_layouts.end()) return &it->second;

  SubLayout L;
  L.n_tile = n_tile;
  L.n_bundles = ceil_div(p->M, n_tile);
  L.n_chunks = ceil_div(p->N, kChunk);
  L.step_ptr.assign(L.n_bundles + 1, 0);
  const int Ks = p->Ks;
  const uint16_t* tiles = reinterpret_cast<const uint16_t*>(p->tiles.data());
  std::vector<uint64_t> pres(size_t(Ks) * L.n_chunks);     // bit ks*16 + r: block (range r, K slice ks) exists
  std::vector<int32_t> slot(size_t(Ks) * L.n_chunks);
  for (int b = 0; b < L.n_bundles; ++b) {
    const int m_lo = b * n_tile, m_hi = std::min(p->M, m_lo + n_tile);
    const int n_ranges = ceil_div(m_hi - m_lo, kSubRange);
    const int p_lo = m_lo / p->g_m, p_hi = ceil_div(m_hi, p->g_m);
    // pass 1: which (range, K slice) blocks exist in which (location, chunk) step
    std::fill(pres.begin(), pres.end(), uint64_t(0));
    for (int pr = p_lo; pr < p_hi; ++pr) {
      const int r_lo = (std::max(pr * p->g_m, m_lo) - m_lo) / kSubRange;
      const int r_hi = (std::min(std::min((pr + 1) * p->g_m, p->M), m_hi) - 1 - m_lo) / kSubRange;
      uint64_t rbits = 0;
      for (int r = r_lo; r <= r_hi; ++r) rbits |= uint64_t(1) << r;
      for (int q = 0; q < p->Q; ++q) {
        const int c_lo = q * p->g_n, c_hi = std::min(p->N, c_lo + p->g_n);
        for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e)
          for (int sl = c_lo / 16; sl <= (c_hi - 1) / 16; ++sl)       // 16-channel slices the group touches
            pres[size_t(p->pos_idx[e]) * L.n_chunks + sl / 4] |= rbits << ((sl % 4) * 16);
      }
    }
    const int32_t first_step = int32_t(L.steps.size());
    for (int ch = 0; ch < L.n_chunks; ++ch)
      for (int kpos = 0; kpos < Ks; ++kpos) {
        uint64_t m = pres[size_t(kpos) * L.n_chunks + ch];
        slot[size_t(kpos) * L.n_chunks + ch] = -1;
        if (!m) continue;
        if (int32_t(L.steps.size()) == first_step) {          // first step: every range starts its accumulator here
          m |= (uint64_t(1) << n_ranges) - 1;
          pres[size_t(kpos) * L.n_chunks + ch] = m;
        }
        slot[size_t(kpos) * L.n_chunks + ch] = int32_t(L.steps.size());
        const int kw = kpos % p->Kw, kh = (kpos / p->Kw) % p->Kh, kt = kpos / (p->Kw * p->Kh);
        SubStep st{};
        st.enc = encode_step(kt, kh, kw, ch);
        st.off64 = unsigned(L.payload.size() / 64);
        st.nblk = __builtin_popcountll(m);
        L.steps.push_back(st);
        L.max_blocks = std::max(L.max_blocks, st.nblk);
        const size_t base = L.payload.size();
        L.payload.resize(base + kSubHeaderBytes + size_t(st.nblk) * kSubBlockBytes, 0);
        int idx = 0;
        for (int bit = 0; bit < 64; ++bit)
          if ((m >> bit) & 1) L.payload[base + size_t(4 * (bit % 16) + bit / 16)] = uint8_t(0x80 | idx++);
      }
    const int32_t end_step = int32_t(L.steps.size());
    L.step_ptr[b + 1] = end_step;
    L.max_steps = std::max(L.max_steps, int(end_step - first_step));
    // pass 2: scatter the kept weights into their blocks
    for (int pr = p_lo; pr < p_hi; ++pr)
      for (int q = 0; q < p->Q; ++q)
        for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e)
          for (int i = 0; i < p->g_m; ++i) {
            const int m = pr * p->g_m + i;
            if (m < m_lo || m >= m_hi) continue;
            const int r = (m - m_lo) / kSubRange, ri = (m - m_lo) % kSubRange;
            for (int j = 0; j < p->g_n; ++j) {
              const int c = q * p->g_n + j;
              if (c >= p->N) continue;
              const SubStep& st = L.steps[slot[size_t(p->pos_idx[e]) * L.n_chunks + c / kChunk]];
              const size_t base = size_t(st.off64) * 64;
              const int ks = (c % kChunk) / 16, kj = c % 16;
              const size_t blk = L.payload[base + size_t(4 * r + ks)] & 0x3F;
              uint16_t* dst = reinterpret_cast<uint16_t*>(L.payload.data() + base + kSubHeaderBytes + blk * kSubBlockBytes);
              dst[((ri / 8) * 2 + kj / 8) * 64 + (ri % 8) * 8 + kj % 8] = tiles[(int64_t(e) * p->g_m + i) * p->g_n + j];
            }
          }
  }
  auto res = p->sub_layouts.emplace(n_tile, std::move(L));
  return &res.first->second;
}

// Small-C_in layout for spatial strides (sh, sw): kernel locations kept by at least one group are
// sorted by the offset of their window inside the staged phase images and paired; each pair is one
// K=16 MMA whose two K halves are the 8 (padded) channels at the two locations.  Operands use the
// no-swizzle core-matrix layout (8 rows x 16 bytes).
static bool build_smallc_packed(rt3d_packed* p, SmallCLayout& L);
const SmallCLayout* get_smallc_layout(rt3d_packed* p, int sh, int sw, bool packed) {
  if (p->dtype != RT3D_BF16 || p->N > 8 || p->M > 256 || sh < 1 || sw < 1 || sh > 4 || sw > 4) return nullptr;
  std::lock_guard<std::mutex> lock(p->mu);
  const int key = sh * 16 + sw + (packed ? 1024 : 0);
  auto it = p->smallc_layouts.find(key);
  if (it != p->smallc_layouts.end()) return it->second.n_pad ? &it->second : nullptr;
  SmallCLayout L;
  L.sh = sh; L.sw = sw;
  L.n_pad = round_up(p->M, 16);
  if (packed) {
    if (!build_smallc_packed(p, L)) L.n_pad = 0;         // remembered as not to be had
    auto res = p->smallc_layouts.emplace(key, std::move(L));
    return res.first->second.n_pad ? &res.first->second : nullptr;
  }
  L.n_phases = sh * sw;
  L.img_w = kSmallCTileW - 1 + ceil_div(p->Kw, sw);
  L.img_h = kSmallCTileH - 1 + ceil_div(p->Kh, sh);
  L.img_t = p->Kt;
  L.phase_stride = round_up(L.img_w * L.img_h * L.img_t * 16, 128);   // a TMA box must land on a 128-byte boundary
  std::vector<uint8_t> used(size_t(p->Ks), 0);
  for (int64_t e = 0; e < p->nnz; ++e) used[p->pos_idx[size_t(e)]] = 1;
  std::vector<std::pair<int, int>> pos;            // (window offset, kernel location)
  for (int k = 0; k < p->Ks; ++k) {
    if (!used[size_t(k)]) continue;
    const int kw = k % p->Kw, kh = (k / p->Kw) % p->Kh, kt = k / (p->Kw * p->Kh);
    const int phase = (kh % sh) * sw + (kw % sw);
    pos.emplace_back(phase * L.phase_stride + ((kt * L.img_h + kh / sh) * L.img_w + kw / sw) * 16, k);
  }
  std::sort(pos.begin(), pos.end());
  L.n_pairs = ceil_div(int(pos.size()), 2);
  L.pair_off.assign(size_t(L.n_pairs) * 2, 0);
  L.wimg.assign(size_t(L.n_pairs) * 2 * L.n_pad * 8, 0);
  std::vector<int> slot(size_t(p->Ks), -1);       // location -> pair*2 + half
  for (size_t i = 0; i < pos.size(); ++i) {
    L.pair_off[i] = pos[i].first;
    slot[size_t(pos[i].second)] = int(i);
  }
  // An odd count leaves the last pair's second K half without a location: zero weights, read through the SAME window
  // as the first half.  (A window 16 bytes further on runs, for the tile's last voxel, past the end of the staged
  // image into shared memory that no load ever wrote; a NaN or infinity there times zero is a NaN in that voxel's
  // accumulators, which a following max-pool silently drops: rare, run-to-run different outputs.)
  if (pos.size() % 2) L.pair_off[pos.size()] = L.pair_off[pos.size() - 1];
  const uint16_t* tiles = reinterpret_cast<const uint16_t*>(p->tiles.data());
  for (int pr = 0; pr < p->P; ++pr)
    for (int q = 0; q < p->Q; ++q)
      for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e) {
        const int s = slot[p->pos_idx[size_t(e)]];
        for (int i = 0; i < p->g_m && pr * p->g_m + i < p->M; ++i)
          for (int j = 0; j < p->g_n && q * p->g_n + j < p->N; ++j) {
            const int m = pr * p->g_m + i, c = q * p->g_n + j;
            L.wimg[((size_t(s) * (L.n_pad / 8) + m / 8) * 8 + m % 8) * 8 + c] =
                tiles[(size_t(e) * p->g_m + i) * p->g_n + j];
          }
      }
  auto res = p->smallc_layouts.emplace(key, std::move(L));
  return &res.first->second;
}

constexpr int kF32MaxKs = 512;      // kernel locations the fp32 kernel's offset table holds

bool f32_layout_possible(const rt3d_packed* p) {
  return p->dtype == RT3D_F32 && p->g_m % 4 == 0 && p->g_n % 4 == 0 && p->Ks <= kF32MaxKs;
}

const F32Layout* get_f32_layout(rt3d_packed* p) {
  if (!f32_layout_possible(p)) return nullptr;
  std::lock_guard<std::mutex> lock(p->mu);
  if (p->f32_layout) return p->f32_layout.get();
  std::unique_ptr<F32Layout> layout(new F32Layout);
  F32Layout& L = *layout;
  L.quads = f32_stage_quads(p->Ks);
  const int n_rows = ceil_div(p->M, 4), n_quads = ceil_div(p->N, 4);
  L.n_sets = ceil_div(n_rows, 2);
  L.n_stages = ceil_div(n_quads, L.quads);
  const int Ks = p->Ks, rm = p->g_m / 4, rn = p->g_n / 4;
  const float* tiles = reinterpret_cast<const float*>(p->tiles.data());
  const int64_t work = int64_t(p->M) * p->N * Ks, grain = int64_t(1) << 18;
  const size_t n_lists = size_t(L.n_stages) * L.n_sets;
  L.entry_ptr.assign(n_lists + 1, 0);
  L.tile_ptr.assign(n_lists + 1, 0);
  L.counts.assign(n_lists, 0);
  // Packed entry that holds (row, quad, location) of one (stage, row set), or -1.
  auto find_kept = [&](int st, int s, std::vector<int32_t>& kept) {
    kept.assign(size_t(2) * L.quads * Ks, -1);
    for (int r = 0; r < 2 && s * 2 + r < n_rows; ++r)
      for (int ql = 0; ql < L.quads && st * L.quads + ql < n_quads; ++ql) {
        const size_t grp = size_t((s * 2 + r) / rm) * p->Q + (st * L.quads + ql) / rn;
        int32_t* at = kept.data() + size_t(r * L.quads + ql) * Ks;
        for (int32_t e = p->group_ptr[grp]; e < p->group_ptr[grp + 1]; ++e) at[p->pos_idx[e]] = e;
      }
  };
  const auto count_entries = [&](int st) {
    std::vector<int32_t> kept;
    for (int s = 0; s < L.n_sets; ++s) {
      find_kept(st, s, kept);
      int count[3] = {0, 0, 0};
      for (int v = 0; v < L.quads * Ks; ++v) {
        const bool e0 = kept[size_t(v)] >= 0, e1 = kept[size_t(L.quads) * Ks + v] >= 0;
        count[0] += e0 && e1; count[1] += e0 && !e1; count[2] += !e0 && e1;
      }
      const size_t at = size_t(st) * L.n_sets + s;
      L.counts[at] = count[0] | count[1] << 16;
      L.entry_ptr[at + 1] = count[0] + count[1] + count[2];
      L.tile_ptr[at + 1] = 2 * count[0] + count[1] + count[2];
    }
  };
  const auto allocate = [&] {
    for (size_t i = 0; i < n_lists; ++i) { L.entry_ptr[i + 1] += L.entry_ptr[i]; L.tile_ptr[i + 1] += L.tile_ptr[i]; }
    L.entries.resize(size_t(L.entry_ptr[n_lists]));
    L.tiles.allocate(size_t(L.tile_ptr[n_lists]) * 64);
    return true;
  };
  two_passes(L.n_stages, work, grain, count_entries, allocate, [&](int st) {
    std::vector<int32_t> kept;
    for (int s = 0; s < L.n_sets; ++s) {
      find_kept(st, s, kept);
      const size_t at = size_t(st) * L.n_sets + s;
      uint32_t* entry = L.entries.data() + L.entry_ptr[at];
      float* out = reinterpret_cast<float*>(L.tiles.data()) + size_t(L.tile_ptr[at]) * 16;
      for (int list = 0; list < 3; ++list)
        for (int ql = 0; ql < L.quads; ++ql)
          for (int k = 0; k < Ks; ++k) {
            const int32_t e[2] = {kept[size_t(ql) * Ks + k], kept[size_t(L.quads + ql) * Ks + k]};
            const int which = e[0] >= 0 ? (e[1] >= 0 ? 0 : 1) : (e[1] >= 0 ? 2 : -1);
            if (which != list) continue;
            *entry++ = uint32_t(k) | uint32_t(ql) << 16;
            for (int r = 0; r < 2; ++r) {
              if (e[r] < 0) continue;
              const int ib = ((s * 2 + r) % rm) * 4, jb = ((st * L.quads + ql) % rn) * 4;
              for (int i = 0; i < 4; ++i, out += 4)
                std::memcpy(out, tiles + (int64_t(e[r]) * p->g_m + ib + i) * p->g_n + jb, 16);
            }
          }
    }
  });
  for (int lg = 0; lg < 4; ++lg)
    for (int st = 0; st < L.n_stages; ++st)
      for (int s = 0; s < L.n_sets; s += 1 << lg) {
        const size_t a = size_t(st) * L.n_sets + s, b = size_t(st) * L.n_sets + std::min(L.n_sets, s + (1 << lg));
        L.max_entries[lg] = std::max(L.max_entries[lg], L.entry_ptr[b] - L.entry_ptr[a]);
        L.max_tiles[lg] = std::max(L.max_tiles[lg], L.tile_ptr[b] - L.tile_ptr[a]);
      }
  p->f32_layout = std::move(layout);
  return p->f32_layout.get();
}

// The packed form: entry e of a row holds columns (2e, 2e + 1), the kernel columns (2a, 2a + 1) read entries from a on; an
// odd last kernel column has entries of its own, with zeros behind it (a column outside the window must not be read even
// against zero weights: NaN x 0 is NaN).
static bool build_smallc_packed(rt3d_packed* p, SmallCLayout& L) {
  const int Kw = p->Kw, pairs = Kw / 2;
  if (p->N > 4 || L.sw != 2 || Kw > 32 || p->Kt > 15) return false;
  struct Entry { int lo, hi; };
  std::vector<Entry> row;                               // the entries of an image row: input columns, -1 = zeros
  struct Half { int slot, tap0, tap1; };
  std::vector<Half> halves;                             // what a kernel row reads: first entry, its two kernel columns
  if (pairs > 0)
    for (int e = 0; e < kSmallCTileW - 1 + pairs; ++e) row.push_back({2 * e, 2 * e + 1});
  for (int a = 0; a < pairs; ++a) halves.push_back({a, 2 * a, 2 * a + 1});
  if (Kw % 2) {
    halves.push_back({int(row.size()), Kw - 1, -1});
    for (int e = 0; e < kSmallCTileW; ++e) row.push_back({2 * e + Kw - 1, -1});
  }
  L.packed = true;
  L.n_phases = 1;
  L.img_w = int(row.size());
  L.img_h = (kSmallCTileH - 1) * L.sh + p->Kh;
  L.img_t = p->Kt;
  L.phase_stride = round_up(L.img_w * L.img_h * L.img_t * 16, 128);
  if (L.img_h > 63 || L.phase_stride > (1 << 16) * 8) return false;
  for (int t = 0; t < L.img_t; ++t)
    for (int h = 0; h < L.img_h; ++h)
      for (int e = 0; e < L.img_w; ++e)
        for (int half = 0; half < 2; ++half) {
          const int col = half ? row[size_t(e)].hi : row[size_t(e)].lo;
          if (col < 0) continue;
          if (col > 63) return false;
          L.ops.push_back(uint32_t(((t * L.img_h + h) * L.img_w + e) * 2 + half) | uint32_t(col) << 16 | uint32_t(h) << 22 |
                          uint32_t(t) << 28);
        }
  std::vector<uint8_t> used(size_t(p->Ks), 0);
  for (int64_t e = 0; e < p->nnz; ++e) used[p->pos_idx[size_t(e)]] = 1;
  std::vector<int> slot(size_t(p->Ks), -1);            // location -> (half index) * 2 + place in the half
  std::vector<int> offs;
  for (int kt = 0; kt < p->Kt; ++kt)
    for (int kh = 0; kh < p->Kh; ++kh)
      for (const Half& hf : halves) {
        const int base = (kt * p->Kh + kh) * Kw;
        const bool a = used[size_t(base + hf.tap0)], b = hf.tap1 >= 0 && used[size_t(base + hf.tap1)];
        if (!a && !b) continue;
        if (a) slot[size_t(base + hf.tap0)] = int(offs.size()) * 2;
        if (b) slot[size_t(base + hf.tap1)] = int(offs.size()) * 2 + 1;
        offs.push_back(((kt * L.img_h + kh) * L.img_w + hf.slot) * 16);
      }
  if (offs.size() % 2) offs.push_back(offs.back());    // the unused half of the last MMA reads the other half's window
  L.n_pairs = int(offs.size()) / 2;
  L.pair_off.assign(offs.begin(), offs.end());
  L.wimg.assign(size_t(L.n_pairs) * 2 * L.n_pad * 8, 0);
  const uint16_t* tiles = reinterpret_cast<const uint16_t*>(p->tiles.data());
  for (int pr = 0; pr < p->P; ++pr)
    for (int q = 0; q < p->Q; ++q)
      for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e) {
        const int at = slot[p->pos_idx[size_t(e)]];
        for (int i = 0; i < p->g_m && pr * p->g_m + i < p->M; ++i)
          for (int j = 0; j < p->g_n && q * p->g_n + j < p->N; ++j) {
            const int m = pr * p->g_m + i, c = q * p->g_n + j;
            L.wimg[((size_t(at / 2) * (L.n_pad / 8) + m / 8) * 8 + m % 8) * 8 + (at % 2) * 4 + c] =
                tiles[(size_t(e) * p->g_m + i) * p->g_n + j];
          }
      }
  return true;
}

static uint64_t next_handle_id() {
  static std::atomic<uint64_t> next_id{1};
  return next_id.fetch_add(1);
}

constexpr size_t kGatherGroup = 64;      // weights of a group that pass 2 gathers at once

// The tiles of one whole group, location by location.  GM, GN: the group's size where it is known when compiling (0: not),
// which turns the gather and the conversion into straight code (512 x 512 x 27, 4x4, eight threads: 1.25 -> 0.7 ms).
template <int GM, int GN>
static void gather_group(const float* base, int64_t row_len, int Ks, const uint16_t* pos, int n, int g_m_, int g_n_, int dtype,
                         unsigned char* out) {
  const int g_m = GM ? GM : g_m_, g_n = GN ? GN : g_n_, step = g_m * g_n;
  float v[GM && GN ? GM * GN : kGatherGroup];
  uint16_t b[GM && GN ? GM * GN : kGatherGroup];
  for (int e = 0; e < n; ++e) {
    for (int i = 0; i < g_m; ++i) {
      const float* at = base + pos[e] + i * row_len;
      for (int j = 0; j < g_n; ++j) v[i * g_n + j] = at[j * Ks];
    }
    if (dtype == RT3D_BF16) {
      for (int i = 0; i < step; ++i) b[i] = f32_to_bf16_bits(v[i]);
      std::memcpy(out, b, size_t(step) * 2);
      out += size_t(step) * 2;
    } else {
      std::memcpy(out, v, size_t(step) * 4);
      out += size_t(step) * 4;
    }
  }
}

static rt3d_status pack_impl(const float* w, const uint8_t* mask, int M, int N, int Kt, int Kh, int Kw,
                             int g_m, int g_n, int dtype, int is_dense, rt3d_packed** out) {
  if (!w || !out) return RT3D_ERR_INVALID_ARG;
  *out = nullptr;
  if (M <= 0 || N <= 0 || Kt <= 0 || Kh <= 0 || Kw <= 0) return RT3D_ERR_INVALID_ARG;
  if (g_m < 1 || g_n < 1 || g_m > kMaxGroup || g_n > kMaxGroup) return RT3D_ERR_INVALID_ARG;
  if (dtype != RT3D_F32 && dtype != RT3D_BF16) return RT3D_ERR_INVALID_ARG;
  const int64_t Ks64 = int64_t(Kt) * Kh * Kw;
  if (Ks64 > 65535) return RT3D_ERR_INVALID_ARG;
  return c_entry([&] {
    std::unique_ptr<rt3d_packed> owner(new rt3d_packed);
    rt3d_packed* const h = owner.get();
    h->id = next_handle_id();
    h->M = M; h->N = N; h->Kt = Kt; h->Kh = Kh; h->Kw = Kw; h->g_m = g_m; h->g_n = g_n;
    h->P = ceil_div(M, g_m); h->Q = ceil_div(N, g_n); h->Ks = int(Ks64);
    h->dtype = dtype; h->is_dense = is_dense;
    const int Ks = h->Ks;
    const size_t esz = dtype == RT3D_BF16 ? 2 : 4;
    const size_t n_groups = size_t(h->P) * h->Q;
    h->group_ptr.resize(n_groups + 1);
    // Both passes are shared between threads by groups, in memory order.
    const int64_t work = int64_t(M) * N * Ks, grain = int64_t(1) << 18;
    // pass 1: group-level decisions with the uniformity check of the KGS definition.  A kernel's bytes are nearly always
    // those of the group's first kernel, so they are compared as a block, and value by value (any nonzero value keeps a
    // weight) only where the blocks differ: 512 x 512 x 27 with 8 threads a millisecond of one thread -> 0.4.
    std::vector<uint8_t> keep(mask ? n_groups * Ks : 0);
    std::atomic<bool> uniform{true}, vanilla{true};
    const auto decide = [&](int grp) {
      if (!mask) { h->group_ptr[size_t(grp) + 1] = Ks; return; }
      const int pr = grp / h->Q, q = grp % h->Q, rows = std::min(g_m, M - pr * g_m), cols = std::min(g_n, N - q * g_n);
      uint8_t* kp = keep.data() + size_t(grp) * Ks;
      const uint8_t* first = mask + (int64_t(pr) * g_m * N + int64_t(q) * g_n) * Ks;
      int kept_here = 0;
      for (int k = 0; k < Ks; ++k) { kp[k] = first[k] != 0; kept_here += kp[k]; }
      for (int i = 0; i < rows; ++i)
        for (int j = 0; j < cols; ++j) {
          const uint8_t* row = first + (int64_t(i) * N + j) * Ks;
          if (std::memcmp(row, first, size_t(Ks)) == 0) continue;
          for (int k = 0; k < Ks; ++k)
            if (kp[k] != uint8_t(row[k] != 0)) uniform = false;
        }
      if (kept_here != 0 && kept_here != Ks && vanilla.load(std::memory_order_relaxed)) vanilla = false;   // written once
      h->group_ptr[size_t(grp) + 1] = kept_here;
    };
    rt3d_status status = RT3D_OK;
    const auto allocate = [&] {
      if (!uniform) { status = RT3D_ERR_MASK_NOT_GROUP_UNIFORM; return false; }
      int64_t nnz = 0;
      for (size_t grp = 0; grp < n_groups; ++grp) {
        nnz += h->group_ptr[grp + 1];
        if (nnz > 0x7FFFFFFF) { status = RT3D_ERR_UNSUPPORTED; return false; }
        h->group_ptr[grp + 1] = int32_t(nnz);
      }
      h->group_ptr[0] = 0;
      h->nnz = nnz;
      h->is_vanilla = vanilla;
      h->pos_idx.resize(size_t(nnz));
      h->tiles.allocate(size_t(nnz) * g_m * g_n * esz);
      return true;
    };
    // pass 2: emit index and tiles.  A small whole group is gathered tile by tile, which writes in order and converts in
    // vectors; otherwise kernel by kernel, which reads in order.
    two_passes(int(n_groups), work, grain, decide, allocate, [&](int grp) {
      const int pr = grp / h->Q, q = grp % h->Q, rows = std::min(g_m, M - pr * g_m), cols = std::min(g_n, N - q * g_n);
      const int32_t e0 = h->group_ptr[size_t(grp)], n_e = h->group_ptr[size_t(grp) + 1] - e0;
      const size_t step = size_t(g_m) * g_n;
      uint16_t* pos = h->pos_idx.data() + e0;
      int n = 0;
      for (int k = 0; k < Ks; ++k)
        if (!mask || keep[size_t(grp) * Ks + k]) pos[n++] = uint16_t(k);
      unsigned char* out = h->tiles.data() + size_t(e0) * step * esz;
      const float* base = w + (int64_t(pr) * g_m * N + int64_t(q) * g_n) * Ks;
      if (rows == g_m && cols == g_n && step <= kGatherGroup) {
        if (g_m == 4 && g_n == 4) gather_group<4, 4>(base, int64_t(N) * Ks, Ks, pos, n_e, 4, 4, dtype, out);
        else if (g_n == 4) gather_group<0, 4>(base, int64_t(N) * Ks, Ks, pos, n_e, g_m, 4, dtype, out);
        else gather_group<0, 0>(base, int64_t(N) * Ks, Ks, pos, n_e, g_m, g_n, dtype, out);
        return;
      }
      if (rows < g_m || cols < g_n) std::memset(out, 0, size_t(n_e) * step * esz);           // kernels that do not exist
      for (int i = 0; i < rows; ++i)
        for (int j = 0; j < cols; ++j) {
          const float* row = base + (int64_t(i) * N + j) * Ks;
          const size_t at = size_t(i) * g_n + j;
          if (dtype == RT3D_BF16) {
            uint16_t* o = reinterpret_cast<uint16_t*>(out) + at;
            for (int e = 0; e < n_e; ++e) o[e * step] = f32_to_bf16_bits(row[pos[e]]);
          } else {
            float* o = reinterpret_cast<float*>(out) + at;
            for (int e = 0; e < n_e; ++e) o[e * step] = row[pos[e]];
          }
        }
    });
    if (status == RT3D_OK) *out = owner.release();
    return status;
  });
}

}  // namespace rt3d

using namespace rt3d;

extern "C" {

rt3d_status rt3d_pack_kgs(const float* w, const uint8_t* mask, int M, int N, int Kt, int Kh, int Kw,
                          int g_m, int g_n, int compute_dtype, rt3d_packed** out) {
  return pack_impl(w, mask, M, N, Kt, Kh, Kw, g_m, g_n, compute_dtype, 0, out);
}

rt3d_status rt3d_pack_dense(const float* w, int M, int N, int Kt, int Kh, int Kw, int compute_dtype,
                            rt3d_packed** out) {
  return pack_impl(w, nullptr, M, N, Kt, Kh, Kw, 4, 4, compute_dtype, 1, out);
}

rt3d_status rt3d_pack_concat(const rt3d_packed* const* parts, int n_parts, rt3d_packed** out) {
  if (!parts || n_parts < 1 || !out) return RT3D_ERR_INVALID_ARG;
  *out = nullptr;
  int64_t nnz = 0, bytes = 0;
  for (int i = 0; i < n_parts; ++i) {
    const rt3d_packed *a = parts[0], *p = parts[i];
    if (!p) return RT3D_ERR_INVALID_ARG;
    if (p->N != a->N || p->Kt != a->Kt || p->Kh != a->Kh || p->Kw != a->Kw || p->g_m != a->g_m || p->g_n != a->g_n ||
        p->dtype != a->dtype || p->is_dense != a->is_dense || (i + 1 < n_parts && p->M % p->g_m))
      return RT3D_ERR_SHAPE;
    nnz += p->nnz;
    bytes += int64_t(p->tiles.size());
  }
  if (nnz > 0x7FFFFFFF) return RT3D_ERR_UNSUPPORTED;
  return c_entry([&] {
    std::unique_ptr<rt3d_packed> h(new rt3d_packed);
    h->id = next_handle_id();
    const rt3d_packed* a = parts[0];
    h->N = a->N; h->Kt = a->Kt; h->Kh = a->Kh; h->Kw = a->Kw; h->g_m = a->g_m; h->g_n = a->g_n; h->Q = a->Q; h->Ks = a->Ks;
    h->dtype = a->dtype; h->is_dense = a->is_dense; h->is_vanilla = 1;
    h->tiles.allocate(size_t(bytes));
    h->group_ptr.push_back(0);
    unsigned char* at = h->tiles.data();
    for (int i = 0; i < n_parts; ++i) {
      const rt3d_packed* p = parts[i];
      h->M += p->M; h->P += p->P;
      h->is_vanilla = h->is_vanilla && p->is_vanilla;
      for (size_t g = 1; g < p->group_ptr.size(); ++g) h->group_ptr.push_back(int32_t(h->nnz) + p->group_ptr[g]);
      h->pos_idx.insert(h->pos_idx.end(), p->pos_idx.begin(), p->pos_idx.end());
      if (p->tiles.size()) std::memcpy(at, p->tiles.data(), p->tiles.size());
      at += p->tiles.size();
      h->nnz += p->nnz;
    }
    *out = h.release();
    return RT3D_OK;
  });
}

rt3d_status rt3d_packed_view_get(const rt3d_packed* p, rt3d_packed_view* v) {
  if (!p || !v) return RT3D_ERR_INVALID_ARG;
  v->M = p->M; v->N = p->N; v->Kt = p->Kt; v->Kh = p->Kh; v->Kw = p->Kw;
  v->g_m = p->g_m; v->g_n = p->g_n; v->P = p->P; v->Q = p->Q; v->Ks = p->Ks;
  v->dtype = p->dtype; v->is_vanilla = p->is_vanilla; v->is_dense = p->is_dense; v->nnz = p->nnz;
  v->group_ptr = p->group_ptr.data();
  v->pos_idx = p->pos_idx.data();
  v->tiles = p->tiles.data();
  return RT3D_OK;
}

rt3d_status rt3d_unpack_to_dense(const rt3d_packed* p, float* w_out) {
  if (!p || !w_out) return RT3D_ERR_INVALID_ARG;
  std::memset(w_out, 0, sizeof(float) * size_t(p->M) * p->N * p->Ks);
  for (int pr = 0; pr < p->P; ++pr)
    for (int q = 0; q < p->Q; ++q)
      for (int32_t e = p->group_ptr[size_t(pr) * p->Q + q]; e < p->group_ptr[size_t(pr) * p->Q + q + 1]; ++e)
        for (int i = 0; i < p->g_m && pr * p->g_m + i < p->M; ++i)
          for (int j = 0; j < p->g_n && q * p->g_n + j < p->N; ++j)
            w_out[(int64_t(pr * p->g_m + i) * p->N + (q * p->g_n + j)) * p->Ks + p->pos_idx[e]] =
                tile_value(p, e, i, j);
  return RT3D_OK;
}

namespace {
rt3d_status unpack_device_layout(const rt3d_packed* p, int n_tile, bool t_groups, float* w_out);
}
rt3d_status rt3d_unpack_device_layout(const rt3d_packed* p, int n_tile, float* w_out) {
  return c_entry([&] { return unpack_device_layout(p, n_tile, false, w_out); });
}
rt3d_status rt3d_unpack_device_layout_tgroups(const rt3d_packed* p, int n_tile, float* w_out) {
  return c_entry([&] { return unpack_device_layout(p, n_tile, true, w_out); });
}
namespace {
rt3d_status unpack_device_layout(const rt3d_packed* p, int n_tile, bool t_groups, float* w_out) {
  if (!p || !w_out) return RT3D_ERR_INVALID_ARG;
  const UmmaLayout* L = get_umma_layout(const_cast<rt3d_packed*>(p), n_tile, t_groups);
  if (!L) return RT3D_ERR_UNSUPPORTED;
  const std::vector<uint16_t> wtiles = fill_umma_tiles(p, *L);
  if (t_groups) {
    // groups tile each bundle's list exactly; inside a group only kt changes, upwards
    if (int(L->grp_ptr.size()) != L->n_bundles + 1 || L->grp_first.size() != size_t(L->grp_ptr.back()) + 1 ||
        L->grp_first.back() != int32_t(L->steps.size()))
      return RT3D_ERR_INVALID_ARG;
    for (int b = 0; b < L->n_bundles; ++b) {
      if (L->grp_ptr[b] > L->grp_ptr[b + 1]) return RT3D_ERR_INVALID_ARG;
      const int32_t first = L->grp_ptr[b] < L->grp_ptr[b + 1] ? L->grp_first[L->grp_ptr[b]] : L->step_ptr[b];
      if (first != L->step_ptr[b]) return RT3D_ERR_INVALID_ARG;
      for (int32_t g = L->grp_ptr[b]; g < L->grp_ptr[b + 1]; ++g) {
        const int32_t s0 = L->grp_first[g], s1 = L->grp_first[g + 1];
        if (s1 <= s0 || s1 - s0 > p->Kt || s1 > L->step_ptr[b + 1]) return RT3D_ERR_INVALID_ARG;
        int kt0, kh0, kw0, ch0;
        decode_step(L->steps[s0], kt0, kh0, kw0, ch0);
        for (int32_t s = s0 + 1; s < s1; ++s) {
          int kt, kh, kw, ch;
          decode_step(L->steps[s], kt, kh, kw, ch);
          if (kh != kh0 || kw != kw0 || ch != ch0 || kt <= kt0) return RT3D_ERR_INVALID_ARG;
          kt0 = kt;
        }
      }
    }
  }
  std::memset(w_out, 0, sizeof(float) * size_t(p->M) * p->N * p->Ks);
  for (int b = 0; b < L->n_bundles; ++b)
    for (int32_t s = L->step_ptr[b]; s < L->step_ptr[b + 1]; ++s) {
      int kt, kh, kw, ch;
      decode_step(L->steps[s], kt, kh, kw, ch);
      const int kpos = (kt * p->Kh + kh) * p->Kw + kw;
      for (int r = 0; r < L->n_tile && b * L->n_tile + r < p->M; ++r)
        for (int j = 0; j < kChunk && ch * kChunk + j < p->N; ++j)
          w_out[(int64_t(b * L->n_tile + r) * p->N + (ch * kChunk + j)) * p->Ks + kpos] =
              bf16_bits_to_f32(wtiles[(size_t(s) * L->n_tile + r) * kChunk + j]);
    }
  return RT3D_OK;
}
}  // namespace

rt3d_status rt3d_unpack_sub_layout(const rt3d_packed* p, int n_tile, float* w_out) {
  if (!p || !w_out) return RT3D_ERR_INVALID_ARG;
  const SubLayout* L = nullptr;
  const rt3d_status built = c_entry([&] { L = get_sub_layout(const_cast<rt3d_packed*>(p), n_tile); return RT3D_OK; });
  if (built != RT3D_OK || !L) return built != RT3D_OK ? built : RT3D_ERR_UNSUPPORTED;
  std::memset(w_out, 0, sizeof(float) * size_t(p->M) * p->N * p->Ks);
  for (int b = 0; b < L->n_bundles; ++b) {
    const int n_ranges = ceil_div(std::min(L->n_tile, p->M - b * L->n_tile), kSubRange);
    for (int32_t s = L->step_ptr[b]; s < L->step_ptr[b + 1]; ++s) {
      const SubStep& st = L->steps[s];
      int kt, kh, kw, ch;
      decode_step(st.enc, kt, kh, kw, ch);
      const int kpos = (kt * p->Kh + kh) * p->Kw + kw;
      const unsigned char* hdr = L->payload.data() + size_t(st.off64) * 64;
      int seen = 0;
      for (int r = 0; r < 16; ++r)
        for (int ks = 0; ks < 4; ++ks) {
          const unsigned char cmd = hdr[4 * r + ks];
          // the first step of a bundle must start every range's accumulator in K slice 0
          if (s == L->step_ptr[b] && ks == 0 && r < n_ranges && !(cmd & 0x80)) return RT3D_ERR_INVALID_ARG;
          if (!(cmd & 0x80)) continue;
          if (r >= n_ranges || (cmd & 0x3F) >= st.nblk) return RT3D_ERR_INVALID_ARG;
          ++seen;
          const uint16_t* blk = reinterpret_cast<const uint16_t*>(hdr + kSubHeaderBytes + size_t(cmd & 0x3F) * kSubBlockBytes);
          for (int i = 0; i < 16; ++i)
            for (int j = 0; j < 16; ++j) {
              const int m = b * L->n_tile + r * 16 + i, c = ch * kChunk + ks * 16 + j;
              const float v = bf16_bits_to_f32(blk[((i / 8) * 2 + j / 8) * 64 + (i % 8) * 8 + j % 8]);
              if (m < p->M && c < p->N) w_out[(int64_t(m) * p->N + c) * p->Ks + kpos] += v;
              else if (v != 0.f) return RT3D_ERR_INVALID_ARG;
            }
        }
      if (seen != st.nblk) return RT3D_ERR_INVALID_ARG;
    }
  }
  return RT3D_OK;
}

}  // extern "C"
