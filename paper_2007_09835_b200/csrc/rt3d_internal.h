// Internal declarations shared by the translation units of librt3d (host side).
#pragma once

#include <cstdint>
#include <cstddef>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <vector>

#include "rt3d.h"
#include "tile_consts.h"

namespace rt3d {

constexpr int kMaxGroup = 256;      // g_m, g_n <= 256 (pack, tensor-core kernels)
constexpr int kMaxGroupSimt = 8;    // the CUDA-core kernel keeps one group row in registers: g_m, g_n <= 8
constexpr int kChunk = 64;          // input channels per tensor-core K step (one 128-byte swizzle row of bf16)
constexpr int kNarrowChunk = 32;    // the same for layers of up to 32
constexpr int kSplitChunk = 32;     // the same of the fp32 tensor-core kernel (one 128-byte row of fp32)
constexpr int kTileM = 128;         // output voxels per tensor-core tile (TMEM lanes)

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline int64_t ceil_div64(int64_t a, int64_t b) { return (a + b - 1) / b; }
inline int round_up(int a, int b) { return ceil_div(a, b) * b; }

// Round-to-nearest-even float -> bfloat16 bits (NaN kept quiet), and back.
// Inline: a function that the library exports is called through its linkage table, once per weight.
inline uint16_t f32_to_bf16_bits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  const uint32_t rounded = u + 0x7FFFu + ((u >> 16) & 1u);          // ties to even
  return uint16_t(((u & 0x7FFFFFFFu) > 0x7F800000u ? u | 0x400000u : rounded) >> 16);    // a NaN stays one
}
float bf16_bits_to_f32(uint16_t b);

// Encoded K step of the tensor-core path: which kernel location and which 64-channel chunk.
inline int32_t encode_step(int kt, int kh, int kw, int chunk) {
  return (kt << 24) | (kh << 18) | (kw << 12) | chunk;
}
inline void decode_step(int32_t s, int& kt, int& kh, int& kw, int& chunk) {
  kt = (s >> 24) & 63; kh = (s >> 18) & 63; kw = (s >> 12) & 63; chunk = s & 4095;
}

// Weight layout consumed by the tcgen05 kernel, derived from the canonical arrays for one
// bundle width n_tile (output channels per accumulator tile).
struct UmmaLayout {
  int n_tile = 0;                    // multiple of 16, <= 256
  int n_bundles = 0;                 // ceil(M / n_tile)
  int chunk = kChunk;                // input channels of a step
  int n_chunks = 0;                  // ceil(N / chunk)
  std::vector<int32_t> step_ptr;     // [n_bundles + 1] offsets into steps / weight tiles
  std::vector<int32_t> steps;        // encoded (kt,kh,kw,chunk), only non-empty steps of each bundle
  std::vector<int32_t> slots;        // [n_bundles][Ks][n_chunks] index of that (location, chunk)'s step, -1 if it has none
  int max_steps = 0;                 // longest bundle list
  bool t_groups = false;             // steps ordered (kh, kw), chunk, kt; groups = runs that differ only in kt
  std::vector<int32_t> grp_ptr;      // [n_bundles + 1] offsets into grp_first            (t_groups only)
  std::vector<int32_t> grp_first;    // first step of each group, + one sentinel           (t_groups only)
};

// Layout for the small-C_in tensor-core kernel (C_in <= 8, channel pitch 8) at spatial strides
// (sh, sw): the input under a 1x16x8 output tile is staged as sh*sw phase images (every sh-th row and
// sw-th column), so that consecutive outputs are consecutive voxels of an image and every kernel
// location is a shifted window of one image.  K is walked in pairs of kernel locations (8 padded
// channels each), one K=16 MMA per pair.
//
// Packed form (C_in <= 4, sw = 2): an image entry of 16 bytes holds four channels of TWO input columns, the two that one
// pair of kernel columns reads, so that a K=16 MMA covers four kernel locations instead of two.  All input rows are staged
// (an output row is sh image rows down), the producer composes the entries from 8-byte copies listed in `ops`.
struct SmallCLayout {
  bool packed = false;
  std::vector<uint32_t> ops;         // packed: destination / 8 in the image | column << 16 | row << 22 | frame << 28
  int sh = 1, sw = 1;
  int n_pad = 0;                     // output channels rounded up to 16 (<= 256)
  int n_pairs = 0;
  int n_phases = 1;                  // sh * sw
  int img_w = 0, img_h = 0, img_t = 0;   // voxels of one phase image
  int phase_stride = 0;              // bytes between phase images in shared memory
  std::vector<int32_t> pair_off;     // [n_pairs][2] byte offset of each location's window inside the staged images
  std::vector<uint16_t> wimg;        // [n_pairs][2][n_pad/8][8][8] bf16 bits, zero where pruned / absent
};

// Layout consumed by the sub-tile kernel: per bundle of n_tile output channels the list of non-empty K steps in
// chunk-major order (all kernel locations of a 64-channel chunk, then the next chunk: the input block under a
// tile is then re-read from the L1 cache), each with its block mask, and the blocks themselves.  A block holds
// W[16 output channels][16 input channels] of one kernel location as four 8 x 8 core matrices
// [row group][K half][8 rows][8 channels] (no-swizzle K-major operand: 128 bytes between K halves, 256 between
// row groups).
struct SubLayout {
  int n_tile = 0, n_bundles = 0, n_chunks = 0;
  std::vector<int32_t> step_ptr;     // [n_bundles + 1]
  std::vector<SubStep> steps;
  std::vector<unsigned char> payload; // per step: 64-byte header + its blocks ([nblk][256] bf16 bits)
  int max_blocks = 0;                // most blocks in one step
  int max_steps = 0;                 // longest bundle list
};

// Runs the body of a C entry point.  No exception crosses it: what can be thrown in the library says that host memory or
// another resource of the process could not be had.
template <typename F>
rt3d_status c_entry(const F& body) noexcept {
  try {
    return body();
  } catch (...) {
    return RT3D_ERR_ALLOC;
  }
}

// Host memory of the packed weights: a block kept from a freed handle, or a new one (pack.cpp).
unsigned char* host_block(size_t bytes);
void host_block_free(unsigned char* p);
void host_blocks_release();

// Bytes that are written once, without the zeros a vector would fill them with first.
class RawBytes {
 public:
  void allocate(size_t n) { data_.reset(host_block(n)); size_ = n; }
  unsigned char* data() { return data_.get(); }
  const unsigned char* data() const { return data_.get(); }
  size_t size() const { return size_; }
  unsigned char operator[](size_t i) const { return data_[i]; }

 private:
  struct Free { void operator()(unsigned char* p) const { host_block_free(p); } };
  std::unique_ptr<unsigned char[], Free> data_;
  size_t size_ = 0;
};

// Layout of the register-blocked fp32 kernel (simt_conv_f32.cu).  Kernel groups are cut into 4 x 4 tiles; a "row set" is
// two consecutive rows of four output channels, a stage is `quads` consecutive quads of input channels.  For each
// (stage, row set), stage-major, three lists of entries, one after the other: the (quad, kernel location) places that
// both rows keep, that only the first and that only the second keeps, each with one tile per row that keeps it.
struct F32Layout {
  int quads = 0, n_sets = 0, n_stages = 0;
  std::vector<int32_t> entry_ptr;    // [n_stages * n_sets + 1]
  std::vector<int32_t> tile_ptr;     // [n_stages * n_sets + 1]
  std::vector<int32_t> counts;       // [n_stages * n_sets] entries of the first list | of the second << 16
  std::vector<uint32_t> entries;     // kernel location | quad inside the stage << 16
  RawBytes tiles;                    // float [tile][4 outputs][4 inputs]
  int max_entries[4] = {0, 0, 0, 0}; // most entries / tiles of a stage in 1, 2, 4, 8 aligned consecutive row sets
  int max_tiles[4] = {0, 0, 0, 0};
};

// Per-device copies of a handle's arrays.
struct DeviceBlob {
  int device = -1;
  void* canonical = nullptr;         // owns the canonical arrays and the first tensor-core layout built from them
  int32_t* group_ptr = nullptr;
  uint16_t* pos_idx = nullptr;
  void* tiles = nullptr;
  struct Umma {
    void* base = nullptr;                       // owns the tiles and index arrays, unless they lie in `canonical`
    void* wtiles = nullptr;
    int32_t* step_ptr = nullptr;
    int32_t* steps = nullptr;
    alignas(64) unsigned char wmap[128];   // CUtensorMap of wtiles, box = one [n_tile][64] tile
    alignas(64) unsigned char wmap_half[128];   // same tensor, box = half a tile (CTA-pair kernel)
    int32_t* grp_ptr = nullptr;                 // t-grouped layouts only
    int32_t* grp_first = nullptr;
    bool ready = false;
  };
  std::map<int, Umma> umma;          // keyed like the handle's layouts
  struct Sub { void* steps = nullptr; int32_t* step_ptr = nullptr; void* blocks = nullptr; bool ready = false; };
  std::map<int, Sub> sub;            // sub-tile kernel, keyed by n_tile
  struct SmallC { void* base = nullptr; unsigned short* wimg = nullptr; int32_t* pairs = nullptr; uint32_t* ops = nullptr; };
  std::map<int, SmallC> smallc;      // small-C_in kernel: weight image, window offsets and copies, keyed like the layouts
  struct F32 { void* base = nullptr; int32_t* entry_ptr = nullptr; int32_t* tile_ptr = nullptr; int32_t* counts = nullptr; uint32_t* entries = nullptr; float* tiles = nullptr; };
  F32 f32;                           // register-blocked fp32 kernel
  // Scratch of the CTA-pair kernel's tail splits: partial tiles, and flags that are zero between launches.  The last one is the
  // largest; the others stay because captured graphs and prepared calls hold their addresses.
  struct Tail { float* partial = nullptr; size_t bytes = 0; int32_t* flags = nullptr; size_t flag_bytes = 0; };
  std::vector<Tail> tails;
  void* stage_x = nullptr; size_t stage_x_bytes = 0;   // staging for rt3d_conv3d_host
  void* stage_y = nullptr; size_t stage_y_bytes = 0;
  int stage_y_pitch = 0;                               // channel pitch at which stage_y's padding holds zeros, 0 = none
  float* stage_bias = nullptr;
  // rt3d_conv3d_host pipelines a large batch in chunks: copy-in and copy-out streams and events
  // (cudaStream_t / cudaEvent_t, created on first use)
  void* host_streams[2] = {nullptr, nullptr};
  void* host_events[18] = {};
};

}  // namespace rt3d

namespace rt3d { struct PreparedCall; }

struct rt3d_packed {
  uint64_t id = 0;                   // never used twice in a process
  int M = 0, N = 0, Kt = 0, Kh = 0, Kw = 0, g_m = 0, g_n = 0, P = 0, Q = 0, Ks = 0;
  int dtype = 0, is_vanilla = 0, is_dense = 0;
  int64_t nnz = 0;
  std::vector<int32_t> group_ptr;
  std::vector<uint16_t> pos_idx;
  rt3d::RawBytes tiles;              // nnz * g_m * g_n elements of float or bf16 bits
  std::mutex mu;                     // guards the lazily built members below
  std::map<int, rt3d::UmmaLayout> umma_layouts;   // keyed by umma_key
  int splits_well = -1;              // fp32: whether three bf16 parts hold every weight and sums lose nothing (-1: not looked at yet)
  std::map<int, rt3d::SubLayout> sub_layouts;     // keyed by n_tile
  std::map<int, rt3d::SmallCLayout> smallc_layouts;   // keyed by sh*16+sw (+ 1024: packed), built on first use
  std::unique_ptr<rt3d::F32Layout> f32_layout;        // built on first use
  std::vector<rt3d::DeviceBlob*> blobs;
  // The last few calls made with this handle, ready to launch again (api.cu); the oldest one gives way.
  std::vector<std::shared_ptr<rt3d::PreparedCall>> calls;
  size_t next_call = 0;
};

namespace rt3d {

// The weight tiles [steps.size()][n_tile][64] of a layout on the host (checks; the device fills its own).
std::vector<uint16_t> fill_umma_tiles(const rt3d_packed* p, const UmmaLayout& L);

inline int umma_key(int n_tile, bool t_groups, bool narrow) { return n_tile + (t_groups ? 4096 : 0) + (narrow ? 8192 : 0); }
// Default bundle width for M output channels: as few bundles as possible with n_tile <= 256.
int default_n_tile(int M);
// Builds (or returns the cached) tensor-core layout; nullptr if the handle cannot use it.
const UmmaLayout* get_umma_layout(rt3d_packed* p, int n_tile, bool t_groups = false, bool narrow = false);
bool umma_layout_possible(const rt3d_packed* p);
// Steps of 32 input channels for the fp32 tensor-core kernel; nullptr if the handle or its weights do not suit it.
const UmmaLayout* get_split_layout(rt3d_packed* p, int n_tile);
// Builds (or returns the cached) layout of the sub-tile kernel; nullptr if the handle cannot use it.
const SubLayout* get_sub_layout(rt3d_packed* p, int n_tile);

// Small-C_in layout (nullptr if the handle does not qualify: needs bf16, N <= 8, M <= 256).
// `packed`: the form with two columns an entry (nullptr unless N <= 4, sw = 2 and the image fits its offsets).
const SmallCLayout* get_smallc_layout(rt3d_packed* p, int sh, int sw, bool packed = false);

// Layout of the register-blocked fp32 kernel (nullptr unless fp32 with group sizes that are multiples of four).
bool f32_layout_possible(const rt3d_packed* p);
const F32Layout* get_f32_layout(rt3d_packed* p);

}  // namespace rt3d
