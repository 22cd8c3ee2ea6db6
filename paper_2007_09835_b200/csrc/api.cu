// C ABI of librt3d: argument validation, per-device weight upload, tile planning, TMA tensor
// maps and kernel dispatch.  All numerical work happens in the kernels launched from here.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <vector>

#include "kernels.h"
#include "kept_blocks.h"
#include "rt3d_internal.h"

using namespace rt3d;

namespace {

std::atomic<int64_t> g_launches{0};
std::atomic<int64_t> g_allocs{0};            // device allocations made by this library (rt3d_alloc_count)

// Device memory of uploaded layouts.  Never destroyed: handles may be freed while the process exits.
KeptBlocks& weight_blocks() {
  static KeptBlocks* kept = new KeptBlocks([](void* p) { cudaFree(p); });
  return *kept;
}

// Every device allocation of the library goes through here.
cudaError_t dev_malloc(void** p, size_t bytes) {
  g_allocs.fetch_add(1);
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    weight_blocks().release_all();
    g_allocs.fetch_add(1);
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) cudaGetLastError();                      // this call's answer, not that of the next one that asks
  return e;
}
template <typename T>
cudaError_t dev_malloc(T** p, size_t bytes) { return dev_malloc(reinterpret_cast<void**>(p), bytes); }

cudaError_t weight_malloc(void** p, size_t bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((*p = weight_blocks().take(bytes, dev)) != nullptr) return cudaSuccess;
  if ((e = dev_malloc(p, bytes)) == cudaSuccess) weight_blocks().note(*p, bytes, dev);
  return e;
}
// `idle`: the caller has waited for the kernels that may read the block, which cudaFree would do; only then is it kept.
void weight_free(void* p, bool idle) { idle ? weight_blocks().give(p) : weight_blocks().drop(p); }

// Planning mode of the calling thread (rt3d_plan_begin / rt3d_plan_end): compute calls do everything they would do
// before their launch (choose the kernel, build and upload weight layouts, size the workspaces) and return.
thread_local bool t_plan_only = false;

// Test hooks of the single-CTA tensor-core kernel (rt3d_debug_set).
std::atomic<long long> g_debug_wait_cycles{-1};      // -1: not set yet (RT3D_DEBUG_TIMEOUT_POLLS is read on first use)
std::atomic<int> g_debug_drop_last_load{0};
// t-grouped CTA-pair variant: on unless the environment says RT3D_T_GROUPS=0; RT3D_DEBUG_T_GROUPS switches it at run time
std::atomic<int> g_ts_enabled{[] { const char* e = getenv("RT3D_T_GROUPS"); return (e && e[0] == '0') ? 0 : 1; }()};
// steps of 32 input channels (kNarrowChunk): RT3D_DEBUG_NARROW switches them off and on
std::atomic<int> g_narrow_enabled{1};
// fp32 on the tensor cores: 0 never, 1 where it is expected to be faster, 2 wherever it can run (tests, comparisons)
std::atomic<int> g_f32_split{1};
long long debug_wait_cycles() {
  long long v = g_debug_wait_cycles.load();
  if (v < 0) {
    const char* e = getenv("RT3D_DEBUG_TIMEOUT_POLLS");
    v = e ? atoll(e) : 0;
    if (v < 0) v = 0;
    g_debug_wait_cycles.store(v);
  }
  return v;
}

// All device blobs of live handles: their tail-split flags are cleared when a kernel reported a timeout.
std::mutex g_blobs_mu;
std::vector<DeviceBlob*> g_blobs;

struct DeviceState {
  bool init = false;
  int sm_count = 0;
  int cc_major = 0;
  int32_t* sched = nullptr;     // [256] words: [2] = error word written by kernels on a bounded-wait expiry
};
std::mutex g_dev_mu;
DeviceState g_dev[64];

// Copies from pageable memory and fills go through the legacy stream and may return before they have reached the device, and
// a caller's non-blocking stream does not wait for that stream: what a kernel reads has to be there before it is launched.
cudaError_t uploads_done() { return cudaStreamSynchronize(cudaStreamLegacy); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);
ReplaceAddressFn g_replace_address = nullptr;

rt3d_status get_device_state(DeviceState** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RT3D_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_dev_mu);
  DeviceState& d = g_dev[dev];
  if (!d.init) {
    if (cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return RT3D_ERR_CUDA;
    if (cudaDeviceGetAttribute(&d.cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return RT3D_ERR_CUDA;
    if (dev_malloc(&d.sched, 256 * sizeof(int32_t)) != cudaSuccess) return RT3D_ERR_ALLOC;
    if (cudaMemset(d.sched, 0, 256 * sizeof(int32_t)) != cudaSuccess || uploads_done() != cudaSuccess) return RT3D_ERR_CUDA;
    if (!g_encode) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult qres;
      if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn)
        return RT3D_ERR_CUDA;
      void* replace = nullptr;
      if (cudaGetDriverEntryPoint("cuTensorMapReplaceAddress", &replace, cudaEnableDefault, &qres) != cudaSuccess || !replace)
        return RT3D_ERR_CUDA;
      g_replace_address = reinterpret_cast<ReplaceAddressFn>(replace);
      g_encode = reinterpret_cast<EncodeTiledFn>(fn);
    }
    d.init = true;
  }
  *out = &d;
  return RT3D_OK;
}

bool valid_dtype(int d) { return d == RT3D_F32 || d == RT3D_BF16; }
size_t elem_size(int d) { return d == RT3D_BF16 ? 2 : 4; }

rt3d_status check_tensor(const rt3d_tensor* t) {
  if (!t || !t->data) return RT3D_ERR_INVALID_ARG;
  if (t->n <= 0 || t->t <= 0 || t->h <= 0 || t->w <= 0 || t->c <= 0) return RT3D_ERR_INVALID_ARG;
  if (!valid_dtype(t->dtype) || t->c_stride < t->c) return RT3D_ERR_INVALID_ARG;
  return RT3D_OK;
}

int64_t tensor_span_bytes(const rt3d_tensor* t) {
  const int64_t vox = int64_t(t->n) * t->t * t->h * t->w;
  return ((vox - 1) * t->c_stride + t->c) * int64_t(elem_size(t->dtype));
}

rt3d_status make_geom(const rt3d_tensor* x, const rt3d_packed* w, const rt3d_conv_params* p, const rt3d_tensor* y,
                      ConvGeom* g) {
  rt3d_status s = check_tensor(x);
  if (s != RT3D_OK) return s;
  if (!w || !p) return RT3D_ERR_INVALID_ARG;
  if (p->st < 1 || p->sh < 1 || p->sw < 1 || p->pt < 0 || p->ph < 0 || p->pw < 0) return RT3D_ERR_INVALID_ARG;
  if (p->algo < RT3D_ALGO_AUTO || p->algo > RT3D_ALGO_UMMA_SUB) return RT3D_ERR_INVALID_ARG;
  if (x->c != w->N || x->dtype != w->dtype) return RT3D_ERR_SHAPE;
  const int64_t To = (int64_t(x->t) + 2 * p->pt - w->Kt) / p->st + 1;
  const int64_t Ho = (int64_t(x->h) + 2 * p->ph - w->Kh) / p->sh + 1;
  const int64_t Wo = (int64_t(x->w) + 2 * p->pw - w->Kw) / p->sw + 1;
  if (x->t + 2 * p->pt < w->Kt || x->h + 2 * p->ph < w->Kh || x->w + 2 * p->pw < w->Kw) return RT3D_ERR_SHAPE;
  if (int64_t(x->n) * x->t * x->h * x->w >= (int64_t(1) << 31)) return RT3D_ERR_UNSUPPORTED;
  g->n = x->n; g->t = x->t; g->h = x->h; g->w = x->w; g->c = x->c; g->xcs = x->c_stride;
  g->To = int(To); g->Ho = int(Ho); g->Wo = int(Wo); g->M = w->M; g->ycs = 0;
  g->Kt = w->Kt; g->Kh = w->Kh; g->Kw = w->Kw;
  g->st = p->st; g->sh = p->sh; g->sw = p->sw; g->pt = p->pt; g->ph = p->ph; g->pw = p->pw;
  g->relu = p->relu ? 1 : 0;
  if (y) {
    s = check_tensor(y);
    if (s != RT3D_OK) return s;
    if (y->n != x->n || y->t != To || y->h != Ho || y->w != Wo || y->c != w->M || y->dtype != w->dtype)
      return RT3D_ERR_SHAPE;
    g->ycs = y->c_stride;
  }
  return RT3D_OK;
}

// Alignment rules of the device entry points.
rt3d_status check_alignment(const rt3d_tensor* t) {
  const int mult = t->dtype == RT3D_BF16 ? 8 : 4;
  if (t->c_stride % mult) return RT3D_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(t->data) % 16) return RT3D_ERR_INVALID_ARG;
  return RT3D_OK;
}

bool overlaps(const rt3d_tensor* a, const rt3d_tensor* b) {
  const char* a0 = static_cast<const char*>(a->data);
  const char* b0 = static_cast<const char*>(b->data);
  return a0 < b0 + tensor_span_bytes(b) && b0 < a0 + tensor_span_bytes(a);
}

// ------------------------------------------------------------------------ prepared calls
// What a caller may ask about the last call, and what tests ask besides (rt3d_debug_get).
struct LastPlan {
  rt3d_plan_info info;
  int step_channels, turned;
  LastPlan(const rt3d_plan_info& i, int step = 0, int turn = 0) : info(i), step_channels(step), turned(turn) {}
};
thread_local LastPlan t_last_plan = rt3d_plan_info{-1, 0, 0, 0, 0};
std::atomic<int> g_plan_epoch{0};              // advanced by rt3d_debug_set: calls prepared before it are prepared again

}  // namespace

namespace rt3d {
// Everything that a convolution call's plan is determined by: no address, so that a call on buffers the handle has not seen is
// found like a repeated one.
struct CallKey {
  uint64_t w2;                                 // the second handle, by its id: its address may be another handle's later
  int32_t geo[24];                             // extents, pitches and dtypes of x, y and the residual
  int32_t p[20];                               // both convolutions' parameters
  int32_t misc[8];                             // device, entry point, fused pool, epoch, which of the two biases there are
};
// The memory that one call works on.
struct CallBuffers {
  const void* x;
  void* y;
  const void* res;
  const float *bias, *bias2;
};
// One call of a handle, ready to launch on any buffers: a user runs a layer on the same few shapes again and again, and
// choosing the kernel and encoding two or three tensor maps cost 1 to 2 us of the host's time for each call.
struct PreparedCall {
  CallKey key;
  LastPlan plan;
  std::function<cudaError_t(const CallBuffers&, cudaStream_t)> launch;
};
}  // namespace rt3d

namespace {

constexpr size_t kPreparedCalls = 8;           // per handle

void put_tensor(const rt3d_tensor* t, int32_t* at) {
  const int32_t v[8] = {1, t->n, t->t, t->h, t->w, t->c, t->c_stride, t->dtype};
  memcpy(at, v, sizeof(v));
}
void put_params(const rt3d_conv_params* p, int32_t* at) {
  const int32_t v[10] = {p->st, p->sh, p->sw, p->pt, p->ph, p->pw, p->relu, p->algo, p->x_pad_zero, p->concurrent};
  memcpy(at, v, sizeof(v));
}
// False for arguments that the call will refuse anyway, what depends on addresses (alignment, overlap) among them.
bool make_key(CallKey* k, const rt3d_tensor* x, const rt3d_packed* w, const float* bias, const rt3d_conv_params* p,
              const rt3d_tensor* y, const rt3d_tensor* res, int entry) {
  int dev = 0;
  if (!x || !w || !p || !y || check_tensor(x) != RT3D_OK || check_tensor(y) != RT3D_OK || (res && check_tensor(res) != RT3D_OK) ||
      check_alignment(x) != RT3D_OK || check_alignment(y) != RT3D_OK || (res && check_alignment(res) != RT3D_OK) ||
      overlaps(x, y) || (res && overlaps(res, y)) || cudaGetDevice(&dev) != cudaSuccess)
    return false;
  memset(k, 0, sizeof(*k));
  put_tensor(x, k->geo);
  put_tensor(y, k->geo + 8);
  if (res) put_tensor(res, k->geo + 16);
  put_params(p, k->p);
  k->misc[0] = dev; k->misc[1] = entry; k->misc[5] = g_plan_epoch.load(); k->misc[6] = bias != nullptr;
  return true;
}

// Tensor maps of a prepared call at the addresses of this one (nullptr: a map that the call has no use for).
struct PlacedMaps {
  CUtensorMap x, y;
  bool ok;
  PlacedMaps(const CUtensorMap& xmap, const void* xa, const CUtensorMap& ymap, void* ya) : x(xmap), y(ymap) {
    ok = (!xa || g_replace_address(&x, const_cast<void*>(xa)) == CUDA_SUCCESS) && (!ya || g_replace_address(&y, ya) == CUDA_SUCCESS);
  }
};

// Runs one call of a handle: from its prepared calls, or prepared now and kept.
class Submit {
 public:
  Submit(rt3d_packed* w, const CallKey& key, const CallBuffers& buffers, cudaStream_t st) : w_(w), key_(key), buffers_(buffers), st_(st) {}
  // true: the call was found and has been run (or only planned), with *status as its result
  bool again(rt3d_status* status) {
    std::shared_ptr<PreparedCall> c;
    {
      std::lock_guard<std::mutex> lock(w_->mu);
      for (const auto& e : w_->calls)
        if (memcmp(&e->key, &key_, sizeof(key_)) == 0) { c = e; break; }
    }
    if (!c) return false;
    *status = run(*c);
    return true;
  }
  bool keep = true;                            // whether the chosen launch is kept for later calls
  // Whether the call goes into a graph that is being captured: nothing can be allocated or uploaded then.
  bool captured() const {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    return !t_plan_only && st_ != nullptr && cudaStreamIsCapturing(st_, &status) == cudaSuccess && status != cudaStreamCaptureStatusNone;
  }
  // A kernel launch chosen for this call.  `launch` must hold by value whatever it needs besides the handle's own memory, and
  // take the addresses of the tensors and biases from its argument.
  rt3d_status operator()(const LastPlan& plan, std::function<cudaError_t(const CallBuffers&, cudaStream_t)> launch) {
    auto c = std::make_shared<PreparedCall>(PreparedCall{key_, plan, std::move(launch)});
    if (keep) {
      std::lock_guard<std::mutex> lock(w_->mu);
      if (w_->calls.size() < kPreparedCalls) w_->calls.push_back(c);
      else w_->calls[w_->next_call++ % kPreparedCalls] = c;
    }
    return run(*c);
  }

 private:
  rt3d_status run(const PreparedCall& c) {
    t_last_plan = c.plan;
    if (t_plan_only) return RT3D_OK;
    if (c.launch(buffers_, st_) != cudaSuccess) return RT3D_ERR_CUDA;
    g_launches.fetch_add(1);
    return RT3D_OK;
  }
  rt3d_packed* w_;
  const CallKey& key_;
  const CallBuffers buffers_;
  cudaStream_t st_;
};

// ------------------------------------------------------------------------- device blobs
DeviceBlob* find_blob(rt3d_packed* h, int dev) {
  for (DeviceBlob* b : h->blobs)
    if (b->device == dev) return b;
  return nullptr;
}

// Returns the blob of the current device, creating it on first use.
rt3d_status get_blob(rt3d_packed* h, DeviceBlob** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return RT3D_ERR_CUDA;
  std::lock_guard<std::mutex> lock(h->mu);
  DeviceBlob* b = find_blob(h, dev);
  if (!b) {
    std::unique_ptr<DeviceBlob> made(new DeviceBlob);
    made->device = dev;
    h->blobs.reserve(h->blobs.size() + 1);
    std::lock_guard<std::mutex> reg(g_blobs_mu);
    g_blobs.push_back(made.get());
    h->blobs.push_back(b = made.release());
  }
  *out = b;
  return RT3D_OK;
}

// Host arrays that become one device allocation: a cudaMalloc costs more than the copy of a small layer's index, so the
// arrays of a layout share one.  `add` remembers an array and the pointer that will refer to its device copy.
class Upload {
 public:
  template <typename T, typename V>
  void add(T** dst, const V& v) {
    const size_t bytes = v.size() * sizeof(*v.data());
    items_[n_++] = Item{reinterpret_cast<void**>(dst), v.data(), bytes, bytes_};
    bytes_ += (bytes + 16 + 255) & ~size_t(255);       // 256-byte aligned parts, readable 16 bytes on
  }
  // A part that is not copied to.
  template <typename T>
  void reserve(T** dst, size_t bytes) {
    items_[n_++] = Item{reinterpret_cast<void**>(dst), nullptr, 0, bytes_};
    bytes_ += (bytes + 16 + 255) & ~size_t(255);
  }
  // Allocates, copies and sets the pointers; *base owns the memory.  Nothing is kept on failure.  `wait`: returns when all of
  // it is on the device (a caller that goes on in the legacy stream and waits for that needs no wait here).
  rt3d_status run(void** base, bool wait = true) {
    if (weight_malloc(base, bytes_) != cudaSuccess) { *base = nullptr; return RT3D_ERR_ALLOC; }
    for (int i = 0; i < n_; ++i) {
      char* d = static_cast<char*>(*base) + items_[i].off;
      if (items_[i].bytes && cudaMemcpy(d, items_[i].src, items_[i].bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
        weight_free(*base, false);
        *base = nullptr;
        return RT3D_ERR_CUDA;
      }
      *items_[i].dst = d;
    }
    if (wait && uploads_done() != cudaSuccess) {
      weight_free(*base, false);
      *base = nullptr;
      return RT3D_ERR_CUDA;
    }
    return RT3D_OK;
  }

 private:
  struct Item { void** dst; const void* src; size_t bytes, off; };
  Item items_[12];
  int n_ = 0;
  size_t bytes_ = 0;
};

void add_canonical(rt3d_packed* h, DeviceBlob* b, Upload& up) {
  up.add(&b->group_ptr, h->group_ptr);
  up.add(&b->pos_idx, h->pos_idx);
  up.add(&b->tiles, h->tiles);
}

// Device copies of the canonical arrays: for the index-driven CUDA-core kernel, and to build the tensor-core layouts from.
rt3d_status get_canonical_locked(rt3d_packed* h, DeviceBlob* b) {
  if (b->canonical) return RT3D_OK;
  Upload up;
  add_canonical(h, b, up);
  return up.run(&b->canonical);
}
rt3d_status get_canonical(rt3d_packed* h, DeviceBlob* b) {
  std::lock_guard<std::mutex> lock(h->mu);
  return get_canonical_locked(h, b);
}

rt3d_status get_umma_blob(rt3d_packed* h, DeviceBlob* blob, const UmmaLayout* L, DeviceBlob::Umma** out) {
  std::lock_guard<std::mutex> lock(h->mu);
  DeviceBlob::Umma& u = blob->umma[umma_key(L->n_tile, L->t_groups, L->chunk != kChunk)];
  if (!u.ready) {
    const size_t wbytes = L->steps.size() * size_t(L->n_tile) * L->chunk * 2;
    // The canonical arrays go to the device once, a quarter to a third of the size of the zero-filled tiles, and a kernel
    // fills the tiles in there: 512 x 512 x 27 at 0.28 kept, 14 MB of tiles: 9 -> 1.6 ms with the allocation.
    // The first layout shares the allocation of the canonical arrays: a cudaMalloc and its cudaFree are 0.2 to 0.4 ms each.
    const bool shared = !blob->canonical;
    void** const base = shared ? &blob->canonical : &u.base;
    int32_t* slots = nullptr;
    Upload up;
    up.reserve(&u.wtiles, wbytes + 1024);
    if (shared) add_canonical(h, blob, up);
    up.add(&u.step_ptr, L->step_ptr);
    up.add(&u.steps, L->steps);
    up.add(&slots, L->slots);
    if (L->t_groups) { up.add(&u.grp_ptr, L->grp_ptr); up.add(&u.grp_first, L->grp_first); }
    const rt3d_status s = up.run(base, wbytes == 0);
    if (s != RT3D_OK) return s;
    const auto fail = [&] { weight_free(*base, false); *base = nullptr; return RT3D_ERR_CUDA; };
    if (wbytes && (launch_fill_umma_tiles(blob->group_ptr, blob->pos_idx, blob->tiles, slots, h->M, h->N, h->Ks, h->g_m, h->g_n,
                                          h->Q, h->P * h->Q, h->nnz, L->n_tile, L->chunk, L->n_chunks, u.wtiles, wbytes) != cudaSuccess ||
                   uploads_done() != cudaSuccess))
      return fail();
    // 2-D map over the weight tiles: rows of a chunk's channels, one box = one tile
    const cuuint64_t rows = L->steps.empty() ? cuuint64_t(L->n_tile) : cuuint64_t(L->steps.size()) * L->n_tile;
    const CUtensorMapSwizzle swizzle = L->chunk == kChunk ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    cuuint64_t dims[2] = {cuuint64_t(L->chunk), rows};
    cuuint64_t strides[1] = {cuuint64_t(L->chunk) * 2};
    cuuint32_t box[2] = {cuuint32_t(L->chunk), cuuint32_t(L->n_tile)};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(reinterpret_cast<CUtensorMap*>(u.wmap), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, u.wtiles, dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail();
    if (L->n_tile % 16 == 0) {
      cuuint32_t box_half[2] = {cuuint32_t(L->chunk), cuuint32_t(L->n_tile / 2)};
      r = g_encode(reinterpret_cast<CUtensorMap*>(u.wmap_half), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, u.wtiles, dims,
                   strides, box_half, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return fail();
    }
    u.ready = true;
  }
  *out = &u;
  return RT3D_OK;
}

bool umma_blob_ready(rt3d_packed* h, DeviceBlob* blob, int key) {
  std::lock_guard<std::mutex> lock(h->mu);
  const auto it = blob->umma.find(key);
  return it != blob->umma.end() && it->second.ready;
}

// A step-list layout that is on the device, the widest with whole pieces of 32 columns where there is one; nullptr: none.
const UmmaLayout* present_umma_layout(rt3d_packed* h, DeviceBlob* blob) {
  std::lock_guard<std::mutex> lock(h->mu);
  const UmmaLayout* best = nullptr;
  for (const auto& kv : blob->umma) {
    const auto it = h->umma_layouts.find(kv.first);
    if (!kv.second.ready || it == h->umma_layouts.end()) continue;
    const auto rank = [](const UmmaLayout& L) { return (L.n_tile % 32 == 0 ? 512 : 0) + L.n_tile; };
    if (!best || rank(it->second) > rank(*best)) best = &it->second;
  }
  return best;
}

// Whether a handle's layouts for the CUDA cores are on the device: the canonical arrays, the register-blocked kernel's.
bool canonical_ready(rt3d_packed* h, DeviceBlob* blob) {
  std::lock_guard<std::mutex> lock(h->mu);
  return blob->canonical != nullptr;
}
bool f32_blob_ready(rt3d_packed* h, DeviceBlob* blob) {
  std::lock_guard<std::mutex> lock(h->mu);
  return blob->f32.base != nullptr;
}

// Device copy of the fp32 tensor-core kernel's layout, with the canonical arrays beside it.
rt3d_status get_split_blob(rt3d_packed* h, DeviceBlob* blob, const UmmaLayout* L, bool pair, DeviceBlob::Umma** out) {
  std::lock_guard<std::mutex> lock(h->mu);
  DeviceBlob::Umma& u = blob->umma[umma_key(L->n_tile, false, false)];
  if (!u.ready) {
    const size_t wbytes = L->steps.size() * size_t(L->n_tile) * 192;
    const bool shared = !blob->canonical;
    void** const base = shared ? &blob->canonical : &u.base;
    int32_t* slots = nullptr;
    Upload up;
    up.reserve(&u.wtiles, wbytes + 1024);
    if (shared) add_canonical(h, blob, up);
    up.add(&u.step_ptr, L->step_ptr);
    up.add(&u.steps, L->steps);
    up.add(&slots, L->slots);
    const rt3d_status s = up.run(base, wbytes == 0);
    if (s != RT3D_OK) return s;
    const auto fail = [&] { weight_free(*base, false); *base = nullptr; return RT3D_ERR_CUDA; };
    if (wbytes && (launch_fill_split_tiles(blob->group_ptr, blob->pos_idx, static_cast<const float*>(blob->tiles), slots, h->M, h->N, h->Ks,
                                           h->g_m, h->g_n, h->Q, h->P * h->Q, h->nnz, L->n_tile, pair ? 2 : 1, L->n_chunks, u.wtiles, wbytes) != cudaSuccess ||
                   uploads_done() != cudaSuccess))
      return fail();
    u.ready = true;
  }
  *out = &u;
  return RT3D_OK;
}

// Device copy of the sub-tile kernel's layout (step records, step offsets, weight blocks).
rt3d_status get_sub_blob(rt3d_packed* h, DeviceBlob* blob, const SubLayout* L, DeviceBlob::Sub** out) {
  std::lock_guard<std::mutex> lock(h->mu);
  DeviceBlob::Sub& u = blob->sub[L->n_tile];
  if (!u.ready) {
    const size_t sbytes = L->steps.size() * sizeof(SubStep), bbytes = L->payload.size();
    if (dev_malloc(&u.steps, sbytes + 64) != cudaSuccess ||
        dev_malloc(&u.step_ptr, L->step_ptr.size() * 4) != cudaSuccess ||
        dev_malloc(&u.blocks, bbytes + 512) != cudaSuccess)
      return RT3D_ERR_ALLOC;
    if ((sbytes && cudaMemcpy(u.steps, L->steps.data(), sbytes, cudaMemcpyHostToDevice) != cudaSuccess) ||
        cudaMemcpy(u.step_ptr, L->step_ptr.data(), L->step_ptr.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        (bbytes && cudaMemcpy(u.blocks, L->payload.data(), bbytes, cudaMemcpyHostToDevice) != cudaSuccess) ||
        uploads_done() != cudaSuccess)
      return RT3D_ERR_CUDA;
    u.ready = true;
  }
  *out = &u;
  return RT3D_OK;
}

// ------------------------------------------------------------------------ tile planning
// Box of output voxels (bn x bt x bh x bw <= 128) that covers the output with the fewest tiles;
// ties go to the wider box along w, then h (longer contiguous runs for the TMA engine).
// `prefer_deep`: ties go first to boxes inside one clip, then to the deeper box along t (the t-grouped CTA-pair
// variant shares one staged input tile between the kt steps; the deeper the box, the less the extra frames weigh).
TileBox choose_box_search(const ConvGeom& g, bool prefer_deep);
// The search is a few thousand iterations; repeated calls on the same shape (every eager forward pass) take the
// answer from a small per-thread table.
TileBox choose_box(const ConvGeom& g, bool prefer_deep = false) {
  struct Entry { int n, To, Ho, Wo, st, sh, sw, deep; TileBox box; };
  thread_local Entry cache[16];
  thread_local int used = 0, next = 0;
  for (int i = 0; i < used; ++i) {
    const Entry& e = cache[i];
    if (e.n == g.n && e.To == g.To && e.Ho == g.Ho && e.Wo == g.Wo && e.st == g.st && e.sh == g.sh && e.sw == g.sw &&
        e.deep == int(prefer_deep))
      return e.box;
  }
  const TileBox box = choose_box_search(g, prefer_deep);
  cache[next] = Entry{g.n, g.To, g.Ho, g.Wo, g.st, g.sh, g.sw, int(prefer_deep), box};
  next = (next + 1) % 16;
  if (used < 16) ++used;
  return box;
}
TileBox choose_box_search(const ConvGeom& g, bool prefer_deep) {
  TileBox best{1, 1, 1, 1};
  long long best_tiles = -1;
  for (int bw = 1; bw <= g.Wo && bw <= kTileM; ++bw) {
    if (bw * g.sw > 256) break;
    for (int bh = 1; bh <= g.Ho && bw * bh <= kTileM; ++bh) {
      if (bh * g.sh > 256) break;
      for (int bt = 1; bt <= g.To && bw * bh * bt <= kTileM; ++bt) {
        if (bt * g.st > 256) break;
        int bn = kTileM / (bw * bh * bt);
        if (bn > g.n) bn = g.n;
        const long long tiles = (long long)ceil_div(g.n, bn) * ceil_div(g.To, bt) * ceil_div(g.Ho, bh) * ceil_div(g.Wo, bw);
        bool better = best_tiles < 0 || tiles < best_tiles;
        if (!better && tiles == best_tiles && prefer_deep && ((bn == 1) != (best.bn == 1) || bt != best.bt)) {
          better = (bn == 1) != (best.bn == 1) ? bn == 1 : bt > best.bt;
        } else if (!better && tiles == best_tiles) {
          if (bw > best.bw) better = true;
          else if (bw == best.bw && bh > best.bh) better = true;
        }
        if (better) { best = TileBox{bn, bt, bh, bw}; best_tiles = tiles; }
      }
    }
  }
  return best;
}

// Box inside one clip for the t-grouped variant where none of the boxes with the fewest tiles suits it: up to a sixteenth
// more tiles, the fewest bytes from L2 (a group's input frames and its Kt weight tiles) over all tiles.  Returns their ratio to
// what the fewest tiles with a box per step read; it is taken up to 0.8, for strided rows, where the larger boxes take the
// copy engine longer, up to 0.68 (0.65 gained 15 % there, 0.71 lost 8 %), and up to 0.6 where it costs the bulk stores.  21 -> 33 channels 3x3x3 on 2 x 10 x 43 x 39 voxels, 286 tiles 10 frames
// deep for 275 tiles of two clips: 37.4 -> 17.8 us; 17 -> 49 on 2 x 5 x 52 x 87 49.4 -> 24.2; 31 -> 238 on 23 x 7 x 37 x 83
// 350 -> 275; 87 -> 154 on 6 x 12 x 90 x 17 147 -> 103.
double choose_box_grouped(const ConvGeom& g, int n_tile, long long fewest, TileBox* out) {
  double best = -1.0;
  for (int bt = 2; bt <= g.To && bt <= kTileM && bt * g.st <= 256; ++bt)
    for (int bh = 1; bh <= g.Ho && bt * bh <= kTileM && bh * g.sh <= 256; ++bh) {
      int bw = kTileM / (bt * bh);
      if (bw > g.Wo) bw = g.Wo;
      if (bw * g.sw > 256) continue;
      bw = ceil_div(g.Wo, ceil_div(g.Wo, bw));              // no wider than the columns need
      const long long tiles = (long long)g.n * ceil_div(g.To, bt) * ceil_div(g.Ho, bh) * ceil_div(g.Wo, bw);
      if (tiles * 16 > fewest * 17) continue;
      const double cost = double(tiles) * (double(bt + g.Kt - 1) * bh * bw + g.Kt * 0.5 * n_tile);
      if (best < 0 || cost < best) { best = cost; *out = TileBox{1, bt, bh, bw}; }
    }
  return best >= 0 ? best / (double(fewest) * g.Kt * (kTileM + 0.5 * n_tile)) : 2.0;
}

// Bundle width, number of K splits and kernel (single CTAs or CTA pairs) for a call.  Model, fitted to timings on B200:
//  - A K step takes its tensor time or the time its operands need from L2, 65 bytes per clock and SM whatever the kernel
//    (at 128 columns 32 KB for a CTA, 24 KB for one of a pair, 14 KB where the kt steps share an input tile): this bounds
//    nearly every layer with few tiles.
//  - A launch has 5 us around its steps, one of CTA pairs 6.9 us (cluster set-up, its tables).
//  - A split costs the shares' way through shared memory and the wait for a cluster's SMs, growing with its size.
// Measured against it: 128 -> 256 at 8 x 28 x 28 (49 tiles, 54 steps) single 18.5 us, pairs 16.0 us; 256 -> 512 at 4 x 14 x 14
// (7 tiles, 108 steps) S = 4: 14.5 us, pairs 19 us; 512 -> 1152 1x3x3 at 8 x 2 x 7 x 7: 192 columns S = 3 16.5 us, 64 columns
// unsplit 21.8 us.  The step count of each candidate width comes from the handle's real step lists where kernel groups
// are tall enough for whole steps to vanish; a narrower bundle that matches the group height can win there.
struct UmmaPlan { int n_tile, n_splits; bool pair; };

// Whether the step-list kernels take a layer in steps of 32 input channels, half the bytes, MMAs and weights of one of 64: layers
// of up to 32.  19 -> 489 channels 3x3x3 on 12 x 6 x 111 x 11 198 -> 120 us, 21 -> 164 on 18 x 16 x 75 x 15 152 -> 114, 17 -> 196 on
// 3 x 3 x 63 x 44 38 -> 26, single steps and small calls 1.0-1.1x.  With more channels, where three steps of 32 would replace two
// of 64, they lose: the copy engine takes rows at a rate, not bytes (77 -> 186 28.4 -> 31.7, 470 -> 182 33 -> 46, 265 -> 511 51 -> 63).
bool narrow_steps(const rt3d_packed* w) { return w->N <= kNarrowChunk && g_narrow_enabled.load(); }

UmmaPlan pick_plan(rt3d_packed* w, const ConvGeom& g, long long m_tiles, int sm_count, bool narrow) {
  const int M = w->M;
  // Of a full step's bytes and MMAs; its hand-shake is the same.  (With few steps the output counts, and a bundle is no wider for
  // it: 24 -> 347 1x3x3 on 14 x 4 x 7 x 7 at 64 columns 6.3 us, at 176 7.6.)
  const double part = narrow && w->Ks > 12 ? 0.5 : 1.0;
  const int widest = default_n_tile(M);
  const bool tall = w->g_m >= 16 && !w->is_dense;
  UmmaPlan best{widest, 1, false};
  double best_ns = -1.0;
  int last = 0;
  for (int b = ceil_div(M, widest);; ++b) {
    // widths that cut M evenly, in whole 32-column pieces below the widest (odd ones for splits only: a layer with enough
    // tiles takes the widest); tall groups: halves, which match their heights
    int n = tall ? (b == ceil_div(M, widest) ? widest : last > 128 ? 128 : last / 2) : round_up(ceil_div(M, b), b == ceil_div(M, widest) ? 16 : 32);
    if (last && (n >= last || n < 32)) {
      if (n < 32 || n <= 32) break;
      continue;
    }
    last = n;
    if (n % 16) break;
    const int bundles = ceil_div(M, n);
    if (n != widest && !tall && n != 128 && n != 64 && bundles * n * 14 > round_up(M, 16) * 15) continue;   // padding columns
    const long long items = m_tiles * bundles;
    double steps = double(w->Ks) * ceil_div(w->N, kChunk);      // full lists: true for groups a few rows high
    if (tall) {
      const UmmaLayout* L = get_umma_layout(w, n);
      if (!L) break;
      steps = items < sm_count ? double(L->max_steps) : double(L->steps.size()) / bundles;
    }
    constexpr double kByteNs = 1.0 / (65.0 * 1.85);
    const double step_ns = std::max({part * 1.08 * n, part * (kTileM * 128.0 + 128.0 * n) * kByteNs, 204.0});
    for (int S = 1; S <= 8; ++S) {
      const int capacity = umma_split_capacity(S, sm_count);
      if (capacity == 0 || (S > 1 && (steps / S < 4 || items >= 2LL * sm_count))) continue;
      if (S == 1 && n != widest && (n & (n - 1))) continue;
      const double waves = double(ceil_div64(items * S, capacity));
      const double ns = S == 1 ? 5000.0 + waves * steps * step_ns : waves * (7100.0 + 0.32 * n * S * S + steps / S * step_ns);
      if (best_ns < 0 || ns < best_ns * 0.98) { best = UmmaPlan{n, S, false}; best_ns = ns; }
    }
    if (umma_pair_supported(n, bundles) && (n == widest || (n & (n - 1)) == 0)) {
      const bool ts = g.Kt >= 2 && g.Kt <= 8 && g.st == 1 && g.To >= 4 && (n <= 128 || g.Kh * g.Kw >= 4);
      const double a_bytes = kTileM * 128.0 * (ts ? 1.25 / g.Kt : 1.0);
      const double pair_ns = std::max({part * (n <= 128 ? 1.3 : 1.1) * n, part * (a_bytes + 64.0 * n) * kByteNs, 165.0});
      // a last round that is not full is shared out along K where the items are long enough
      const double rounds = double((m_tiles + 1) / 2 * bundles) / (sm_count / 2);
      const double whole = std::ceil(rounds) * steps * pair_ns, shared = 5000.0 + rounds * steps * pair_ns;
      const double ns = 6900.0 + (rounds <= 1.0 || whole < shared ? whole : shared);
      if (ns < best_ns * 0.97) { best = UmmaPlan{n, 1, true}; best_ns = ns; }
    }
    if (n == 32) break;
  }
  return best;
}

bool umma_eligible(const DeviceState* d, const rt3d_packed* w, const rt3d_tensor* x, const rt3d_tensor* y,
                   const rt3d_conv_params* p) {
  if (d->cc_major != 10) return false;
  if (!umma_layout_possible(w)) return false;
  if (x->c_stride % 8 || y->c_stride % 8) return false;
  if (p->st > 8 || p->sh > 8 || p->sw > 8) return false;
  if (int64_t(x->w) * x->c_stride * 2 >= (int64_t(1) << 40)) return false;
  return true;
}

// `extra_t`: frames added to the box along t (the t-grouped CTA-pair variant stages Kt - 1 more; temporal stride 1).
rt3d_status encode_xmap(const rt3d_tensor* x, const ConvGeom& g, const TileBox& box, CUtensorMap* map, int extra_t = 0, int chunk = kChunk) {
  const cuuint64_t cs = cuuint64_t(x->c_stride) * 2;
  cuuint64_t dims[5] = {cuuint64_t(x->c), cuuint64_t(x->w), cuuint64_t(x->h), cuuint64_t(x->t), cuuint64_t(x->n)};
  cuuint64_t strides[4] = {cs, cs * x->w, cs * x->w * x->h, cs * x->w * x->h * x->t};
  // with a traversal stride s the engine loads ceil(box / s) elements, so a box of b outputs spans b*s inputs
  cuuint32_t bx[5] = {cuuint32_t(chunk), cuuint32_t(box.bw * g.sw), cuuint32_t(box.bh * g.sh), cuuint32_t(box.bt * g.st + extra_t),
                      cuuint32_t(box.bn)};
  cuuint32_t estr[5] = {1, cuuint32_t(g.sw), cuuint32_t(g.sh), cuuint32_t(g.st), 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, x->data, dims, strides, bx, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, chunk == kChunk ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? RT3D_OK : RT3D_ERR_CUDA;
}

// Block of 32 output voxels (w, h, t, n extents) that one epilogue warp owns in a box of bw x bh x bt x bn
// voxels; false when 32 consecutive box rows are not a rectangular block.
bool warp_block(int bw, int bh, int bt, int bn, int sb[4]) {
  if ((bw * bh * bt * bn) % 32) return false;
  int rem = 32;
  const int dims_box[4] = {bw, bh, bt, bn};
  for (int i = 0; i < 4; ++i) {
    sb[i] = 1;
    if (rem == 1) continue;
    const int d = dims_box[i];
    if (d >= rem) { if (d % rem) return false; sb[i] = rem; rem = 1; }
    else { if (rem % d) return false; sb[i] = d; rem /= d; }
  }
  return rem == 1;
}

// Output tensor map for the TMA-store epilogue: box = 32 channels x the voxels one epilogue warp stores per
// piece (its block of 32 voxels, divided by the fused pooling window), 64-byte swizzle.  The tensor is y,
// i.e. already the pooled one when pooling is fused.
bool encode_ymap(const rt3d_tensor* y, const int sb[4], int pw, int ph, int pt, CUtensorMap* map) {
  if (y->c < 32 || sb[0] % pw || sb[1] % ph || sb[2] % pt) return false;
  const cuuint64_t cs = cuuint64_t(y->c_stride) * 2;
  cuuint64_t dims[5] = {cuuint64_t(y->c), cuuint64_t(y->w), cuuint64_t(y->h), cuuint64_t(y->t), cuuint64_t(y->n)};
  cuuint64_t strides[4] = {cs, cs * y->w, cs * y->w * y->h, cs * y->w * y->h * y->t};
  cuuint32_t bx[5] = {32, cuuint32_t(sb[0] / pw), cuuint32_t(sb[1] / ph), cuuint32_t(sb[2] / pt), cuuint32_t(sb[3])};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, y->data, dims, strides, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Box for a call with fused pooling: fewest tiles among the boxes whose extents and whose per-warp block
// are multiples of the pooling window (every window then lies inside one warp's 32 voxels).
bool choose_box_pool_search(const ConvGeom& g, int pw, int ph, int pt, TileBox* out, int sb_out[4], bool prefer_deep);
bool choose_box_pool(const ConvGeom& g, int pw, int ph, int pt, TileBox* out, int sb_out[4], bool prefer_deep = false) {
  struct Entry { int n, To, Ho, Wo, st, sh, sw, pw, ph, pt, deep; bool ok; TileBox box; int sb[4]; };   // as in choose_box
  thread_local Entry cache[16];
  thread_local int used = 0, next = 0;
  for (int i = 0; i < used; ++i) {
    const Entry& e = cache[i];
    if (e.n == g.n && e.To == g.To && e.Ho == g.Ho && e.Wo == g.Wo && e.st == g.st && e.sh == g.sh && e.sw == g.sw &&
        e.pw == pw && e.ph == ph && e.pt == pt && e.deep == int(prefer_deep)) {
      if (e.ok) { *out = e.box; for (int k = 0; k < 4; ++k) sb_out[k] = e.sb[k]; }
      return e.ok;
    }
  }
  Entry e{g.n, g.To, g.Ho, g.Wo, g.st, g.sh, g.sw, pw, ph, pt, int(prefer_deep), false, TileBox{1, 1, 1, 1}, {1, 1, 1, 1}};
  e.ok = choose_box_pool_search(g, pw, ph, pt, &e.box, e.sb, prefer_deep);
  cache[next] = e;
  next = (next + 1) % 16;
  if (used < 16) ++used;
  if (e.ok) { *out = e.box; for (int k = 0; k < 4; ++k) sb_out[k] = e.sb[k]; }
  return e.ok;
}
bool choose_box_pool_search(const ConvGeom& g, int pw, int ph, int pt, TileBox* out, int sb_out[4], bool prefer_deep) {
  long long best_tiles = -1;
  for (int bw = pw; bw <= kTileM && bw <= round_up(g.Wo, pw); bw += pw) {
    if (bw * g.sw > 256) break;
    for (int bh = ph; bw * bh <= kTileM && bh <= round_up(g.Ho, ph); bh += ph) {
      if (bh * g.sh > 256) break;
      for (int bt = pt; bw * bh * bt <= kTileM && bt <= round_up(g.To, pt); bt += pt) {
        if (bt * g.st > 256) break;
        int bn = kTileM / (bw * bh * bt);
        if (bn > g.n) bn = g.n;
        int sb[4];
        if (!warp_block(bw, bh, bt, bn, sb) || sb[0] % pw || sb[1] % ph || sb[2] % pt) continue;
        const long long tiles = (long long)ceil_div(g.n, bn) * ceil_div(g.To, bt) * ceil_div(g.Ho, bh) * ceil_div(g.Wo, bw);
        bool better = best_tiles < 0 || tiles < best_tiles;
        if (!better && tiles == best_tiles) {
          if (prefer_deep && ((bn == 1) != (out->bn == 1) || bt != out->bt)) better = (bn == 1) != (out->bn == 1) ? bn == 1 : bt > out->bt;
          else better = bw > out->bw;
        }
        if (better) {
          best_tiles = tiles;
          *out = TileBox{bn, bt, bh, bw};
          for (int i = 0; i < 4; ++i) sb_out[i] = sb[i];
        }
      }
    }
  }
  return best_tiles > 0;
}

// Small-C_in kernel: bf16, C_in <= 8 stored at pitch 8, spatial strides <= 4, M <= 256.
bool smallc_eligible(const DeviceState* d, rt3d_packed* w, const rt3d_tensor* x, const rt3d_tensor* y,
                     const rt3d_conv_params* p, const SmallCLayout** out) {
  if (d->cc_major != 10 || w->dtype != RT3D_BF16) return false;
  if (x->c > 8 || x->c_stride != 8 || y->c_stride % 8) return false;
  if (p->st > 8 || p->sh > 4 || p->sw > 4) return false;
  if (w->Kt > 16 || w->Kh > 32 || w->Kw > 32) return false;
  const SmallCLayout* L = get_smallc_layout(w, p->sh, p->sw);
  if (!L) return false;
  const SmallCLayout* P = get_smallc_layout(w, p->sh, p->sw, true);
  if (P && P->n_pairs < L->n_pairs && smallc_smem_bytes(P->n_pairs, P->n_pad, P->phase_stride, int(P->ops.size())) <= 227 * 1024) {
    *out = P;
    return true;
  }
  if (L->img_w * p->sw > 256 || L->img_h * p->sh > 256) return false;
  if (smallc_smem_bytes(L->n_pairs, L->n_pad, L->n_phases * L->phase_stride) > 227 * 1024) return false;
  *out = L;
  return true;
}

rt3d_status launch_smallc(rt3d_packed* w, DeviceBlob* blob, const DeviceState* d, const SmallCLayout* L,
                          const rt3d_tensor* x, const ConvGeom& g, const float* bias, rt3d_tensor* y, Submit& submit,
                          const void* residual, int rcs, int pool_h, int pool_w, bool x_pad_zero) {
  // pooled rows leave as whole 32-channel pieces through the bulk-store epilogue; a trailing 16-channel piece is
  // written by plain per-voxel stores, which know nothing of pooling
  if (pool_h * pool_w > 1 && L->n_pad % 32) return RT3D_ERR_UNSUPPORTED;
  DeviceBlob::SmallC* sc = nullptr;
  {
    std::lock_guard<std::mutex> lock(w->mu);
    sc = &blob->smallc[L->sh * 16 + L->sw + (L->packed ? 1024 : 0)];
    if (!sc->base) {
      Upload up;
      up.add(&sc->wimg, L->wimg);
      up.add(&sc->pairs, L->pair_off);
      up.add(&sc->ops, L->ops);
      const rt3d_status s = up.run(&sc->base);
      if (s != RT3D_OK) return s;
    }
  }
  SmallCArgs a;
  a.g = g;
  a.n_pad = L->n_pad; a.n_pairs = L->n_pairs;
  a.n_phases = L->n_phases; a.phase_stride = L->phase_stride;
  a.img_w = L->img_w; a.phase_bytes = L->img_w * L->img_h * L->img_t * 16;
  a.tiles_h = ceil_div(g.Ho, kSmallCTileH); a.tiles_w = ceil_div(g.Wo, kSmallCTileW);
  a.tmem_cols = 0;
  a.residual = residual; a.rcs = rcs;
  a.pool_t = 1; a.pool_h = pool_h; a.pool_w = pool_w;
  a.wimg = sc->wimg; a.pair_off = sc->pairs;
  a.ops = L->packed ? sc->ops : nullptr; a.n_ops = int(L->ops.size()); a.img_h = L->img_h; a.x = x->data;
  a.bias = bias; a.y = y->data; a.sched = d->sched;
  // input as [n][t][h][w][8]: one box = one phase image of a 1 x 16 x 8 output tile (every sh-th row and
  // sw-th column: a traversal stride s loads ceil(box / s) elements), no swizzle
  CUtensorMap xmap;
  const cuuint64_t cs = 16;
  cuuint64_t dims[5] = {cuuint64_t(x->c), cuuint64_t(x->w), cuuint64_t(x->h), cuuint64_t(x->t), cuuint64_t(x->n)};
  cuuint64_t strides[4] = {cs, cs * x->w, cs * x->w * x->h, cs * x->w * x->h * x->t};
  cuuint32_t bx[5] = {8, cuuint32_t(L->img_w * g.sw), cuuint32_t(L->img_h * g.sh), cuuint32_t(L->img_t), 1};
  cuuint32_t estr[5] = {1, cuuint32_t(g.sw), cuuint32_t(g.sh), 1, 1};
  // Unit column stride and all 8 channels real (or the caller vouches for zero padding channels): merge the (w, channel) axes, so that the engine fetches each
  // image row as one contiguous run instead of one 16-byte request per voxel (the tile load was the
  // kernel's bottleneck).  Otherwise the separate channel axis stays: its out-of-range
  // fill is what zeroes the padding channels, whatever the caller's buffer holds there.
  a.merged_cw = (!L->packed && g.sw == 1 && (x->c == 8 || x_pad_zero) && L->img_w * 8 <= 256) ? 1 : 0;
  if (a.merged_cw) {
    dims[0] = cuuint64_t(x->w) * 8; dims[1] = 1;
    strides[0] = cs;                                   // the unit axis never moves
    bx[0] = cuuint32_t(L->img_w * 8); bx[1] = 1;
    estr[1] = 1;
  }
  memset(&xmap, 0, sizeof(xmap));
  if (!L->packed &&
      g_encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, x->data, dims, strides, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return RT3D_ERR_CUDA;
  CUtensorMap ymap{};
  const int sb[4] = {kSmallCTileW, 4, 1, 1};          // a warp owns 4 rows of 8 voxels of the 16 x 8 tile
  a.store_tma = encode_ymap(y, sb, pool_w, pool_h, 1, &ymap) ? 1 : 0;
  if (!a.store_tma && pool_h * pool_w > 1) return RT3D_ERR_UNSUPPORTED;
  const int sms = d->sm_count;
  return submit(rt3d_plan_info{3, L->n_pad, 1, 0, pool_h * pool_w > 1 ? 1 : 0}, [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, a.ops ? nullptr : c.x, ymap, a.store_tma ? c.y : nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    SmallCArgs now = a;
    now.x = c.x; now.y = c.y; now.bias = c.bias; now.residual = c.res;
    return launch_conv_umma_smallc(now, &m.x, a.store_tma ? &m.y : nullptr, sms, st);
  });
}

// The handle's tail-split scratch on this device: at least `bytes` of partial tiles and `flag_bytes` of flags, which every
// kernel that uses them leaves zeroed.  A larger one is at least twice the last, so that all of them take at most twice the
// largest; none moves or goes before the handle does.
rt3d_status get_tail(rt3d_packed* w, DeviceBlob* blob, size_t bytes, size_t flag_bytes, DeviceBlob::Tail* out) {
  std::lock_guard<std::mutex> lock(w->mu);
  if (blob->tails.empty() || blob->tails.back().bytes < bytes || blob->tails.back().flag_bytes < flag_bytes) {
    DeviceBlob::Tail t;
    if (!blob->tails.empty()) { t.bytes = 2 * blob->tails.back().bytes; t.flag_bytes = 2 * blob->tails.back().flag_bytes; }
    t.bytes = std::max(t.bytes, bytes);
    t.flag_bytes = std::max(t.flag_bytes, flag_bytes);
    std::lock_guard<std::mutex> reg(g_blobs_mu);               // others walk the lists of all handles
    blob->tails.reserve(blob->tails.size() + 1);
    if (dev_malloc(&t.partial, t.bytes) != cudaSuccess) return RT3D_ERR_ALLOC;
    if (dev_malloc(&t.flags, t.flag_bytes) != cudaSuccess) { cudaFree(t.partial); return RT3D_ERR_ALLOC; }
    if (cudaMemset(t.flags, 0, t.flag_bytes) != cudaSuccess || uploads_done() != cudaSuccess) {
      cudaFree(t.partial); cudaFree(t.flags);
      return RT3D_ERR_CUDA;
    }
    blob->tails.push_back(t);
  }
  *out = blob->tails.back();
  return RT3D_OK;
}

// Whether the epilogue's pieces are turned in shared memory (umma_common.cuh: epilogue_row_turned): those that load a residual
// and those that box stores cannot take.  Measured over 110 random layers, in favour of turning: with a residual, 1.05-1.57x
// from 64 columns on (24 -> 466 channels 3x1x1 on 19 x 8 x 46 x 13 126 -> 80 us), 0.86-1.19x below (30 -> 20 14.8 -> 17.3); without one
// 1.04-1.2x from 64 columns and nine steps on (110 -> 138 1x3x3 on 7 x 12 x 29 x 88 86 -> 71), 0.78-0.94x below (58 -> 18 3x1x1
// 14.8 -> 19.0, 150 -> 398 in three steps 40 -> 45), where a tile waits for its last piece.
bool turn_pieces(int n_tile, int steps, bool box_stores, bool residual) {
  return n_tile >= 64 && (residual || (!box_stores && steps >= 9));
}

// Resident-weight kernel for thin stride-1 layers: used when the layer qualifies and (unless forced) has
// at least one tile per SM.  *launched = false (and RT3D_OK) when the caller should take another kernel.
rt3d_status try_halo(rt3d_packed* w, DeviceBlob* blob, DeviceState* d, const rt3d_tensor* x, const ConvGeom& g,
                     const float* bias, rt3d_tensor* y, const void* res_data, int res_pitch, bool dense_entry,
                     bool forced, Submit& submit, bool* launched) {
  *launched = false;
  if (g.st != 1 || g.sh != 1 || g.sw != 1 || w->M > 256) return RT3D_OK;
  const int n_tile = round_up(w->M, 16);
  const int n_chunks = ceil_div(w->N, kChunk);
  // cheap size screen before the layout is built: all locations kept is the upper bound
  if (!dense_entry && w->is_dense == 0 && size_t(w->Ks) * n_chunks * (n_tile / 2) * 128 > size_t(4) * 227 * 1024) return RT3D_OK;
  HaloArgs h;
  UmmaArgs& a = h.u;
  a.g = g;
  // tile: 8 voxels along w times 16 (t, h) lines; one frame thick unless the kernel is 1 high
  int bt = 1, bh = 16;
  if (g.Kh == 1) {
    long long best = -1;
    for (int t = 1; t <= 16; t *= 2) {
      const int hh = 16 / t;
      const long long cost = (long long)ceil_div(g.To, t) * ceil_div(g.Ho, hh) * (t + g.Kt - 1) * hh;
      if (best < 0 || cost < best) { best = cost; bt = t; bh = hh; }
    }
  }
  a.box = TileBox{1, bt, bh, 8};
  a.tiles_n = g.n; a.tiles_t = ceil_div(g.To, bt); a.tiles_h = ceil_div(g.Ho, bh); a.tiles_w = ceil_div(g.Wo, 8);
  const long long m_tiles = (long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w;
  if (!forced && m_tiles < d->sm_count) return RT3D_OK;
  if (m_tiles > (1ll << 30)) return RT3D_OK;
  const UmmaLayout* L = get_umma_layout(w, n_tile);
  if (!L || L->n_bundles != 1) return RT3D_OK;
  a.n_tile = L->n_tile; a.n_bundles = 1; a.n_chunks = L->n_chunks;
  a.dense = dense_entry ? 1 : 0;
  a.steps_dense = w->Ks * L->n_chunks;
  h.n_steps = dense_entry ? a.steps_dense : L->step_ptr[1];
  if (!umma_halo_plan(&h, dense_entry ? nullptr : L->steps.data())) return RT3D_OK;
  // waste of the fixed 16 x 8 tile against the free-form boxes of the other kernels
  if (!forced && m_tiles * 128 > 3 * ((long long)g.n * g.To * g.Ho * g.Wo) / 2) return RT3D_OK;
  DeviceBlob::Umma* u = nullptr;
  rt3d_status s = get_umma_blob(w, blob, L, &u);
  if (s != RT3D_OK) return s;
  a.step_ptr = u->step_ptr; a.steps = u->steps;
  a.bias = bias; a.y = y->data; a.sched = d->sched;
  a.residual = res_data; a.rcs = res_pitch;
  a.pool_t = a.pool_h = a.pool_w = 1;
  a.n_splits = 1;
  a.tail_workers = 0; a.tail_scratch = nullptr; a.tail_flags = nullptr;
  a.ts = 0; a.grp_ptr = nullptr; a.grp_first = nullptr; a.ts_a_bytes = 0; a.ts_frame_bytes = 0; a.ts_table = 0; a.ts_phases = 1;
  a.wait_cycles = 0; a.debug_drop_last_load = 0;
  ConvGeom unit = g;                       // the staged block is a plain box of input voxels
  CUtensorMap xmap, ymap{};
  if ((s = encode_xmap(x, unit, TileBox{1, h.ht, h.hh, h.hw}, &xmap)) != RT3D_OK) return s;
  int sb[4] = {1, 1, 1, 1};
  const bool rect = warp_block(a.box.bw, a.box.bh, a.box.bt, a.box.bn, sb);
  a.sbw = sb[0]; a.sbh = sb[1];
  a.store_tma = (rect && encode_ymap(y, sb, 1, 1, 1, &ymap)) ? 1 : 0;
  a.turned = turn_pieces(a.n_tile, h.n_steps, a.store_tma != 0, res_data != nullptr) ? 1 : 0;
  a.narrow = 0;
  *launched = true;
  const int sms = d->sm_count;
  const void* wmap = u->wmap_half;
  return submit(LastPlan({4, a.n_tile, 1, 0, 0}, kChunk, a.turned), [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, c.x, ymap, h.u.store_tma ? c.y : nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    HaloArgs now = h;
    now.u.y = c.y; now.u.bias = c.bias; now.u.residual = c.res;
    return launch_conv_umma_halo(now, &m.x, wmap, h.u.store_tma ? &m.y : nullptr, sms, st);
  });
}

// Sub-tile kernel: blocks of 16 x 16 channels in which no kernel group keeps the step's location are skipped.
// Runs only when asked for (RT3D_ALGO_UMMA_SUB): measured on B200 it loses to the masked-dense CTA-pair kernel at
// every group size and pruning rate of the sweep, because moving a step's input tile through shared memory into
// tensor memory costs about as much as the dense MMAs of that step.
// *launched = false (and RT3D_OK) when the handle cannot use it.
rt3d_status try_sub(rt3d_packed* w, DeviceBlob* blob, DeviceState* d, const rt3d_tensor* x, const ConvGeom& g,
                    const float* bias, rt3d_tensor* y, const void* res_data, int res_pitch, Submit& submit, bool* launched) {
  *launched = false;
  if (w->is_dense) return RT3D_OK;
  SubArgs a;
  a.g = g;
  a.box = choose_box(g);
  a.tiles_n = ceil_div(g.n, a.box.bn); a.tiles_t = ceil_div(g.To, a.box.bt);
  a.tiles_h = ceil_div(g.Ho, a.box.bh); a.tiles_w = ceil_div(g.Wo, a.box.bw);
  const long long m_tiles = (long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w;
  if (m_tiles > (1ll << 30)) return RT3D_OK;
  const SubLayout* L = get_sub_layout(w, 0);
  if (!L) return RT3D_OK;
  a.n_tile = L->n_tile; a.n_bundles = L->n_bundles;
  if (!umma_sub_plan(&a, L->max_blocks)) return RT3D_OK;
  DeviceBlob::Sub* u = nullptr;
  rt3d_status s = get_sub_blob(w, blob, L, &u);
  if (s != RT3D_OK) return s;
  a.steps = static_cast<const SubStep*>(u->steps); a.step_ptr = u->step_ptr; a.blocks = u->blocks;
  a.bias = bias; a.y = y->data; a.sched = d->sched;
  a.residual = res_data; a.rcs = res_pitch;
  CUtensorMap xmap, ymap{};
  if ((s = encode_xmap(x, g, a.box, &xmap)) != RT3D_OK) return s;
  int sb[4] = {1, 1, 1, 1};
  const bool rect = warp_block(a.box.bw, a.box.bh, a.box.bt, a.box.bn, sb);
  a.store_tma = (rect && encode_ymap(y, sb, 1, 1, 1, &ymap)) ? 1 : 0;
  *launched = true;
  const int sms = d->sm_count;
  return submit(rt3d_plan_info{6, a.n_tile, 1, 0, 0}, [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, c.x, ymap, a.store_tma ? c.y : nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    SubArgs now = a;
    now.y = c.y; now.bias = c.bias; now.residual = c.res;
    return launch_conv_umma_sub(now, &m.x, a.store_tma ? &m.y : nullptr, sms, st);
  });
}

// Device copy of the register-blocked fp32 kernel's layout.
rt3d_status get_f32_blob(rt3d_packed* h, DeviceBlob* blob, const F32Layout* L, DeviceBlob::F32** out) {
  std::lock_guard<std::mutex> lock(h->mu);
  DeviceBlob::F32& u = blob->f32;
  if (!u.base) {
    Upload up;
    up.add(&u.entry_ptr, L->entry_ptr);
    up.add(&u.tile_ptr, L->tile_ptr);
    up.add(&u.counts, L->counts);
    up.add(&u.entries, L->entries);
    up.add(&u.tiles, L->tiles);
    const rt3d_status s = up.run(&u.base);
    if (s != RT3D_OK) return s;
  }
  *out = &u;
  return RT3D_OK;
}

// Up to 16 input channels half of every step is empty, and the CUDA cores skip what is pruned: only unpruned layers of more than 32
// outputs go to the tensor cores.  Over 130 random layers of 8 to 16 channels, of those that split_is_faster would send: unpruned
// ones of more than 32 outputs 1.02 to 3.5 times faster there (15 -> 118 3x3x3 on 3 x 12 x 56 x 31 77.6 -> 23.7 us), of up to 32
// 0.74 to 1.6, pruned ones 0.89 to 1.5.
bool split_fills_steps(const rt3d_packed* w) { return w->N > 16 || (w->M > 32 && w->nnz == int64_t(w->P) * w->Q * w->Ks); }

// What a drain warp does again for a tile whose rows are all infinite or NaN, while the other roles wait for it: for every four
// output channels (fewer where a kernel group ends), every entry that their groups may have, four input channels at a time.
// Handles with more than kSplitAgain stay on the CUDA cores.  606 -> 128 channels 3x3x3 at 1 x 1 groups, 0.9 kept, just below it:
// 361 ms for a tile of NaNs, a sixth of what the waits allow (4 x 4 groups never come near: 59 ms at 1212 channels).
constexpr int64_t kSplitAgain = 1 << 20;
int64_t split_again(const rt3d_packed* w) {
  const int64_t passes = w->g_m % 4 == 0 ? 16 : w->g_m == 1 ? 64 : 32;       // over a warp's columns, at most 64
  return passes * w->Q * w->Ks * ceil_div(w->g_n, 4);
}
bool split_rows_bounded(const rt3d_packed* w) { return split_again(w) <= kSplitAgain && int64_t(w->Ks) * w->N <= 32768; }

// Bundle width there: as few bundles of up to 128 channels as there can be.
int split_n_tile(int M) { return round_up(ceil_div(M, ceil_div(M, 128)), 16); }

// Whether an fp32 call is expected to take less time on the tensor cores than on the CUDA cores.  Both models are fitted to 92
// random layers (8-160 input and 16-160 output channels, 0.2-1 kept, 6-530 us) on B200.  CUDA cores: the cycles of the plan
// search at 0.656 ns, 3 us around them (half of the layers within 0.83-1.1 of it).  Tensor cores: 8 us around the rounds of
// items over the SMs, per round its steps and the output of a tile; a step costs 0.31 us at up to 48 columns, 0.44 at 128
// (0.85-1.1).  The margin leaves ties where they were: 27 -> 145 channels 3x3x3 on 2 x 4 x 16 x 44 24.2 us and 24.3.  Taken by
// this rule the 92 layers gain 1.19x in the mean (the better of both each time: 1.23x), 64 -> 128 on 2 x 16 x 56 x 56 3.1x.
bool split_is_faster(const rt3d_packed* w, const F32SplitArgs& a, int sm_count) {
  if (!split_fills_steps(w)) return false;
  const double density = double(w->nnz) / (double(w->P) * w->Q * w->Ks);
  const double groups = double(std::max(1, kSplitChunk / w->g_n)) * std::max(1, a.n_tile / w->g_m);     // that share a step
  const double steps = double(w->Ks) * ceil_div(w->N, kSplitChunk) * (w->is_dense ? 1.0 : 1.0 - std::pow(1.0 - density, groups));
  const int ctas = a.pair ? 2 : 1;
  const double tiles = double(a.tiles_n) * a.tiles_t * a.tiles_h * a.tiles_w;
  const double rounds = std::ceil(std::ceil(tiles / ctas) * a.n_bundles / (sm_count / ctas));
  const double step_us = a.n_tile <= 48 ? 0.31 : a.n_tile <= 64 ? 0.34 : a.n_tile <= 96 ? 0.36 : 0.44;
  const double tile_us = a.n_tile <= 48 ? 0.5 : a.n_tile <= 64 ? 2.0 : a.n_tile <= 96 ? 3.2 : 4.0;
  F32Plan plans[kF32MaxPlans];
  double cycles = 0.0;
  conv_f32_plans(a.g, density, sm_count, plans, &cycles);
  // group sizes that are not multiples of four run the first CUDA-core kernel, which is several times slower
  const double cuda_core_us = (3.0 + cycles * 0.656e-3) * (f32_layout_possible(w) ? 1.0 : 3.0);
  return 8.0 + rounds * (steps * step_us + tile_us) < 0.95 * cuda_core_us;
}

// fp32 on the tensor cores, each value as three bf16 ones.
// *launched = false (and RT3D_OK) when the handle or the shape does not suit it, the CUDA cores are faster (unless `anyway`: what
// they need is not there), or the call is being captured and the layout is not on the device.
rt3d_status try_split(rt3d_packed* w, DeviceBlob* blob, DeviceState* d, const rt3d_tensor* x, const ConvGeom& g, const float* bias,
                      rt3d_tensor* y, const void* res_data, int res_pitch, bool anyway, Submit& submit, bool* launched) {
  *launched = false;
  const int mode = g_f32_split.load();
  if (mode == 0 || d->cc_major != 10 || w->dtype != RT3D_F32 || x->c_stride % 4 || y->c_stride % 4 || (res_data && res_pitch % 4)) return RT3D_OK;
  if (g.st > 8 || g.sh > 8 || g.sw > 8 || int64_t(x->w) * x->c_stride * 4 >= (int64_t(1) << 40)) return RT3D_OK;
  if (int64_t(g.n) * g.To * g.Ho * g.Wo > 0x7fffffff) return RT3D_OK;
  if (!split_rows_bounded(w)) return RT3D_OK;
  F32SplitArgs a;
  a.g = g;
  a.box = choose_box(g);
  a.tiles_n = ceil_div(g.n, a.box.bn); a.tiles_t = ceil_div(g.To, a.box.bt);
  a.tiles_h = ceil_div(g.Ho, a.box.bh); a.tiles_w = ceil_div(g.Wo, a.box.bw);
  a.n_tile = split_n_tile(w->M); a.n_bundles = ceil_div(w->M, a.n_tile);
  // More steps to an accumulator cut more addends off, fewer wait more often for its sums to be drained: 128 columns take 169 us
  // with eight and 178 with four (96: 131 and 134, up to 64 columns 2 % less with eight).  Against 64 bits, over
  // 300 random layers and inputs of both signs and of one, this rule leaves at most 0.81 of the CUDA cores' error; eight everywhere
  // leave 0.93 on wide bundles and 1.01 up to 64 columns.  With more than 48 steps the CUDA cores' sums are long too.
  a.period = a.n_tile > 64 && w->Ks * ceil_div(w->N, kSplitChunk) > 48 ? 8 : 4;
  if (!umma_f32_plan(&a) || (long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w * a.n_bundles > (1ll << 30)) return RT3D_OK;
  if (mode == 1 && !split_is_faster(w, a, d->sm_count)) {
    if (!anyway) return RT3D_OK;
    submit.keep = false;
  }
  const UmmaLayout* L = get_split_layout(w, a.n_tile);
  if (!L) return RT3D_OK;
  if (submit.captured() && !umma_blob_ready(w, blob, umma_key(L->n_tile, false, false))) {
    submit.keep = false;                                   // one of the CUDA cores' layouts may be there
    return RT3D_OK;
  }
  DeviceBlob::Umma* u = nullptr;
  rt3d_status s = get_split_blob(w, blob, L, a.pair != 0, &u);
  if (s == RT3D_ERR_ALLOC) {                               // the CUDA cores' layout is a fraction of this one's size
    submit.keep = false;
    return RT3D_OK;
  }
  if (s != RT3D_OK) return s;
  a.last_chunk = L->n_chunks - 1;
  a.last_k16 = w->N - a.last_chunk * kSplitChunk > 16 ? 2 : 1;
  a.step_ptr = u->step_ptr; a.steps = u->steps; a.wtiles = static_cast<const unsigned char*>(u->wtiles);
  a.x = nullptr; a.y = nullptr; a.bias = nullptr; a.residual = nullptr; a.rcs = res_pitch;
  a.group_ptr = blob->group_ptr; a.pos_idx = blob->pos_idx; a.tiles = static_cast<const float*>(blob->tiles);
  a.g_m = w->g_m; a.g_n = w->g_n; a.Q = w->Q;
  a.again = int(split_again(w));
  a.sched = d->sched;
  const cuuint64_t cs = cuuint64_t(x->c_stride) * 4;
  cuuint64_t dims[5] = {cuuint64_t(x->c), cuuint64_t(x->w), cuuint64_t(x->h), cuuint64_t(x->t), cuuint64_t(x->n)};
  cuuint64_t strides[4] = {cs, cs * x->w, cs * x->w * x->h, cs * x->w * x->h * x->t};
  cuuint32_t bx[5] = {cuuint32_t(kSplitChunk), cuuint32_t(a.box.bw * g.sw), cuuint32_t(a.box.bh * g.sh), cuuint32_t(a.box.bt * g.st),
                      cuuint32_t(a.box.bn)};
  cuuint32_t estr[5] = {1, cuuint32_t(g.sw), cuuint32_t(g.sh), cuuint32_t(g.st), 1};
  CUtensorMap xmap;
  if (g_encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, x->data, dims, strides, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return RT3D_ERR_CUDA;
  *launched = true;
  const int sms = d->sm_count;
  return submit(rt3d_plan_info{8, a.n_tile, 1, 0, 0}, [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, c.x, xmap, nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    F32SplitArgs now = a;
    now.x = static_cast<const float*>(c.x); now.y = static_cast<float*>(c.y);
    now.bias = c.bias; now.residual = static_cast<const float*>(c.res);
    return launch_conv_umma_f32(now, &m.x, sms, st);
  });
}

// Register-blocked fp32 kernel: every fp32 call whose kernel groups are whole 4 x 4 tiles.
// *launched = false (and RT3D_OK) when the handle or the shape cannot use it.
rt3d_status try_f32(rt3d_packed* w, DeviceBlob* blob, DeviceState* d, const rt3d_tensor* x, const ConvGeom& g,
                    const float* bias, rt3d_tensor* y, const void* res_data, int res_pitch, Submit& submit, bool* launched) {
  *launched = false;
  if (!f32_layout_possible(w)) return RT3D_OK;
  F32Plan plans[kF32MaxPlans];
  double cycles = 0.0;
  const int n_plans = conv_f32_plans(g, double(w->nnz) / (double(w->P) * w->Q * w->Ks), d->sm_count, plans, &cycles);
  F32Args a;
  a.g = g;
  for (int i = 0; i < n_plans; ++i) {
    const F32Layout* L = get_f32_layout(w);
    if (!L || !conv_f32_fill(plans[i], *L, &a)) continue;
    DeviceBlob::F32* u = nullptr;
    rt3d_status s = get_f32_blob(w, blob, L, &u);
    if (s != RT3D_OK) return s;
    a.entry_ptr = u->entry_ptr; a.tile_ptr = u->tile_ptr; a.counts = u->counts; a.entries = u->entries; a.tiles = u->tiles;
    a.x = static_cast<const float*>(x->data); a.y = static_cast<float*>(y->data);
    a.bias = bias; a.residual = static_cast<const float*>(res_data); a.rcs = res_pitch;
    *launched = true;
    const F32Plan plan = plans[i];
    return submit(rt3d_plan_info{0, 0, 1, 0, 0}, [=](const CallBuffers& c, cudaStream_t st) {
      F32Args now = a;
      now.x = static_cast<const float*>(c.x); now.y = static_cast<float*>(c.y);
      now.bias = c.bias; now.residual = static_cast<const float*>(c.res);
      return launch_conv_f32(now, plan, st);
    });
  }
  return RT3D_OK;
}

// Which layouts the step-list kernels may choose from: all; those of steps of 64 channels; one that is on the device.  The others are
// for calls that are being captured, which cannot upload the layout that they would choose, on handles of up to 32 channels: theirs
// come in steps of 32 or 64, so that earlier calls and rt3d_packed_prepare may have left a layout of either kind.
enum class StepLists { kAll, kWide, kPresent };
rt3d_status conv_body(const rt3d_tensor* x, const rt3d_packed* wc, const float* bias, const rt3d_conv_params* p,
                      rt3d_tensor* y, void* stream, bool dense_entry, const rt3d_fusion* fz, StepLists lists = StepLists::kAll) {
  CallKey key;
  CallBuffers buffers{};
  if (make_key(&key, x, wc, bias, p, y, fz ? fz->residual : nullptr, dense_entry ? 1 : 0)) {
    if (fz) { key.misc[2] = fz->pool_t; key.misc[3] = fz->pool_h; key.misc[4] = fz->pool_w; }
    buffers = CallBuffers{x->data, y->data, fz && fz->residual ? fz->residual->data : nullptr, bias, nullptr};
    rt3d_status found;
    if (Submit(const_cast<rt3d_packed*>(wc), key, buffers, static_cast<cudaStream_t>(stream)).again(&found)) return found;
  }
  ConvGeom g;
  if (!y) return RT3D_ERR_INVALID_ARG;
  const bool pooled = fz && (fz->pool_t != 1 || fz->pool_h != 1 || fz->pool_w != 1);
  if (fz && (fz->pool_t < 1 || fz->pool_t > 2 || fz->pool_h < 1 || fz->pool_h > 2 || fz->pool_w < 1 || fz->pool_w > 2))
    return RT3D_ERR_INVALID_ARG;
  const int pl_t = fz ? fz->pool_t : 1, pl_h = fz ? fz->pool_h : 1, pl_w = fz ? fz->pool_w : 1;
  rt3d_status s = make_geom(x, wc, p, pooled ? nullptr : y, &g);
  if (s != RT3D_OK) return s;
  if (pooled) {                     // y holds the pooled tensor; g keeps the extents of the convolution output
    if ((s = check_tensor(y)) != RT3D_OK) return s;
    if (y->n != g.n || y->t != g.To / pl_t || y->h != g.Ho / pl_h || y->w != g.Wo / pl_w || y->c != wc->M ||
        y->dtype != wc->dtype || y->t < 1 || y->h < 1 || y->w < 1)
      return RT3D_ERR_SHAPE;
    if (fz->residual) return RT3D_ERR_UNSUPPORTED;
    g.ycs = y->c_stride;
  }
  if ((s = check_alignment(x)) != RT3D_OK || (s = check_alignment(y)) != RT3D_OK) return s;
  if (overlaps(x, y)) return RT3D_ERR_INVALID_ARG;
  const rt3d_tensor* res = fz ? fz->residual : nullptr;
  if (res) {
    if ((s = check_tensor(res)) != RT3D_OK || (s = check_alignment(res)) != RT3D_OK) return s;
    if (res->n != g.n || res->t != g.To || res->h != g.Ho || res->w != g.Wo || res->c != g.M || res->dtype != wc->dtype)
      return RT3D_ERR_SHAPE;
    if (overlaps(res, y)) return RT3D_ERR_INVALID_ARG;
  }
  const void* res_data = res ? res->data : nullptr;
  const int res_pitch = res ? res->c_stride : 0;
  if (dense_entry && !wc->is_dense) return RT3D_ERR_INVALID_ARG;
  rt3d_packed* w = const_cast<rt3d_packed*>(wc);
  DeviceState* d = nullptr;
  if ((s = get_device_state(&d)) != RT3D_OK) return s;
  DeviceBlob* blob = nullptr;
  if ((s = get_blob(w, &blob)) != RT3D_OK) return s;
  Submit submit(w, key, buffers, static_cast<cudaStream_t>(stream));
  submit.keep = lists == StepLists::kAll;
  const bool narrow = lists == StepLists::kAll && narrow_steps(w);

  const bool can_umma = umma_eligible(d, w, x, y, p);
  const bool can_simt = w->g_m <= kMaxGroupSimt && w->g_n <= kMaxGroupSimt;
  if (!can_umma && !can_simt) return RT3D_ERR_UNSUPPORTED;
  if (p->algo == RT3D_ALGO_SIMT && !can_simt) return RT3D_ERR_UNSUPPORTED;
  const bool want_umma = p->algo == RT3D_ALGO_UMMA || p->algo == RT3D_ALGO_UMMA_PAIR || p->algo == RT3D_ALGO_UMMA_HALO ||
                         p->algo == RT3D_ALGO_UMMA_SUB;
  if (want_umma && !can_umma) return RT3D_ERR_UNSUPPORTED;
  const bool use_umma = want_umma || (p->algo == RT3D_ALGO_AUTO && can_umma);
  if (!use_umma) {
    if (pooled) return RT3D_ERR_UNSUPPORTED;
    // a call that is being captured takes what is there: after a call on the tensor cores that is their layout and the canonical
    // arrays, after one on the CUDA cores the register-blocked kernel's layout or the canonical arrays
    const bool without = submit.captured() && f32_layout_possible(w) && !f32_blob_ready(w, blob);
    bool launched = false;
    if (p->algo == RT3D_ALGO_AUTO) {
      s = try_split(w, blob, d, x, g, bias, y, res_data, res_pitch, without, submit, &launched);
      if (s != RT3D_OK || launched) return s;
    }
    if (without && canonical_ready(w, blob)) submit.keep = false;
    else s = try_f32(w, blob, d, x, g, bias, y, res_data, res_pitch, submit, &launched);
    if (s != RT3D_OK || launched) return s;
    if ((s = get_canonical(w, blob)) != RT3D_OK) return s;
    return submit(rt3d_plan_info{0, 0, 1, 0, 0}, [=](const CallBuffers& c, cudaStream_t st) {
      return launch_conv_simt(w->dtype, g, c.x, c.y, blob->group_ptr, blob->pos_idx, blob->tiles, c.bias, w->g_m, w->g_n,
                              w->P, w->Q, dense_entry, c.res, res_pitch, st);
    });
  }

  const SmallCLayout* SL = nullptr;
  if (p->algo != RT3D_ALGO_UMMA_PAIR && p->algo != RT3D_ALGO_UMMA_HALO && p->algo != RT3D_ALGO_UMMA_SUB && (!pooled || pl_t == 1) &&
      smallc_eligible(d, w, x, y, p, &SL)) {
    return launch_smallc(w, blob, d, SL, x, g, bias, y, submit, res_data, res_pitch, pl_h, pl_w, p->x_pad_zero != 0);
  }

  if ((p->algo == RT3D_ALGO_AUTO || p->algo == RT3D_ALGO_UMMA_HALO) && !pooled) {
    bool launched = false;
    s = try_halo(w, blob, d, x, g, bias, y, res_data, res_pitch, dense_entry, p->algo == RT3D_ALGO_UMMA_HALO, submit, &launched);
    if (s != RT3D_OK || launched) return s;
  }
  if (p->algo == RT3D_ALGO_UMMA_HALO) return RT3D_ERR_UNSUPPORTED;
  if (p->algo == RT3D_ALGO_UMMA_SUB) {
    bool launched = false;
    if (!pooled && !dense_entry) {
      s = try_sub(w, blob, d, x, g, bias, y, res_data, res_pitch, submit, &launched);
      if (s != RT3D_OK || launched) return s;
    }
    return RT3D_ERR_UNSUPPORTED;
  }

  UmmaArgs a;
  a.g = g;
  int sb[4] = {1, 1, 1, 1};
  bool rect;
  if (pooled) {
    if (!choose_box_pool(g, pl_w, pl_h, pl_t, &a.box, sb)) return RT3D_ERR_UNSUPPORTED;
    rect = true;
  } else {
    a.box = choose_box(g);
    rect = warp_block(a.box.bw, a.box.bh, a.box.bt, a.box.bn, sb);
  }
  a.pool_t = pl_t; a.pool_h = pl_h; a.pool_w = pl_w; a.sbw = sb[0]; a.sbh = sb[1];
  a.tiles_n = ceil_div(g.n, a.box.bn); a.tiles_t = ceil_div(g.To, a.box.bt);
  a.tiles_h = ceil_div(g.Ho, a.box.bh); a.tiles_w = ceil_div(g.Wo, a.box.bw);
  long long m_tiles = (long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w;
  const UmmaLayout* present = lists == StepLists::kPresent ? present_umma_layout(w, blob) : nullptr;
  UmmaPlan plan = present ? UmmaPlan{present->n_tile, 1, false} : pick_plan(w, g, m_tiles, d->sm_count, narrow);
  if (pooled) {                     // pooling lives in the TMA-store epilogue, which a K split does not use
    // A layer this small is faster split over K and pooled by a second launch: AUTO declines the fusion.
    if (p->algo == RT3D_ALGO_AUTO && plan.n_splits > 1) return RT3D_ERR_UNSUPPORTED;
    plan.n_splits = 1;
  }
  // CTA pairs: two tiles per MMA.  Taken when every SM has a tile or the plan finds them faster; forced by RT3D_ALGO_UMMA_PAIR.
  bool use_pair = false;
  if (p->algo == RT3D_ALGO_UMMA_PAIR) {
    plan = UmmaPlan{present ? present->n_tile : default_n_tile(w->M), 1, true};
    if (!umma_pair_supported(plan.n_tile, ceil_div(w->M, plan.n_tile))) return RT3D_ERR_UNSUPPORTED;
    use_pair = true;
  } else if (p->algo == RT3D_ALGO_AUTO && plan.n_splits == 1 && !present &&
             umma_pair_supported(plan.n_tile, ceil_div(w->M, plan.n_tile)) &&
             (plan.pair || m_tiles * ceil_div(w->M, plan.n_tile) >= d->sm_count)) {
    use_pair = true;
  }
  if (pooled && plan.n_tile % 32) return RT3D_ERR_UNSUPPORTED;      // pooled rows leave as whole 32-channel pieces
  // CTA pairs on bundles up to 128 wide with a kernel that is 2 or 3 deep: one deeper input tile per (kh, kw, chunk)
  // (its box: among the boxes with as few tiles, one inside a single clip and as deep along t as possible; where none suits,
  // one inside a clip that reads less from L2 at up to a sixteenth more tiles: choose_box_grouped)
  bool use_ts = false;
  // (up to twelve locations on single CTAs stay with steps of 64: the S3D-shaped forward, whose branches are such layers of 16 to 32
  // channels, takes 772 us as a graph and 778 in steps of 32.  Repeated by themselves 60 random calls of that kind take 0.77 to 1.02
  // of the time in steps of 32, 0.967 in the mean.)
  a.narrow = present ? present->chunk != kChunk : narrow && (use_pair || w->Ks > 12);
  UmmaArgs probe = a;
  // (wide bundles: only kernels that are also wide in space; a 3x1x1 layer with 192-wide bundles lost 8 us of 43
  // inside the S3D-shaped forward with it, while 3x3x3 layers gain 1-4 %)
  if (use_pair && !present && g_ts_enabled.load() && g.st <= 2 && g.Kt >= 2 && g.Kt <= 8 && (plan.n_tile <= 128 || g.Kh * g.Kw >= 4)) {
    int sb2[4] = {1, 1, 1, 1};
    TileBox deep = a.box;
    const bool ok2 = pooled ? choose_box_pool(g, pl_w, pl_h, pl_t, &deep, sb2, true)
                            : (deep = choose_box(g, true), warp_block(deep.bw, deep.bh, deep.bt, deep.bn, sb2) == rect);
    const long long tiles2 = (long long)ceil_div(g.n, deep.bn) * ceil_div(g.To, deep.bt) * ceil_div(g.Ho, deep.bh) * ceil_div(g.Wo, deep.bw);
    if (ok2 && tiles2 == m_tiles) {
      probe.box = deep;
      probe.sbw = sb2[0]; probe.sbh = sb2[1];
      probe.tiles_n = ceil_div(g.n, deep.bn); probe.tiles_t = ceil_div(g.To, deep.bt);
      probe.tiles_h = ceil_div(g.Ho, deep.bh); probe.tiles_w = ceil_div(g.Wo, deep.bw);
    }
    probe.n_tile = plan.n_tile; probe.n_bundles = ceil_div(w->M, plan.n_tile); probe.dense = dense_entry && !a.narrow ? 1 : 0;
    use_ts = umma_pair_ts_supported(&probe, w->Ks * ceil_div(w->N, kChunk) * probe.n_bundles);
    const double ratio = use_ts || pooled ? 2.0 : choose_box_grouped(g, plan.n_tile, m_tiles, &deep);
    const bool rect2 = ratio < 1.0 && warp_block(deep.bw, deep.bh, deep.bt, deep.bn, sb2);
    if (ratio <= (rect && !rect2 ? 0.6 : g.sh * g.sw > 1 ? 0.68 : 0.8)) {
      probe.box = deep;
      probe.sbw = sb2[0]; probe.sbh = sb2[1];
      probe.tiles_n = g.n; probe.tiles_t = ceil_div(g.To, deep.bt);
      probe.tiles_h = ceil_div(g.Ho, deep.bh); probe.tiles_w = ceil_div(g.Wo, deep.bw);
      use_ts = umma_pair_ts_supported(&probe, w->Ks * ceil_div(w->N, kChunk) * probe.n_bundles);
      if (use_ts) {
        rect = rect2;
        m_tiles = (long long)probe.tiles_n * probe.tiles_t * probe.tiles_h * probe.tiles_w;
      }
    }
    if (use_ts) {
      a.box = probe.box; a.sbw = probe.sbw; a.sbh = probe.sbh;
      a.tiles_n = probe.tiles_n; a.tiles_t = probe.tiles_t; a.tiles_h = probe.tiles_h; a.tiles_w = probe.tiles_w;
      for (int i = 0; i < 4; ++i) sb[i] = sb2[i];
    }
  }
  const UmmaLayout* L = present ? present : get_umma_layout(w, plan.n_tile, use_ts, a.narrow != 0);
  if (!L) return RT3D_ERR_UNSUPPORTED;
  if (!present && narrow_steps(w) && submit.captured() && !umma_blob_ready(w, blob, umma_key(L->n_tile, use_ts, a.narrow != 0))) {
    if (narrow) return conv_body(x, wc, bias, p, y, stream, dense_entry, fz, StepLists::kWide);
    if (present_umma_layout(w, blob)) return conv_body(x, wc, bias, p, y, stream, dense_entry, fz, StepLists::kPresent);
  }
  DeviceBlob::Umma* u = nullptr;
  if ((s = get_umma_blob(w, blob, L, &u)) != RT3D_OK) return s;
  a.n_tile = L->n_tile; a.n_bundles = L->n_bundles; a.n_chunks = L->n_chunks;
  a.dense = dense_entry && !a.narrow && L->t_groups == use_ts ? 1 : 0;       // computed steps come in the layout's own order
  a.steps_dense = w->Ks * L->n_chunks;
  a.step_ptr = u->step_ptr; a.steps = u->steps;
  a.bias = bias; a.y = y->data; a.sched = d->sched;
  a.residual = res_data; a.rcs = res_pitch;
  a.n_splits = plan.n_splits;
  a.tail_workers = 0; a.tail_scratch = nullptr; a.tail_flags = nullptr;
  a.ts = 0; a.grp_ptr = nullptr; a.grp_first = nullptr; a.ts_a_bytes = 0; a.ts_frame_bytes = 0; a.ts_table = 0; a.ts_phases = 1;
  a.wait_cycles = debug_wait_cycles(); a.debug_drop_last_load = g_debug_drop_last_load.load();
  if (use_ts) {
    a.ts = 1; a.grp_ptr = u->grp_ptr; a.grp_first = u->grp_first;
    a.ts_a_bytes = probe.ts_a_bytes; a.ts_frame_bytes = probe.ts_frame_bytes; a.ts_table = probe.ts_table;
    a.ts_phases = probe.ts_phases;
  }
  CUtensorMap xmap;
  if ((s = encode_xmap(x, g, a.box, &xmap, use_ts ? ((g.Kt - 1) / g.st) * g.st : 0, L->chunk)) != RT3D_OK) return s;
  CUtensorMap ymap{};
  a.store_tma = (a.n_splits == 1 && rect && encode_ymap(y, sb, pl_w, pl_h, pl_t, &ymap)) ? 1 : 0;
  if (pooled && !a.store_tma) return RT3D_ERR_UNSUPPORTED;
  a.turned = use_pair && !pooled &&
             turn_pieces(a.n_tile, int(L->steps.size()) / a.n_bundles * L->chunk / kChunk, a.store_tma != 0, res_data != nullptr) ? 1 : 0;
  if (use_pair) {
    // items that do not fill a last round of CTA pairs are cut along K and shared
    // (its CTA pairs wait for one another, which needs the whole grid resident at once: not used when the caller
    // says that other kernels may run beside this call)
    size_t tail_bytes = 0, flag_bytes = 0;
    // (nor for AUTO when there are fewer items than pairs: what it would gain there, the cluster split gains with less)
    const long long pairs = (m_tiles + 1) / 2 * L->n_bundles;
    if (!p->concurrent && !present && (p->algo != RT3D_ALGO_AUTO || pairs >= d->sm_count / 2))
      umma_pair_tail_plan(&a, L->step_ptr.data(), d->sm_count, &tail_bytes, &flag_bytes, use_ts ? L->grp_ptr.data() : nullptr);
    if (a.tail_workers > 0) {
      DeviceBlob::Tail t;
      if ((s = get_tail(w, blob, tail_bytes, flag_bytes, &t)) != RT3D_OK) return s;
      a.tail_scratch = t.partial; a.tail_flags = t.flags;
      // up to a round and a half: the shared tiles, which are not turned, and one more each; it is their latency that counts
      // (83 -> 150 channels with a residual on 3 x 13 x 23 x 19, 76 items: 30.9 us, turned 31.2)
      if (pairs * 4 < d->sm_count * 3) a.turned = 0;
    }
  }
  const int sms = d->sm_count;
  const void* wmap = use_pair ? u->wmap_half : u->wmap;
  return submit(LastPlan({use_pair ? (use_ts ? 7 : 2) : 1, a.n_tile, a.n_splits, a.tail_workers, pooled ? 1 : 0}, L->chunk, a.turned),
                [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, c.x, ymap, a.store_tma ? c.y : nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    UmmaArgs now = a;
    now.y = c.y; now.bias = c.bias; now.residual = c.res;
    const void* ym = a.store_tma ? &m.y : nullptr;
    return use_pair ? launch_conv_umma_pair(now, &m.x, wmap, ym, sms, st) : launch_conv_umma(now, &m.x, wmap, ym, sms, st);
  });
}


// Fused spatial -> temporal pair.  Argument errors first (as the two separate calls would report them), then
// the eligibility screen of the one-kernel path.
rt3d_status conv2plus1d_body(const rt3d_tensor* x, const rt3d_packed* wsc, const float* bias_s, const rt3d_conv_params* ps,
                             const rt3d_packed* wtc, const float* bias_t, const rt3d_conv_params* pt,
                             const rt3d_tensor* res, rt3d_tensor* y, void* stream) {
  if (!wsc || !wtc || !ps || !pt || !y) return RT3D_ERR_INVALID_ARG;
  CallKey key;
  CallBuffers buffers{};
  if (make_key(&key, x, wsc, bias_s, ps, y, res, 2)) {
    key.w2 = wtc->id; key.misc[7] = bias_t != nullptr;
    put_params(pt, key.p + 10);
    buffers = CallBuffers{x->data, y->data, res ? res->data : nullptr, bias_s, bias_t};
    rt3d_status found;
    if (Submit(const_cast<rt3d_packed*>(wsc), key, buffers, static_cast<cudaStream_t>(stream)).again(&found)) return found;
  }
  ConvGeom g;
  rt3d_status s = make_geom(x, wsc, ps, nullptr, &g);
  if (s != RT3D_OK) return s;
  if (pt->st < 1 || pt->sh < 1 || pt->sw < 1 || pt->pt < 0 || pt->ph < 0 || pt->pw < 0) return RT3D_ERR_INVALID_ARG;
  if ((s = check_tensor(y)) != RT3D_OK) return s;
  if (wtc->N != wsc->M || wtc->dtype != wsc->dtype) return RT3D_ERR_SHAPE;
  if (g.To + 2 * pt->pt < wtc->Kt || g.Ho + 2 * pt->ph < wtc->Kh || g.Wo + 2 * pt->pw < wtc->Kw) return RT3D_ERR_SHAPE;
  const int64_t To2 = (int64_t(g.To) + 2 * pt->pt - wtc->Kt) / pt->st + 1;
  const int64_t Ho2 = (int64_t(g.Ho) + 2 * pt->ph - wtc->Kh) / pt->sh + 1;
  const int64_t Wo2 = (int64_t(g.Wo) + 2 * pt->pw - wtc->Kw) / pt->sw + 1;
  if (y->n != g.n || y->t != To2 || y->h != Ho2 || y->w != Wo2 || y->c != wtc->M || y->dtype != wtc->dtype)
    return RT3D_ERR_SHAPE;
  if ((s = check_alignment(x)) != RT3D_OK || (s = check_alignment(y)) != RT3D_OK) return s;
  if (overlaps(x, y)) return RT3D_ERR_INVALID_ARG;
  if (res) {
    if ((s = check_tensor(res)) != RT3D_OK || (s = check_alignment(res)) != RT3D_OK) return s;
    if (res->n != y->n || res->t != y->t || res->h != y->h || res->w != y->w || res->c != y->c || res->dtype != y->dtype)
      return RT3D_ERR_SHAPE;
    if (overlaps(res, y)) return RT3D_ERR_INVALID_ARG;
  }
  // what the one-kernel path takes
  if (wsc->dtype != RT3D_BF16) return RT3D_ERR_UNSUPPORTED;
  if (wsc->Kt != 1 || g.st != 1 || g.sh != 1 || g.sw != 1 || g.pt != 0 || wsc->N > kChunk || wsc->M > 256) return RT3D_ERR_UNSUPPORTED;
  if (wtc->Kt != 3 || wtc->Kh != 1 || wtc->Kw != 1 || pt->st != 1 || pt->sh != 1 || pt->sw != 1 || pt->pt != 1 ||
      pt->ph != 0 || pt->pw != 0 || wtc->M > 256)
    return RT3D_ERR_UNSUPPORTED;
  rt3d_packed* ws = const_cast<rt3d_packed*>(wsc);
  rt3d_packed* wt = const_cast<rt3d_packed*>(wtc);
  DeviceState* d = nullptr;
  if ((s = get_device_state(&d)) != RT3D_OK) return s;
  if (!umma_eligible(d, ws, x, y, ps) || !umma_layout_possible(wt)) return RT3D_ERR_UNSUPPORTED;
  if (res && res->c_stride % 8) return RT3D_ERR_UNSUPPORTED;
  StArgs a;
  a.g = g;
  a.c_mid = ws->M;
  a.n1 = round_up(ws->M, 16); a.n2 = round_up(wt->M, 16);
  if (2 * a.n1 + 3 * a.n2 > 512) return RT3D_ERR_UNSUPPORTED;
  const UmmaLayout* L1 = get_umma_layout(ws, a.n1);
  const UmmaLayout* L2 = get_umma_layout(wt, a.n2);
  if (!L1 || !L2 || L1->n_bundles != 1 || L2->n_bundles != 1 || L1->n_chunks != 1) return RT3D_ERR_UNSUPPORTED;
  a.n_steps1 = L1->step_ptr[1]; a.n_steps2 = L2->step_ptr[1];
  if (!umma_st_plan(&a, L1->steps.data(), L2->steps.data())) return RT3D_ERR_UNSUPPORTED;
  DeviceBlob *blob1 = nullptr, *blob2 = nullptr;
  if ((s = get_blob(ws, &blob1)) != RT3D_OK || (s = get_blob(wt, &blob2)) != RT3D_OK) return s;
  // a pair that is being captured and whose layers have left their steps of 32 channels only: two calls take those
  Submit submit(ws, key, buffers, static_cast<cudaStream_t>(stream));
  const auto elsewhere = [](rt3d_packed* h, DeviceBlob* b, const UmmaLayout* L) {
    return narrow_steps(h) && !umma_blob_ready(h, b, umma_key(L->n_tile, false, false)) && present_umma_layout(h, b);
  };
  if (submit.captured() && (elsewhere(ws, blob1, L1) || elsewhere(wt, blob2, L2))) return RT3D_ERR_UNSUPPORTED;
  DeviceBlob::Umma *u1 = nullptr, *u2 = nullptr;
  if ((s = get_umma_blob(ws, blob1, L1, &u1)) != RT3D_OK || (s = get_umma_blob(wt, blob2, L2, &u2)) != RT3D_OK) return s;
  a.M2 = wt->M; a.ycs = y->c_stride; a.relu2 = pt->relu ? 1 : 0;
  a.bias1 = bias_s; a.bias2 = bias_t; a.y = y->data;
  a.residual = res ? res->data : nullptr; a.rcs = res ? res->c_stride : 0;
  a.sched = d->sched;
  CUtensorMap xmap;
  ConvGeom unit = g;
  if ((s = encode_xmap(x, unit, TileBox{1, 1, a.hh, a.hw}, &xmap)) != RT3D_OK) return s;
  const int sms = d->sm_count;
  const void *m1 = u1->wmap_half, *m2 = u2->wmap_half;
  return submit(rt3d_plan_info{5, a.n1, 1, 0, 0}, [=](const CallBuffers& c, cudaStream_t st) {
    const PlacedMaps m(xmap, c.x, xmap, nullptr);
    if (!m.ok) return cudaErrorInvalidValue;
    StArgs now = a;
    now.y = c.y; now.bias1 = c.bias; now.bias2 = c.bias2; now.residual = c.res;
    return launch_conv_umma_st(now, &m.x, m1, m2, sms, st);
  });
}

// The two as the entry points call them: no exception leaves.
rt3d_status conv_impl(const rt3d_tensor* x, const rt3d_packed* w, const float* bias, const rt3d_conv_params* p,
                      rt3d_tensor* y, void* stream, bool dense_entry, const rt3d_fusion* fz = nullptr) {
  return c_entry([&] { return conv_body(x, w, bias, p, y, stream, dense_entry, fz); });
}
rt3d_status conv2plus1d_impl(const rt3d_tensor* x, const rt3d_packed* ws, const float* bias_s, const rt3d_conv_params* ps,
                             const rt3d_packed* wt, const float* bias_t, const rt3d_conv_params* pt,
                             const rt3d_tensor* res, rt3d_tensor* y, void* stream) {
  return c_entry([&] { return conv2plus1d_body(x, ws, bias_s, ps, wt, bias_t, pt, res, y, stream); });
}

}  // namespace

// ------------------------------------------------------------------ entry point without allocation
// Size limit of rt3d_conv3d_sparse_noalloc's K split: output tiles and fp32 partial tiles of a call.  The split needs no such
// memory; the limit is part of the interface, so that what was refused stays refused.
#define RT3D_NOALLOC_PARTIAL_TILES 128                                   /* 128 x 256 fp32 each */
#define RT3D_NOALLOC_PARTIAL_BYTES (RT3D_NOALLOC_PARTIAL_TILES * 128 * 256 * 4)   /* 16 MiB */

extern "C" {

rt3d_status rt3d_conv2plus1d_fused(const rt3d_tensor* x, const rt3d_packed* w_s, const float* bias_s,
                                   const rt3d_conv_params* p_s, const rt3d_packed* w_t, const float* bias_t,
                                   const rt3d_conv_params* p_t, const rt3d_tensor* residual, rt3d_tensor* y,
                                   void* stream) {
  return conv2plus1d_impl(x, w_s, bias_s, p_s, w_t, bias_t, p_t, residual, y, stream);
}

rt3d_status rt3d_conv3d_sparse(const rt3d_tensor* x, const rt3d_packed* w, const float* bias,
                               const rt3d_conv_params* p, rt3d_tensor* y, void* stream) {
  return conv_impl(x, w, bias, p, y, stream, false);
}

rt3d_status rt3d_conv3d_dense(const rt3d_tensor* x, const rt3d_packed* w, const float* bias,
                              const rt3d_conv_params* p, rt3d_tensor* y, void* stream) {
  return conv_impl(x, w, bias, p, y, stream, true);
}

rt3d_status rt3d_conv3d_sparse_fused(const rt3d_tensor* x, const rt3d_packed* w, const float* bias,
                                     const rt3d_conv_params* p, const rt3d_fusion* fusion, rt3d_tensor* y,
                                     void* stream) {
  if (!fusion || !w) return RT3D_ERR_INVALID_ARG;
  return conv_impl(x, w, bias, p, y, stream, w->is_dense != 0, fusion);
}

rt3d_status rt3d_conv3d_host(const rt3d_tensor* x, rt3d_packed* w, const float* bias, const rt3d_conv_params* p,
                             rt3d_tensor* y, void* stream) {
  ConvGeom g;
  if (!y) return RT3D_ERR_INVALID_ARG;
  rt3d_status s = make_geom(x, w, p, y, &g);
  if (s != RT3D_OK) return s;
  DeviceBlob* blob = nullptr;
  if ((s = c_entry([&] { return get_blob(w, &blob); })) != RT3D_OK) return s;
  const size_t xb = size_t(tensor_span_bytes(x)), yb = size_t(tensor_span_bytes(y));
  {
    std::lock_guard<std::mutex> lock(w->mu);
    if (blob->stage_x_bytes < xb) {
      cudaFree(blob->stage_x);
      blob->stage_x = nullptr; blob->stage_x_bytes = 0;
      if (dev_malloc(&blob->stage_x, xb + 256) != cudaSuccess) return RT3D_ERR_ALLOC;
      blob->stage_x_bytes = xb;
    }
    if (blob->stage_y_bytes < yb) {
      cudaFree(blob->stage_y);
      blob->stage_y = nullptr; blob->stage_y_bytes = 0; blob->stage_y_pitch = 0;
      if (dev_malloc(&blob->stage_y, yb + 256) != cudaSuccess) return RT3D_ERR_ALLOC;
      blob->stage_y_bytes = yb;
      blob->stage_y_pitch = 0;
    }
    // The padding channels, which no kernel writes, are copied out with the rest: zeros, not what the memory held before or
    // what a call of another pitch left there.
    if (y->c_stride == w->M) {
      blob->stage_y_pitch = 0;
    } else if (blob->stage_y_pitch != y->c_stride) {
      if (cudaMemsetAsync(blob->stage_y, 0, blob->stage_y_bytes, static_cast<cudaStream_t>(stream)) != cudaSuccess) return RT3D_ERR_CUDA;
      blob->stage_y_pitch = y->c_stride;
    }
    if (!blob->stage_bias && dev_malloc(&blob->stage_bias, size_t(w->M) * 4) != cudaSuccess)
      return RT3D_ERR_ALLOC;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (bias && cudaMemcpyAsync(blob->stage_bias, bias, size_t(w->M) * 4, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return RT3D_ERR_CUDA;
  const float* bias_d = bias ? blob->stage_bias : nullptr;
  // Clips are independent, so a large batch goes through in up to eight chunks of whole clips: chunk k+1 is
  // copied in on one stream while chunk k is convolved on the caller's stream and chunk k-1 is copied out on a
  // third (PCIe is full duplex; the call is bound by the larger of the two copies instead of their sum).
  constexpr int kHostChunks = 8;
  const int n_chunks = (x->n >= 2 && xb + yb >= (size_t(8) << 20)) ? (x->n < kHostChunks ? x->n : kHostChunks) : 1;
  if (n_chunks == 1) {
    if (cudaMemcpyAsync(blob->stage_x, x->data, xb, cudaMemcpyHostToDevice, st) != cudaSuccess) return RT3D_ERR_CUDA;
    rt3d_tensor xd = *x, yd = *y;
    xd.data = blob->stage_x;
    yd.data = blob->stage_y;
    s = conv_impl(&xd, w, bias_d, p, &yd, stream, w->is_dense != 0);
    if (s != RT3D_OK) return s;
    if (cudaMemcpyAsync(y->data, blob->stage_y, yb, cudaMemcpyDeviceToHost, st) != cudaSuccess) return RT3D_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return RT3D_ERR_CUDA;
    return RT3D_OK;
  }
  {
    std::lock_guard<std::mutex> lock(w->mu);
    for (void*& hs : blob->host_streams)
      if (!hs) {
        cudaStream_t ns;
        if (cudaStreamCreateWithFlags(&ns, cudaStreamNonBlocking) != cudaSuccess) return RT3D_ERR_CUDA;
        hs = ns;
      }
    for (void*& he : blob->host_events)
      if (!he) {
        cudaEvent_t ne;
        if (cudaEventCreateWithFlags(&ne, cudaEventDisableTiming) != cudaSuccess) return RT3D_ERR_CUDA;
        he = ne;
      }
  }
  cudaStream_t s_in = static_cast<cudaStream_t>(blob->host_streams[0]);
  cudaStream_t s_out = static_cast<cudaStream_t>(blob->host_streams[1]);
  auto ev = [&](int i) { return static_cast<cudaEvent_t>(blob->host_events[i]); };
  const size_t es = elem_size(x->dtype);
  const size_t x_clip = size_t(x->t) * x->h * x->w * x->c_stride * es, y_clip = size_t(y->t) * y->h * y->w * y->c_stride * es;
  bool cuda_ok = cudaEventRecord(ev(0), st) == cudaSuccess && cudaStreamWaitEvent(s_in, ev(0), 0) == cudaSuccess &&
                 cudaStreamWaitEvent(s_out, ev(0), 0) == cudaSuccess;
  rt3d_status cs = RT3D_OK;
  int n0 = 0;
  for (int k = 0; k < n_chunks && cuda_ok && cs == RT3D_OK; ++k) {
    const int n1 = int((long long)x->n * (k + 1) / n_chunks), nc = n1 - n0;
    const size_t xo = size_t(n0) * x_clip, yo = size_t(n0) * y_clip;
    const size_t xn = n1 == x->n ? xb - xo : size_t(nc) * x_clip, yn = n1 == x->n ? yb - yo : size_t(nc) * y_clip;
    cuda_ok = cudaMemcpyAsync(static_cast<char*>(blob->stage_x) + xo, static_cast<const char*>(x->data) + xo, xn,
                              cudaMemcpyHostToDevice, s_in) == cudaSuccess &&
              cudaEventRecord(ev(1 + k), s_in) == cudaSuccess && cudaStreamWaitEvent(st, ev(1 + k), 0) == cudaSuccess;
    if (!cuda_ok) break;
    rt3d_tensor xd = *x, yd = *y;
    xd.n = nc; yd.n = nc;
    xd.data = static_cast<char*>(blob->stage_x) + xo;
    yd.data = static_cast<char*>(blob->stage_y) + yo;
    cs = conv_impl(&xd, w, bias_d, p, &yd, stream, w->is_dense != 0);
    if (cs != RT3D_OK) break;
    cuda_ok = cudaEventRecord(ev(1 + kHostChunks + k), st) == cudaSuccess &&
              cudaStreamWaitEvent(s_out, ev(1 + kHostChunks + k), 0) == cudaSuccess &&
              cudaMemcpyAsync(static_cast<char*>(y->data) + yo, static_cast<char*>(blob->stage_y) + yo, yn,
                              cudaMemcpyDeviceToHost, s_out) == cudaSuccess;
    n0 = n1;
  }
  // the caller's stream ends up behind everything this call enqueued, whatever happened
  const bool joined = cudaEventRecord(ev(17), s_out) == cudaSuccess && cudaStreamWaitEvent(st, ev(17), 0) == cudaSuccess &&
                      cudaEventRecord(ev(0), s_in) == cudaSuccess && cudaStreamWaitEvent(st, ev(0), 0) == cudaSuccess;
  const bool synced = cudaStreamSynchronize(st) == cudaSuccess;
  if (cs != RT3D_OK) return cs;
  return (cuda_ok && joined && synced) ? RT3D_OK : RT3D_ERR_CUDA;
}

static rt3d_status prepare_body(rt3d_packed* p) {
  DeviceState* d = nullptr;
  rt3d_status s = get_device_state(&d);
  if (s != RT3D_OK) return s;
  DeviceBlob* blob = nullptr;
  if ((s = get_blob(p, &blob)) != RT3D_OK) return s;
  if (d->cc_major == 10 && umma_layout_possible(p)) {
    const UmmaLayout* L = get_umma_layout(p, 0);
    DeviceBlob::Umma* u = nullptr;
    if (L && (s = get_umma_blob(p, blob, L, &u)) != RT3D_OK) return s;
  } else if (const F32Layout* L = get_f32_layout(p)) {
    DeviceBlob::F32* u = nullptr;
    if ((s = get_f32_blob(p, blob, L, &u)) != RT3D_OK) return s;
  } else if ((s = get_canonical(p, blob)) != RT3D_OK) {
    return s;
  }
  F32SplitArgs split;
  split.n_tile = split_n_tile(p->M); split.n_bundles = ceil_div(p->M, split.n_tile);
  if (d->cc_major == 10 && p->dtype == RT3D_F32 && split_fills_steps(p) && split_rows_bounded(p) && g_f32_split.load() && umma_f32_plan(&split)) {
    DeviceBlob::Umma* u = nullptr;
    const UmmaLayout* L = get_split_layout(p, split.n_tile);
    // without the device memory for it calls run on the CUDA cores
    if (L && (s = get_split_blob(p, blob, L, split.pair != 0, &u)) != RT3D_OK && s != RT3D_ERR_ALLOC) return s;
  }
  for (int S = 2; S <= 8; ++S) umma_split_capacity(S, d->sm_count);      // what the K splits ask the runtime, once per device
  return cudaDeviceSynchronize() == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
}

rt3d_status rt3d_packed_prepare(rt3d_packed* p) {
  if (!p) return RT3D_ERR_INVALID_ARG;
  return c_entry([&] { return prepare_body(p); });
}

void rt3d_packed_free(rt3d_packed* p) {
  if (!p) return;
  int cur = -1;
  const bool have_dev = !p->blobs.empty() && cudaGetDevice(&cur) == cudaSuccess;
  {
    std::lock_guard<std::mutex> reg(g_blobs_mu);
    for (DeviceBlob* b : p->blobs)
      g_blobs.erase(std::remove(g_blobs.begin(), g_blobs.end(), b), g_blobs.end());
  }
  for (DeviceBlob* b : p->blobs) {
    const bool idle = have_dev && cudaSetDevice(b->device) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    weight_free(b->canonical, idle);
    for (auto& kv : b->umma) weight_free(kv.second.base, idle);
    cudaFree(b->stage_x); cudaFree(b->stage_y); cudaFree(b->stage_bias);
    for (void* hs : b->host_streams) if (hs) cudaStreamDestroy(static_cast<cudaStream_t>(hs));
    for (void* he : b->host_events) if (he) cudaEventDestroy(static_cast<cudaEvent_t>(he));
    for (auto& kv : b->smallc) weight_free(kv.second.base, idle);
    weight_free(b->f32.base, idle);
    for (auto& kv : b->sub) { cudaFree(kv.second.steps); cudaFree(kv.second.step_ptr); cudaFree(kv.second.blocks); }
    for (const DeviceBlob::Tail& t : b->tails) { cudaFree(t.partial); cudaFree(t.flags); }
    delete b;
  }
  if (have_dev && cur >= 0) cudaSetDevice(cur);
  delete p;
}

void rt3d_release_kept(void) {
  host_blocks_release();
  weight_blocks().release_all();
}

rt3d_status rt3d_maxpool3d(const rt3d_tensor* x, int kt, int kh, int kw, int st, int sh, int sw, int pt, int ph,
                           int pw, rt3d_tensor* y, void* stream) {
  rt3d_status s;
  if ((s = check_tensor(x)) != RT3D_OK || (s = check_tensor(y)) != RT3D_OK) return s;
  if (kt < 1 || kh < 1 || kw < 1 || st < 1 || sh < 1 || sw < 1 || pt < 0 || ph < 0 || pw < 0) return RT3D_ERR_INVALID_ARG;
  if (pt >= kt || ph >= kh || pw >= kw) return RT3D_ERR_INVALID_ARG;   // every window must see an input
  if (x->t + 2 * pt < kt || x->h + 2 * ph < kh || x->w + 2 * pw < kw) return RT3D_ERR_SHAPE;
  const int To = (x->t + 2 * pt - kt) / st + 1, Ho = (x->h + 2 * ph - kh) / sh + 1, Wo = (x->w + 2 * pw - kw) / sw + 1;
  if (y->n != x->n || y->t != To || y->h != Ho || y->w != Wo || y->c != x->c || y->dtype != x->dtype) return RT3D_ERR_SHAPE;
  // windows that start inside the padding but end before the tensor would see nothing
  if ((To - 1) * st - pt >= x->t || (Ho - 1) * sh - ph >= x->h || (Wo - 1) * sw - pw >= x->w) return RT3D_ERR_SHAPE;
  if ((s = check_alignment(x)) != RT3D_OK || (s = check_alignment(y)) != RT3D_OK) return s;
  if (overlaps(x, y)) return RT3D_ERR_INVALID_ARG;
  if (t_plan_only) return RT3D_OK;
  cudaError_t e = launch_maxpool3d(x->dtype, x->data, x->n, x->t, x->h, x->w, x->c, x->c_stride, kt, kh, kw, st, sh, sw,
                                   pt, ph, pw, y->data, To, Ho, Wo, y->c_stride, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return RT3D_ERR_CUDA;
  g_launches.fetch_add(1);
  return RT3D_OK;
}

rt3d_status rt3d_add_relu(const rt3d_tensor* a, const rt3d_tensor* b, int relu, rt3d_tensor* y, void* stream) {
  rt3d_status s;
  if ((s = check_tensor(a)) != RT3D_OK || (s = check_tensor(b)) != RT3D_OK || (s = check_tensor(y)) != RT3D_OK) return s;
  if (a->n != b->n || a->t != b->t || a->h != b->h || a->w != b->w || a->c != b->c || a->dtype != b->dtype) return RT3D_ERR_SHAPE;
  if (a->n != y->n || a->t != y->t || a->h != y->h || a->w != y->w || a->c != y->c || a->dtype != y->dtype) return RT3D_ERR_SHAPE;
  if ((s = check_alignment(a)) != RT3D_OK || (s = check_alignment(b)) != RT3D_OK || (s = check_alignment(y)) != RT3D_OK) return s;
  const int64_t vox = int64_t(a->n) * a->t * a->h * a->w;
  if (t_plan_only) return RT3D_OK;
  cudaError_t e = launch_add_relu(a->dtype, a->data, a->c_stride, b->data, b->c_stride, y->data, y->c_stride, vox, a->c,
                                  relu ? 1 : 0, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return RT3D_ERR_CUDA;
  g_launches.fetch_add(1);
  return RT3D_OK;
}

rt3d_status rt3d_copy_f32(const rt3d_copy* copies, int32_t n, void* stream) {
  if (!copies || n < 1) return RT3D_ERR_INVALID_ARG;
  for (int32_t i = 0; i < n; ++i)
    if (!copies[i].dst || copies[i].count < 1) return RT3D_ERR_INVALID_ARG;
  if (t_plan_only) return RT3D_OK;
  for (int32_t i = 0; i < n; i += kCopiesPerLaunch) {
    if (launch_copy_f32(copies + i, std::min(n - i, kCopiesPerLaunch), static_cast<cudaStream_t>(stream)) != cudaSuccess)
      return RT3D_ERR_CUDA;
    g_launches.fetch_add(1);
  }
  return RT3D_OK;
}

rt3d_status rt3d_run_calls(const rt3d_call* calls, int32_t n, void* const* streams, int32_t n_streams, int32_t* failed) {
  if (failed) *failed = -1;
  if (!calls || n < 0 || !streams || n_streams < 1) return RT3D_ERR_INVALID_ARG;
  // Events of the record / wait steps: one set per host thread and device.  A wait refers to the record issued last before
  // it, so a set serves one run after the other.
  struct Events {
    int device = -1;
    cudaEvent_t slot[RT3D_CALL_SLOTS] = {};
  };
  struct EventSets {
    std::vector<Events> sets;
    ~EventSets() {
      for (Events& e : sets)
        for (cudaEvent_t ev : e.slot)
          if (ev) cudaEventDestroy(ev);
    }
  };
  thread_local EventSets own;
  Events* events = nullptr;
  for (int32_t i = 0; i < n; ++i) {
    const rt3d_call& c = calls[i];
    rt3d_status s = RT3D_ERR_INVALID_ARG;
    if (c.lane >= 0 && c.lane < n_streams) {
      void* st = streams[c.lane];
      rt3d_tensor y = c.y;
      switch (c.kind) {
        case RT3D_CALL_SPARSE: s = conv_impl(&c.x, c.w, c.bias, &c.p, &y, st, false); break;
        case RT3D_CALL_DENSE: s = conv_impl(&c.x, c.w, c.bias, &c.p, &y, st, true); break;
        case RT3D_CALL_FUSED: {
          const rt3d_fusion fz{c.r.data ? &c.r : nullptr, c.k[0], c.k[1], c.k[2]};
          s = rt3d_conv3d_sparse_fused(&c.x, c.w, c.bias, &c.p, &fz, &y, st);
          break;
        }
        case RT3D_CALL_PAIR:
          s = conv2plus1d_impl(&c.x, c.w, c.bias, &c.p, c.w2, c.bias2, &c.p2, c.r.data ? &c.r : nullptr, &y, st);
          break;
        case RT3D_CALL_MAXPOOL:
          s = rt3d_maxpool3d(&c.x, c.k[0], c.k[1], c.k[2], c.k[3], c.k[4], c.k[5], c.k[6], c.k[7], c.k[8], &y, st);
          break;
        case RT3D_CALL_ADD: s = rt3d_add_relu(&c.x, &c.r, c.k[0], &y, st); break;
        case RT3D_CALL_COPY: s = rt3d_copy_f32(static_cast<const rt3d_copy*>(c.x.data), c.k[0], st); break;
        case RT3D_CALL_RECORD:
        case RT3D_CALL_WAIT: {
          if (c.k[0] < 0 || c.k[0] >= RT3D_CALL_SLOTS) break;
          if (!events) {
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess) { s = RT3D_ERR_CUDA; break; }
            for (Events& e : own.sets)
              if (e.device == dev) events = &e;
            if (!events) {
              s = c_entry([&] { own.sets.emplace_back(); return RT3D_OK; });
              if (s != RT3D_OK) break;
              events = &own.sets.back();
              events->device = dev;
            }
          }
          cudaEvent_t& ev = events->slot[c.k[0]];
          if (!ev && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) { s = RT3D_ERR_CUDA; break; }
          const cudaError_t e = c.kind == RT3D_CALL_RECORD ? cudaEventRecord(ev, static_cast<cudaStream_t>(st))
                                                           : cudaStreamWaitEvent(static_cast<cudaStream_t>(st), ev, 0);
          s = e == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
          break;
        }
      }
    }
    if (s != RT3D_OK) {
      if (failed) *failed = i;
      return s;
    }
  }
  return RT3D_OK;
}

rt3d_status rt3d_conv3d_cost(const rt3d_tensor* x, const rt3d_packed* w, const rt3d_conv_params* p,
                             int64_t* kept_macs, int64_t* dense_macs, int64_t* alg_bytes) {
  ConvGeom g;
  rt3d_status s = make_geom(x, w, p, nullptr, &g);
  if (s != RT3D_OK) return s;
  const int64_t vox_out = int64_t(g.n) * g.To * g.Ho * g.Wo;
  // kept weights that exist (ragged groups hold fewer than g_m*g_n kernels)
  int64_t kept_w = 0;
  for (int pr = 0; pr < w->P; ++pr) {
    const int rows = std::min(w->g_m, w->M - pr * w->g_m);
    for (int q = 0; q < w->Q; ++q) {
      const int cols = std::min(w->g_n, w->N - q * w->g_n);
      kept_w += int64_t(w->group_ptr[size_t(pr) * w->Q + q + 1] - w->group_ptr[size_t(pr) * w->Q + q]) * rows * cols;
    }
  }
  if (kept_macs) *kept_macs = vox_out * kept_w;
  if (dense_macs) *dense_macs = vox_out * int64_t(w->M) * w->N * w->Ks;
  if (alg_bytes) {
    const int64_t e = int64_t(elem_size(w->dtype));
    const int64_t vox_in = int64_t(g.n) * g.t * g.h * g.w;
    *alg_bytes = vox_in * g.c * e + vox_out * g.M * e + w->nnz * w->g_m * w->g_n * e + w->nnz * 2 +
                 int64_t(w->P) * w->Q * 4 + 4 + int64_t(w->M) * 4;
  }
  return RT3D_OK;
}

rt3d_status rt3d_conv3d_query_algo(const rt3d_tensor* x, const rt3d_packed* w, const rt3d_conv_params* p,
                                   const rt3d_tensor* y, int* algo) {
  ConvGeom g;
  if (!algo || !y) return RT3D_ERR_INVALID_ARG;
  rt3d_status s = make_geom(x, w, p, y, &g);
  if (s != RT3D_OK) return s;
  DeviceState* d = nullptr;
  if ((s = get_device_state(&d)) != RT3D_OK) return s;
  const bool can = umma_eligible(d, w, x, y, p);
  if (p->algo == RT3D_ALGO_UMMA && !can) return RT3D_ERR_UNSUPPORTED;
  *algo = (p->algo == RT3D_ALGO_SIMT || !can) ? RT3D_ALGO_SIMT : RT3D_ALGO_UMMA;
  return RT3D_OK;
}

rt3d_status rt3d_last_plan(rt3d_plan_info* info) {
  if (!info || t_last_plan.info.kernel < 0) return RT3D_ERR_INVALID_ARG;
  *info = t_last_plan.info;
  return RT3D_OK;
}

long long rt3d_debug_get(int what) {
  if (what == RT3D_DEBUG_STEP_CHANNELS) return t_last_plan.step_channels;
  if (what == RT3D_DEBUG_TURNED) return t_last_plan.turned;
  if (what != RT3D_DEBUG_WAIT_SITE) return -1;
  DeviceState* d = nullptr;
  if (get_device_state(&d) != RT3D_OK) return -1;
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  int32_t word = 0;
  if (cudaMemcpy(&word, d->sched + 2, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
  return word;
}

rt3d_status rt3d_last_device_status(void* stream) {
  DeviceState* d = nullptr;
  rt3d_status s = get_device_state(&d);
  if (s != RT3D_OK) return s;
  if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return RT3D_ERR_CUDA;
  int32_t word = 0;
  if (cudaMemcpy(&word, d->sched + 2, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return RT3D_ERR_CUDA;
  if (word != 0) {
    cudaMemset(d->sched + 2, 0, 4);
    // A kernel that gave up may have left tail-split flags non-zero (they are cleared by the pair that finishes a tile):
    // clear them for every handle on this device, so that later calls do not take a stale flag for a share that is there.
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) {
      cudaDeviceSynchronize();
      std::lock_guard<std::mutex> reg(g_blobs_mu);
      for (DeviceBlob* b : g_blobs)
        if (b->device == dev)
          for (const DeviceBlob::Tail& t : b->tails) cudaMemset(t.flags, 0, t.flag_bytes);
    }
    uploads_done();
    return RT3D_ERR_TIMEOUT;
  }
  return RT3D_OK;
}

rt3d_status rt3d_conv3d_sparse_noalloc(const rt3d_tensor* x, const rt3d_packed* wc, const float* bias,
                                       const rt3d_conv_params* p, rt3d_tensor* y, void* stream) {
  ConvGeom g;
  if (!y) return RT3D_ERR_INVALID_ARG;
  rt3d_status s = make_geom(x, wc, p, y, &g);
  if (s != RT3D_OK) return s;
  if ((s = check_alignment(x)) != RT3D_OK || (s = check_alignment(y)) != RT3D_OK) return s;
  if (overlaps(x, y)) return RT3D_ERR_INVALID_ARG;
  if (p->algo == RT3D_ALGO_SIMT) return RT3D_ERR_UNSUPPORTED;
  rt3d_packed* w = const_cast<rt3d_packed*>(wc);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RT3D_ERR_CUDA;
  // everything that needs an allocation must already exist: device state, weight blobs (rt3d_packed_prepare)
  DeviceState* d = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (g_dev[dev].init) d = &g_dev[dev];
  }
  if (!d) return RT3D_ERR_NOT_PREPARED;
  if (!umma_eligible(d, w, x, y, p)) return RT3D_ERR_UNSUPPORTED;
  const int n_tile = default_n_tile(w->M);
  DeviceBlob* blob = nullptr;
  DeviceBlob::Umma* u = nullptr;
  const UmmaLayout* L = nullptr;
  {
    std::lock_guard<std::mutex> lock(w->mu);
    blob = find_blob(w, dev);
    // steps of 64, which rt3d_packed_prepare uploads, or the steps of 32 of an earlier call
    for (const int key : {umma_key(n_tile, false, false), umma_key(n_tile, false, true)}) {
      if (!blob || u) break;
      const auto it = blob->umma.find(key);
      const auto li = w->umma_layouts.find(key);
      if (it != blob->umma.end() && it->second.ready && li != w->umma_layouts.end()) { u = &it->second; L = &li->second; }
    }
  }
  if (!u) return RT3D_ERR_NOT_PREPARED;

  UmmaArgs a;
  a.g = g;
  a.box = choose_box(g);
  a.tiles_n = ceil_div(g.n, a.box.bn); a.tiles_t = ceil_div(g.To, a.box.bt);
  a.tiles_h = ceil_div(g.Ho, a.box.bh); a.tiles_w = ceil_div(g.Wo, a.box.bw);
  a.n_tile = L->n_tile; a.n_bundles = L->n_bundles; a.n_chunks = L->n_chunks;
  a.dense = 0;
  a.steps_dense = w->Ks * L->n_chunks;
  a.step_ptr = u->step_ptr; a.steps = u->steps;
  a.bias = bias; a.y = y->data; a.sched = d->sched;
  // Split rule of this entry point: as many K splits (at most 8) as keep every SM busy, each with at
  // least 8 of the K steps of the layer's longest step list.
  const long long tiles = (long long)a.tiles_n * a.tiles_t * a.tiles_h * a.tiles_w * L->n_bundles;
  long long splits = tiles > 0 ? d->sm_count / tiles : 1;
  if (splits > 8) splits = 8;
  if (splits > L->max_steps / 8) splits = L->max_steps / 8;
  while (splits > 1 && umma_split_capacity(int(splits), d->sm_count) == 0) --splits;
  if (splits < 1) splits = 1;
  a.n_splits = int(splits);
  a.residual = nullptr; a.rcs = 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (a.n_splits > 1 && (tiles * a.n_splits * kTileM * L->n_tile * 4LL > RT3D_NOALLOC_PARTIAL_BYTES || tiles > RT3D_NOALLOC_PARTIAL_TILES))
    return RT3D_ERR_WORKSPACE;
  CUtensorMap xmap;
  if ((s = encode_xmap(x, g, a.box, &xmap, 0, L->chunk)) != RT3D_OK) return s;
  CUtensorMap ymap;
  int sb[4];
  a.pool_t = a.pool_h = a.pool_w = 1; a.sbw = a.sbh = 1;
  a.tail_workers = 0; a.tail_scratch = nullptr; a.tail_flags = nullptr;
  a.ts = 0; a.grp_ptr = nullptr; a.grp_first = nullptr; a.ts_a_bytes = 0; a.ts_frame_bytes = 0; a.ts_table = 0; a.ts_phases = 1;
  a.wait_cycles = 0; a.debug_drop_last_load = 0;
  a.turned = 0; a.narrow = L->chunk != kChunk;
  a.store_tma = (a.n_splits == 1 && warp_block(a.box.bw, a.box.bh, a.box.bt, a.box.bn, sb) &&
                 encode_ymap(y, sb, 1, 1, 1, &ymap)) ? 1 : 0;
  if (launch_conv_umma(a, &xmap, u->wmap, a.store_tma ? &ymap : nullptr, d->sm_count, st) != cudaSuccess) return RT3D_ERR_CUDA;
  g_launches.fetch_add(1);
  t_last_plan = LastPlan({1, a.n_tile, a.n_splits, 0, 0}, L->chunk);
  return RT3D_OK;
}

int64_t rt3d_launch_count(void) { return g_launches.load(); }

int64_t rt3d_alloc_count(void) { return g_allocs.load(); }

void rt3d_plan_begin(void) { t_plan_only = true; }
void rt3d_plan_end(void) { t_plan_only = false; }

rt3d_status rt3d_debug_set(int what, long long value) {
  g_plan_epoch.fetch_add(1);
  if (what == RT3D_DEBUG_WAIT_CYCLES) { if (value < 0) return RT3D_ERR_INVALID_ARG; g_debug_wait_cycles.store(value); return RT3D_OK; }
  if (what == RT3D_DEBUG_DROP_LAST_LOAD) { g_debug_drop_last_load.store(value != 0); return RT3D_OK; }
  if (what == RT3D_DEBUG_T_GROUPS) { g_ts_enabled.store(value != 0); return RT3D_OK; }
  if (what == RT3D_DEBUG_NARROW) { g_narrow_enabled.store(value != 0); return RT3D_OK; }
  if (what == RT3D_DEBUG_F32_SPLIT) { if (value < 0 || value > 2) return RT3D_ERR_INVALID_ARG; g_f32_split.store(int(value)); return RT3D_OK; }
  if (what == RT3D_DEBUG_POISON) {
    DeviceState* d = nullptr;
    rt3d_status s = get_device_state(&d);
    if (s != RT3D_OK) return s;
    if (d->cc_major != 10) return RT3D_ERR_UNSUPPORTED;
    if (launch_debug_poison(uint32_t(value), d->sm_count, d->sched + 8, nullptr) != cudaSuccess) return RT3D_ERR_CUDA;
    if (cudaDeviceSynchronize() != cudaSuccess) return RT3D_ERR_CUDA;
    // the tail splits' partial tiles in global memory too (all ones: NaNs as fp32); their flags stay zero
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RT3D_ERR_CUDA;
    std::lock_guard<std::mutex> reg(g_blobs_mu);
    for (DeviceBlob* b : g_blobs)
      if (b->device == dev)
        for (const DeviceBlob::Tail& t : b->tails)
          if (cudaMemset(t.partial, 0xFF, t.bytes) != cudaSuccess) return RT3D_ERR_CUDA;
    return uploads_done() == cudaSuccess ? RT3D_OK : RT3D_ERR_CUDA;
  }
  return RT3D_ERR_INVALID_ARG;
}


const char* rt3d_status_string(rt3d_status s) {
  switch (s) {
    case RT3D_OK: return "ok";
    case RT3D_ERR_INVALID_ARG: return "invalid argument";
    case RT3D_ERR_SHAPE: return "shape or dtype mismatch";
    case RT3D_ERR_MASK_NOT_GROUP_UNIFORM: return "mask is not uniform inside a kernel group";
    case RT3D_ERR_UNSUPPORTED: return "unsupported";
    case RT3D_ERR_ALLOC: return "allocation failed";
    case RT3D_ERR_CUDA: return "CUDA error";
    case RT3D_ERR_TIMEOUT: return "device-side wait timed out";
    case RT3D_ERR_WORKSPACE: return "request needs more than the library's fixed workspace";
    case RT3D_ERR_NOT_PREPARED: return "handle not prepared on this device (call rt3d_packed_prepare first)";
  }
  return "unknown status";
}

const char* rt3d_version(void) { return "rt3d-b200 0.1 (sm_100a)"; }

}  // extern "C"
