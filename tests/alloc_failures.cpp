// Every allocation of the packers and of the layouts derived from a handle fails once, alone and with all that follow it,
// on whichever thread makes it: the call must say RT3D_ERR_ALLOC and the next one must work.  Built with pack.cpp alone.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <new>
#include <vector>

#include "rt3d_internal.h"

static std::atomic<long> g_left{-1};      // allocations until the one that fails; -1: none does
static std::atomic<bool> g_go_on{false};  // the later ones fail too

void* operator new(size_t n) {
  long left = g_left.load();
  while (left >= 0 && !g_left.compare_exchange_weak(left, left > 0 ? left - 1 : (g_go_on ? 0 : -1))) {}
  void* p = left == 0 ? nullptr : std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void* operator new(size_t n, const std::nothrow_t&) noexcept {
  try { return operator new(n); } catch (const std::bad_alloc&) { return nullptr; }
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

namespace rt3d { struct PreparedCall {}; }
extern "C" void rt3d_packed_free(rt3d_packed* p) { delete p; }     // no device blobs here

static int fail(const char* what, long k, int status) {
  std::printf("%s: allocation %ld: status %d\n", what, k, status);
  return 1;
}

// `call` works on a handle that `fresh` makes anew (nullptr: it makes its own and frees it).
static int each_allocation(const char* what, const std::function<rt3d_packed*()>& fresh, const std::function<int(rt3d_packed*)>& call) {
  for (int go_on = 0; go_on < 2; ++go_on)
    for (long k = 0;; ++k) {
      rt3d_packed* h = fresh ? fresh() : nullptr;
      g_go_on = go_on != 0;
      g_left = k;
      int s = call(h);
      const bool failed = go_on ? g_left.load() == 0 : g_left.load() < 0;
      g_left = -1;
      if (s != RT3D_OK && s != RT3D_ERR_ALLOC) return fail(what, k, s);
      if (s == RT3D_ERR_ALLOC && (s = call(h)) != RT3D_OK) return fail(what, k, s);      // and then it works
      if (h) rt3d_packed_free(h);
      if (!failed) {
        std::printf("%s: %ld allocations\n", what, k);
        break;
      }
    }
  return 0;
}

int main() {
  const int M = 256, N = 256, Ks = 27;
  std::vector<float> w(size_t(M) * N * Ks);
  std::vector<uint8_t> mask(w.size());
  for (size_t i = 0; i < w.size(); ++i) {
    w[i] = float(i % 1000) - 500.f;
    const size_t m = i / (size_t(N) * Ks), c = i / Ks % N, k = i % Ks;
    mask[i] = ((m / 4) * 31 + (c / 4) * 17 + k * 7) % 5 < 2;
  }
  std::vector<float> back(w.size());
  const auto pack = [&](int dtype) {
    rt3d_packed* h = nullptr;
    if (rt3d_pack_kgs(w.data(), mask.data(), M, N, 3, 3, 3, 4, 4, dtype, &h) != RT3D_OK) std::abort();
    return h;
  };
  const auto bf16 = [&] { return pack(RT3D_BF16); };
  rt3d_packed* part = pack(RT3D_F32);
  const rt3d_packed* parts[2] = {part, part};
  int bad = 0;
  bad |= each_allocation("pack", nullptr, [&](rt3d_packed*) {
    rt3d_packed* h = reinterpret_cast<rt3d_packed*>(8);
    const int s = rt3d_pack_kgs(w.data(), mask.data(), M, N, 3, 3, 3, 4, 4, RT3D_BF16, &h);
    if ((h != nullptr) != (s == RT3D_OK)) return -1;
    if (h) rt3d_packed_free(h);
    return s;
  });
  bad |= each_allocation("concat", nullptr, [&](rt3d_packed*) {
    rt3d_packed* h = reinterpret_cast<rt3d_packed*>(8);
    const int s = rt3d_pack_concat(parts, 2, &h);
    if ((h != nullptr) != (s == RT3D_OK)) return -1;
    if (h) rt3d_packed_free(h);
    return s;
  });
  bad |= each_allocation("fp32 layout", [&] { return pack(RT3D_F32); }, [&](rt3d_packed* h) {
    try {
      return rt3d::get_f32_layout(h) ? int(RT3D_OK) : -1;
    } catch (const std::bad_alloc&) {                     // its caller's entry point makes a status of it
      return int(RT3D_ERR_ALLOC);
    }
  });
  bad |= each_allocation("tensor-core layout", bf16, [&](rt3d_packed* h) { return rt3d_unpack_device_layout(h, 0, back.data()); });
  bad |= each_allocation("t-grouped layout", bf16, [&](rt3d_packed* h) { return rt3d_unpack_device_layout_tgroups(h, 128, back.data()); });
  bad |= each_allocation("sub-tile layout", bf16, [&](rt3d_packed* h) { return rt3d_unpack_sub_layout(h, 0, back.data()); });
  rt3d_packed_free(part);
  if (!bad) std::printf("ok\n");
  return bad;
}
