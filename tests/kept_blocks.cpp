// Blocks kept between handles: which are found again, which go, and that the bounds hold.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <thread>

#include "kept_blocks.h"

static std::vector<void*> g_gone;
static std::mutex g_mu;
static void release(void* p) {
  std::lock_guard<std::mutex> lock(g_mu);
  g_gone.push_back(p);
}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
  const size_t MB = size_t(1) << 20;
  rt3d::KeptBlocks kept(release);
  char at[64];
  const auto gone = [&](const char* p) { return int(std::count(g_gone.begin(), g_gone.end(), (void*)p)); };
  // found again at the size asked for up to a quarter more, on its device only; a request that finds none drops none
  kept.note(at, 10 * MB, 0);
  kept.give(at);
  CHECK(!kept.take(10 * MB + 1, 0) && !kept.take(8 * MB - 1, 0) && !kept.take(10 * MB, 1) && g_gone.empty());
  CHECK(kept.take(8 * MB, 0) == at && !kept.take(10 * MB, 0));
  kept.give(at);
  CHECK(kept.take(10 * MB, 0) == at);
  kept.drop(at);                                            // not kept: released at once
  CHECK(gone(at) == 1 && !kept.take(10 * MB, 0));
  // small, oversized and unknown blocks are released when they come
  kept.note(at + 1, (256 << 10) - 1, 0);
  kept.note(at + 2, 32 * MB + 1, 0);
  for (int i = 1; i <= 3; ++i) { kept.give(at + i); CHECK(gone(at + i) == 1); }
  // 64 MB in all: the oldest goes first, one that was taken and given again counts as new
  for (int i = 10; i < 14; ++i) { kept.note(at + i, 16 * MB, 0); kept.give(at + i); }
  CHECK(kept.take(16 * MB, 0) == at + 10);
  kept.give(at + 10);
  kept.note(at + 14, 17 * MB, 0);
  kept.give(at + 14);
  CHECK(gone(at + 11) == 1 && gone(at + 12) == 1 && gone(at + 13) == 0 && gone(at + 10) == 0 && gone(at + 14) == 0);
  kept.release_all();
  CHECK(gone(at + 10) == 1 && gone(at + 13) == 1 && gone(at + 14) == 1 && !kept.take(16 * MB, 0));
  // several threads: a block has one owner at a time, and every one is released once
  static std::atomic<long> made{0}, freed{0};
  static std::atomic<bool> shared{false};
  rt3d::KeptBlocks real([](void* p) { ++freed; std::free(p); });
  std::vector<std::thread> threads;
  for (int t = 0; t < 4; ++t)
    threads.emplace_back([&] {
      for (int i = 0; i < 5000; ++i) {
        auto* p = static_cast<std::atomic<int>*>(real.take(4 * MB, 0));
        if (!p) {
          p = new (std::calloc(1, 64)) std::atomic<int>(0);
          ++made;
          real.note(p, 4 * MB, 0);
        }
        if (p->exchange(1)) shared = true;
        p->store(0);
        if (i % 50 == 49) real.drop(p); else real.give(p);
        if (i % 300 == 299) real.release_all();
      }
    });
  for (std::thread& t : threads) t.join();
  real.release_all();
  CHECK(!shared && made == freed);
  std::printf("ok\n");
  return 0;
}
