// Large blocks of freed handles, kept for the next handle.
//
// A pruning loop packs, uploads and frees a layer again and again, and most of that was memory management: the page faults
// of a fresh 4 MB block (1 ms), cudaMalloc and cudaFree of 18 MB (0.45 and 0.55 ms).  512 x 512 x 27 at 0.28 kept, packed,
// uploaded, read back and freed: 4.9 -> 2.6 ms (2.0 since).  A process that only loads layers never finds a kept block.
// Bounds: at most kMost bytes in all, no block over half of that; the oldest ones go when a new one needs the room.  All of
// them go on request and before an allocation is given up.
#pragma once
#include <cstddef>
#include <mutex>
#include <new>
#include <unordered_map>
#include <vector>

namespace rt3d {

class KeptBlocks {
 public:
  static constexpr size_t kSmallest = size_t(256) << 10, kMost = size_t(64) << 20;

  explicit KeptBlocks(void (*release)(void*)) : release_(release) {}

  // A kept block of at least `bytes` and at most a quarter more, on `device`; nullptr if there is none.
  void* take(size_t bytes, int device) {
    if (bytes < kSmallest) return nullptr;
    std::lock_guard<std::mutex> lock(mu_);
    for (size_t i = 0; i < kept_.size(); ++i)
      if (kept_[i].device == device && kept_[i].bytes >= bytes && kept_[i].bytes - bytes <= bytes / 4) {
        void* const p = kept_[i].p;
        out_[p] = kept_[i];
        total_ -= kept_[i].bytes;
        kept_.erase(kept_.begin() + long(i));
        return p;
      }
    return nullptr;
  }
  // Tells of a block that the caller allocated, so that give() knows its size; one that is not noted for want of memory is
  // released there.
  void note(void* p, size_t bytes, int device) noexcept {
    if (bytes < kSmallest || bytes > kMost / 2) return;
    try {
      std::lock_guard<std::mutex> lock(mu_);
      kept_.reserve(out_.size() + kept_.size() + 1);      // room for all of them, so that give() allocates nothing
      out_[p] = Block{p, bytes, device};
    } catch (const std::bad_alloc&) {
    }
  }
  // Keeps a block or releases it.  Nothing may use it any more.
  void give(void* p) noexcept {
    if (!p) return;
    std::unique_lock<std::mutex> lock(mu_);
    auto it = out_.find(p);
    if (it == out_.end()) {
      lock.unlock();
      release_(p);
      return;
    }
    const Block b = it->second;
    out_.erase(it);
    kept_.push_back(b);
    total_ += b.bytes;
    while (total_ > kMost) drop_oldest(lock);
  }
  // Releases a block that shall not be kept.
  void drop(void* p) noexcept {
    if (!p) return;
    {
      std::lock_guard<std::mutex> lock(mu_);
      out_.erase(p);
    }
    release_(p);
  }
  // Releases every kept block.
  void release_all() noexcept {
    std::unique_lock<std::mutex> lock(mu_);
    while (!kept_.empty()) drop_oldest(lock);
  }

 private:
  struct Block { void* p; size_t bytes; int device; };
  void drop_oldest(std::unique_lock<std::mutex>& lock) noexcept {
    const Block b = kept_.front();
    kept_.erase(kept_.begin());
    total_ -= b.bytes;
    lock.unlock();                                        // releasing device memory waits for the device
    release_(b.p);
    lock.lock();
  }
  void (*release_)(void*);
  std::mutex mu_;
  std::vector<Block> kept_;                               // oldest first
  std::unordered_map<void*, Block> out_;
  size_t total_ = 0;
};

}  // namespace rt3d
