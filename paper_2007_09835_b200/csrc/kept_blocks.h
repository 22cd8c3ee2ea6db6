// Large blocks of freed handles, kept for the next handle.
//
// A pruning loop packs, uploads and frees a layer again and again, and most of that was memory management: the page faults
// of a fresh 4 MB block (1 ms), cudaMalloc and cudaFree of 18 MB (0.45 and 0.55 ms).  512 x 512 x 27 at 0.28 kept, packed,
// uploaded, read back and freed: 4.9 -> 2.6 ms (2.0 since).
// Bounds: at most kMost bytes in all, no block over half of that; a request that finds nothing that fits gives every kept
// block of its kind back to the system first, so that blocks of sizes no longer asked for do not stay.
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
    std::vector<void*> gone;
    void* p = nullptr;
    {
      std::lock_guard<std::mutex> lock(mu_);
      for (size_t i = 0; i < kept_.size(); ++i)
        if (kept_[i].device == device && kept_[i].bytes >= bytes && kept_[i].bytes - bytes <= bytes / 4) {
          p = kept_[i].p;
          out_[p] = kept_[i];
          total_ -= kept_[i].bytes;
          kept_.erase(kept_.begin() + long(i));
          break;
        }
      if (!p) drop_locked(gone);
    }
    for (void* g : gone) release_(g);
    return p;
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
  // Keeps a block or releases it.
  void give(void* p) noexcept {
    if (!p) return;
    {
      std::lock_guard<std::mutex> lock(mu_);
      auto it = out_.find(p);
      if (it != out_.end()) {
        const Block b = it->second;
        out_.erase(it);
        if (total_ + b.bytes <= kMost) {
          kept_.push_back(b);
          total_ += b.bytes;
          return;
        }
      }
    }
    release_(p);
  }

 private:
  struct Block { void* p; size_t bytes; int device; };
  void drop_locked(std::vector<void*>& gone) {
    for (const Block& b : kept_) gone.push_back(b.p);    // all of them, or none if it throws
    kept_.clear();
    total_ = 0;
  }
  void (*release_)(void*);
  std::mutex mu_;
  std::vector<Block> kept_;
  std::unordered_map<void*, Block> out_;
  size_t total_ = 0;
};

}  // namespace rt3d
