// zmc_pinned.h — a bounded free list of page-locked buffers.
#pragma once

#include <algorithm>
#include <cstddef>
#include <mutex>
#include <vector>

namespace zmc {

struct PinnedBuf {
  char* p = nullptr;
  size_t bytes = 0;
};

// Buffers kept for reuse across calls, the `keep` largest of those given back.  Each
// call holds its buffer for its duration, so concurrent calls never share one.  Source
// has `static int get(void**, size_t)` (0 or an error) and `static void put(void*)`.
template <class Source>
class PinnedPool {
 public:
  explicit PinnedPool(size_t keep) : keep_(keep) {}

  // The smallest kept buffer of at least `bytes`, or a new one; 0 or the source's error.
  int take(size_t bytes, PinnedBuf* out) {
    {
      std::lock_guard<std::mutex> lk(mu_);
      auto best = free_.end();
      for (auto it = free_.begin(); it != free_.end(); ++it)
        if (it->bytes >= bytes && (best == free_.end() || it->bytes < best->bytes)) best = it;
      if (best != free_.end()) {
        *out = *best;
        free_.erase(best);
        return 0;
      }
    }
    void* p = nullptr;
    const int error = Source::get(&p, bytes);
    if (error == 0) *out = {static_cast<char*>(p), bytes};
    return error;
  }

  void give(PinnedBuf b) {
    if (!b.p) return;
    {
      std::lock_guard<std::mutex> lk(mu_);
      free_.push_back(b);
      if (free_.size() <= keep_) return;
      auto it = std::min_element(
          free_.begin(), free_.end(),
          [](const PinnedBuf& x, const PinnedBuf& y) { return x.bytes < y.bytes; });
      b = *it;
      free_.erase(it);
    }
    Source::put(b.p);
  }

 private:
  const size_t keep_;
  std::mutex mu_;
  std::vector<PinnedBuf> free_;
};

}  // namespace zmc
