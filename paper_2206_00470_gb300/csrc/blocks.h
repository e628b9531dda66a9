// Scratch blocks kept for reuse on one stream (host code, no CUDA).
#pragma once

#include <cstddef>
#include <cstdint>
#include <unordered_map>
#include <vector>

namespace adapm {

// A block given back is handed out again to later work of the same stream,
// whose order makes that safe (what other streams do with a block is waited
// for before it is given back).  Taking and giving back are host bookkeeping,
// where a pool allocation and its free are two calls into the driver (0.7 to 1
// us each, six pairs a push).  Sizes are rounded up to one of four steps per
// power of two.  Blocks above kLargest are not kept, and not more than kKeep
// bytes in all: beyond that, blocks of the size that has gone unused longest
// go back to the pool, which the context owns and destroys.  An allocation
// that fails gives every kept block back to the pool, where their memory
// serves any size, and is tried once more.
//
// Mem is the pool on the cache's stream: int alloc(void** p, size_t bytes),
// 0 for success, and void free(void* p), both in the stream's order.
class BlockCache {
 public:
  static constexpr size_t kLargest = 64u << 20, kKeep = 512u << 20;

  // capturing: the stream records a graph.  Its blocks come from the pool and
  // go back to it inside the graph (a kept block would outlive its allocation
  // node, or be handed to other work while the graph runs).  What a recorded
  // call gives back it took itself: blocks that outlive a call are an intent's,
  // and intents and advances are refused then.
  template <class Mem>
  int take(Mem mem, size_t bytes, bool capturing, void** p) {
    if (bytes > kLargest || capturing) {
      const int e = mem.alloc(p, bytes);
      if (e == 0 || capturing || kept_ == 0) return e;
      drop_all(mem);
      return mem.alloc(p, bytes);
    }
    const size_t size = round_up(bytes);
    const auto it = kept_of_.find(size);
    if (it != kept_of_.end()) {
      it->second.used = ++clock_;
      if (!it->second.blocks.empty()) {
        *p = it->second.blocks.back();
        it->second.blocks.pop_back();
        kept_ -= size;
        return 0;
      }
    }
    int e = mem.alloc(p, size);
    if (e != 0 && kept_ != 0) {
      drop_all(mem);
      e = mem.alloc(p, size);
    }
    if (e == 0) {
      try {
        size_[*p] = size;
      } catch (...) {   // no host memory to remember it by: given back like any other
      }
    }
    return e;
  }

  template <class Mem>
  void give(Mem mem, void* p) {
    const auto it = size_.find(p);
    if (it == size_.end()) {   // one that is not kept
      mem.free(p);
      return;
    }
    const size_t size = it->second;
    try {
      Kept& k = kept_of_[size];
      k.used = ++clock_;
      while (kept_ + size > kKeep && drop_oldest(mem)) {
      }
      k.blocks.push_back(p);
      kept_ += size;
    } catch (...) {
      size_.erase(p);
      mem.free(p);
    }
  }

  // Every kept block, when the stream is idle and nothing more is taken.
  template <class Free>
  void release(Free free) {
    for (auto& k : kept_of_)
      for (void* p : k.second.blocks) free(p);
    kept_of_.clear();
    size_.clear();
    kept_ = 0;
  }

  size_t kept() const { return kept_; }

 private:
  struct Kept {
    std::vector<void*> blocks;
    uint64_t used = 0;   // clock_ when a block of this size was last taken or given back
  };
  static size_t round_up(size_t bytes) {
    if (bytes <= 1024) return 1024;
    size_t step = 256;
    while (step * 8 < bytes) step <<= 1;   // four steps between 4 * step and 8 * step
    return (bytes + step - 1) / step * step;
  }
  // A block of the size unused longest goes back to the pool; false: none is kept.
  template <class Mem>
  bool drop_oldest(Mem mem) {
    Kept* oldest = nullptr;
    size_t size = 0;
    for (auto& k : kept_of_) {
      if (k.second.blocks.empty() || (oldest && oldest->used <= k.second.used)) continue;
      oldest = &k.second;
      size = k.first;
    }
    if (!oldest) return false;
    void* p = oldest->blocks.back();
    oldest->blocks.pop_back();
    kept_ -= size;
    size_.erase(p);
    mem.free(p);
    return true;
  }
  template <class Mem>
  void drop_all(Mem mem) {
    while (drop_oldest(mem)) {
    }
  }

  std::unordered_map<size_t, Kept> kept_of_;   // by size (about a hundred sizes at most)
  std::unordered_map<void*, size_t> size_;     // of every block that will be kept when given back
  size_t kept_ = 0;
  uint64_t clock_ = 0;
};

}  // namespace adapm
