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
// bytes in all: beyond that, blocks of the class that has gone unused longest
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
    const int c = size_class(bytes);
    Kept& k = kept_of_[c];
    k.used = ++clock_;
    if (!k.blocks.empty()) {
      *p = k.blocks.back();
      k.blocks.pop_back();
      kept_ -= class_bytes(c);
      return 0;
    }
    int e = mem.alloc(p, class_bytes(c));
    if (e != 0 && kept_ != 0) {
      drop_all(mem);
      e = mem.alloc(p, class_bytes(c));
    }
    if (e == 0) {
      try {
        class_of_[*p] = c;
      } catch (...) {   // no host memory to remember it by: given back like any other
      }
    }
    return e;
  }

  template <class Mem>
  void give(Mem mem, void* p) {
    const auto it = class_of_.find(p);
    if (it == class_of_.end()) {   // one that is not kept
      mem.free(p);
      return;
    }
    Kept& k = kept_of_[it->second];
    const size_t size = class_bytes(it->second);
    k.used = ++clock_;
    while (kept_ + size > kKeep && drop_oldest(mem)) {
    }
    try {
      k.blocks.push_back(p);
      kept_ += size;
    } catch (...) {
      class_of_.erase(p);
      mem.free(p);
    }
  }

  // Every kept block, when the stream is idle and nothing more is taken.
  template <class Free>
  void release(Free free) {
    for (Kept& k : kept_of_) {
      for (void* p : k.blocks) free(p);
      k.blocks.clear();
    }
    class_of_.clear();
    kept_ = 0;
  }

  size_t kept() const { return kept_; }

 private:
  struct Kept {
    std::vector<void*> blocks;
    uint64_t used = 0;   // clock_ when a block of this class was last taken or given back
  };
  // Class 4 e + q holds blocks of up to (5 + q) * 256 * 2^e bytes, q = 0 .. 3;
  // class 0 those of up to 1280.
  static constexpr int kClasses = 64;
  static size_t class_bytes(int c) { return (size_t)(5 + c % 4) << (8 + c / 4); }
  static int size_class(size_t bytes) {
    int e = 0;
    while (((size_t)8 << (8 + e)) < bytes) ++e;
    const size_t step = (size_t)1 << (8 + e);
    const int q = (int)((bytes + step - 1) >> (8 + e)) - 5;
    return 4 * e + (q < 0 ? 0 : q);
  }
  // A block of the class unused longest goes back to the pool; false: none is kept.
  template <class Mem>
  bool drop_oldest(Mem mem) {
    int oldest = -1;
    for (int c = 0; c < kClasses; ++c)
      if (!kept_of_[c].blocks.empty() && (oldest < 0 || kept_of_[c].used < kept_of_[oldest].used)) oldest = c;
    if (oldest < 0) return false;
    void* p = kept_of_[oldest].blocks.back();
    kept_of_[oldest].blocks.pop_back();
    kept_ -= class_bytes(oldest);
    class_of_.erase(p);
    mem.free(p);
    return true;
  }
  template <class Mem>
  void drop_all(Mem mem) {
    while (drop_oldest(mem)) {
    }
  }

  Kept kept_of_[kClasses];
  std::unordered_map<void*, int> class_of_;   // of every block that will be kept when given back
  size_t kept_ = 0;
  uint64_t clock_ = 0;
};

}  // namespace adapm
