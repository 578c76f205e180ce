// Device blocks that their owners keep between calls, and allocations that may
// take them back.
//
// A block is used by one call of its owner at a time.  Between calls it lies
// idle, and the first allocation of the library that the device has no room
// for, for whichever handle and from whichever thread, frees every idle block
// and tries once more.  Dev supplies alloc(void **, size_t) -> bool and
// free(void *).
#pragma once
#include <algorithm>
#include <cstddef>
#include <mutex>
#include <vector>

namespace lbeh {

struct KeptBlock {
  void *p = nullptr;
  size_t bytes = 0;
};

template <class Dev> class KeptBlocks {
  std::mutex m;
  std::vector<KeptBlock *> idle;
  void free_block(KeptBlock &b) {
    if (b.p) Dev::free(b.p);
    b = KeptBlock{};
  }
  bool alloc_locked(void **p, size_t bytes) {
    if (Dev::alloc(p, bytes)) return true;
    if (!idle.empty()) {
      for (KeptBlock *b : idle) free_block(*b);
      idle.clear();
      if (Dev::alloc(p, bytes)) return true;
    }
    *p = nullptr;
    return false;
  }
  void unlist(KeptBlock &b) { idle.erase(std::remove(idle.begin(), idle.end(), &b), idle.end()); }

 public:
  bool alloc(void **p, size_t bytes) {
    std::lock_guard<std::mutex> l(m);
    return alloc_locked(p, bytes);
  }
  // the block for the owner's call, of at least `bytes`; null where there is no room
  void *take(KeptBlock &b, size_t bytes) {
    std::lock_guard<std::mutex> l(m);
    unlist(b);
    if (b.bytes < bytes) {
      free_block(b);
      if (alloc_locked(&b.p, bytes)) b.bytes = bytes;
    }
    return b.p;
  }
  // the call has ended, its work on the device too: idle up to `most` bytes, freed above
  void put(KeptBlock &b, size_t most) {
    std::lock_guard<std::mutex> l(m);
    if (b.bytes > most) free_block(b);
    else if (b.p) idle.push_back(&b);
  }
  void drop(KeptBlock &b) {
    std::lock_guard<std::mutex> l(m);
    unlist(b);
    free_block(b);
  }
};

}  // namespace lbeh
