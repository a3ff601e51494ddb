// Device memory of one context.
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstddef>
#include <vector>

#include "../../include/gpumap.h"

namespace gm {

// With the caller's allocator every buffer is an allocation of its own.
// Without, small buffers are cut from slabs (the first one sized for
// everything map_create needs); a piece of a slab that is given back is kept
// for the next request of about its size.  A buffer above a quarter of a later
// slab that fits neither a kept piece nor the rest of the newest slab is an
// allocation of its own, freed at once, so that slabs cost little memory (0.2-2
// % above 1 MB held).  A context holds some seventy buffers, and their
// allocation and release one by one was most of the cost of a small context,
// above all with several threads at it (a stream-ordered allocation takes a
// lock of the device): hierarchical multisection of an RGG of 2^17 vertices by
// 8 threads 38.5 -> 26.9 ms, 16 served jobs 33.3 -> 21.6 ms.
// A buffer that is put back may be handed out again at once, in the order of
// the context's stream: work on another stream that uses it (the partitioners
// of a hierarchical multisection read their parent's arrays from streams of
// their own) must have been waited for before.
struct DevMem {
  static constexpr size_t kSlabMax = 1 << 20;       // a later slab: 1/128 of what is held, up to this
  static constexpr size_t kSlabReserve = 64 << 20;  // a first slab of at most this size
  map_alloc_fn afn = nullptr;
  map_free_fn ffn = nullptr;
  void* user = nullptr;
  cudaStream_t st = nullptr;
  struct Block {
    void* p;
    size_t bytes;
    bool slab;  // cut from a slab
    bool used;  // handed out; else (slabs only) kept for a later request
  };
  std::vector<Block> blocks;  // the allocations handed out and every piece of a slab
  std::vector<Block> slabs;
  char* cur = nullptr;  // rest of the newest slab
  size_t cur_left = 0;
  size_t total = 0;
  size_t peak = 0;  // largest `total` so far

  void reserve(size_t bytes) {  // the first slab
    if (!afn && bytes <= kSlabReserve) add_slab((bytes + 255) & ~(size_t)255);
  }

  void* get(size_t bytes) {
    if (bytes == 0) bytes = 16;
    bytes = (bytes + 255) & ~(size_t)255;
    room(blocks, 2);
    if (!(afn && ffn)) {
      Block* best = nullptr;  // the smallest kept piece that is not much too large
      for (Block& b : blocks)
        if (!b.used && b.bytes >= bytes && b.bytes <= bytes + bytes / 4 + 4096 && (!best || b.bytes < best->bytes))
          best = &b;
      if (best) {
        best->used = true;
        return best->p;
      }
      const size_t slab = std::min<size_t>(kSlabMax, std::max<size_t>(256 << 10, total / 128));
      if (bytes <= cur_left || bytes < slab / 4) {
        if (bytes > cur_left) add_slab(slab);
        void* p = cur;
        cur += bytes;
        cur_left -= bytes;
        blocks.push_back({p, bytes, true, true});
        return p;
      }
    }
    void* p = raw(bytes);
    blocks.push_back({p, bytes, false, true});
    return p;
  }

  void put(void* p) noexcept {  // (called while failures are cleaned up: it allocates nothing)
    for (size_t i = 0; i < blocks.size(); i++) {
      Block& b = blocks[i];
      if (b.p != p || !b.used) continue;
      if (b.slab) {
        b.used = false;
        return;
      }
      raw_free(b.p, b.bytes);
      total -= b.bytes;
      b = blocks.back();
      blocks.pop_back();
      return;
    }
  }

  void release_all() noexcept {
    for (const Block& b : blocks)
      if (!b.slab) raw_free(b.p, b.bytes);
    for (const Block& s : slabs) raw_free(s.p, s.bytes);
    blocks.clear();
    slabs.clear();
    cur_left = 0;
    total = 0;
  }

  template <class T>
  T* make(size_t count) {
    return static_cast<T*>(get(count * sizeof(T)));
  }

 private:
  void* obtain(size_t bytes);  // from the device or the caller's allocator; throws
  void raw_free(void* p, size_t bytes) noexcept;

  static void room(std::vector<Block>& v, size_t more) {  // the next push_backs do not allocate
    if (v.capacity() - v.size() < more) v.reserve(2 * v.capacity() + more);
  }

  void* raw(size_t bytes) {
    void* p = obtain(bytes);
    total += bytes;
    peak = std::max(peak, total);
    return p;
  }

  void add_slab(size_t bytes) {
    room(slabs, 1);
    room(blocks, 2);  // the rest of the slab before, and the piece to come
    char* p = static_cast<char*>(raw(bytes));
    if (cur_left) blocks.push_back({cur, cur_left, true, false});
    slabs.push_back({p, bytes, false, true});
    cur = p;
    cur_left = bytes;
  }
};

}  // namespace gm
