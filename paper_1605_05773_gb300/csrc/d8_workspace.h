// d8_workspace.h -- a context's device workspace: one block, grown on demand.
// (Host code without CUDA calls of its own, so that it runs against any
// allocator.)
#pragma once
#include <cstddef>
#include <cstdint>

namespace d8 {

struct Workspace {
  void* p = nullptr;
  size_t bytes = 0;
  size_t refused = SIZE_MAX;  // sizes from here on found no room beside or instead of the present block

  // At least `need` bytes, `want` of them if there is room; false if there is
  // no room for `need` (the block is gone then).  A block that holds `need` is
  // given up for a larger one only once that is there, and a size that found no
  // room is not asked for again while the block stays: a call that can do with
  // `need` then neither allocates nor waits.
  // Mem: void* alloc(size_t) (null: no room); void release(void*), which waits
  // for the work that may still use the block.
  template <class Mem>
  bool ensure(Mem& mem, size_t want, size_t need) {
    if (bytes >= want || (bytes >= need && want >= refused)) return true;
    if (bytes >= need) {
      void* q = mem.alloc(want);
      if (!q) {
        refused = want;
        return true;
      }
      if (p) mem.release(p);
      p = q;
      bytes = want;
      return true;
    }
    if (p) mem.release(p);
    p = nullptr;
    bytes = 0;
    refused = SIZE_MAX;
    size_t n = want;
    p = mem.alloc(n);
    if (!p && need < want) {
      refused = want;
      n = need;
      p = mem.alloc(n);
    }
    if (p) bytes = n;
    return p != nullptr;
  }
};

}  // namespace d8
