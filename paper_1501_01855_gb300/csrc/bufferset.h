// Buffers that grow together. Host code without CUDA, so that a failing allocator can be put in.
#pragma once
#include <stddef.h>

#include <initializer_list>

namespace ovl {

struct BufferSlot {
  void** p;
  size_t bytes;
};

// Release what the slots hold and allocate every one anew: alloc(void**, size_t) returns 0 or an
// error. When one cannot be had, all are released: every pointer is null (the caller sets its sizes
// to zero), so that a later call neither uses nor keeps a part of the set.
template <typename Alloc, typename Release>
int renew_all(std::initializer_list<BufferSlot> set, Alloc alloc, Release release) {
  auto drop = [&]() {
    for (const BufferSlot& b : set) {
      if (*b.p) release(*b.p);
      *b.p = nullptr;
    }
  };
  drop();
  for (const BufferSlot& b : set) {
    const int e = static_cast<int>(alloc(b.p, b.bytes));
    if (e != 0) {
      *b.p = nullptr;
      drop();
      return e;
    }
  }
  return 0;
}

}  // namespace ovl
