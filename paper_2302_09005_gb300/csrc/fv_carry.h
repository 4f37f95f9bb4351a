// fv_carry.h -- the two buffers in which fv_run_steps carries primitives from
// step to step: grown, never shrunk, in the library's own form (`full`
// elements each, a third more than the documented one in 3D) or, where
// memory does not allow that, in the documented form (`doc` elements).  Host
// code; the allocator is the caller's.
#pragma once

#include <stdint.h>

namespace fv {

struct CarryBuffers {
  void* p[2] = {nullptr, nullptr};
  int64_t cap = 0;   // elements of each
  bool doc = false;  // sized for the documented form: the own one did not fit
};

// Whether the buffers must grow for a run that needs `full` or `doc`
// elements.  Once the own form did not fit, the documented one suffices.
inline bool carry_must_grow(const CarryBuffers& b, int64_t full, int64_t doc) {
  return full > b.cap && !(b.doc && doc <= b.cap);
}

enum class CarryAlloc { Ok, NoMemory, Error };

// Replaces the buffers: alloc(&p, elements) returns a CarryAlloc, release(p)
// frees.  On failure the handle keeps none.
template <typename Alloc, typename Release>
inline CarryAlloc carry_grow(CarryBuffers& b, int64_t full, int64_t doc, const Alloc& alloc,
                             const Release& release) {
  auto drop = [&] {
    for (void*& p : b.p) {
      if (p) release(p);
      p = nullptr;
    }
    b.cap = 0;
  };
  CarryAlloc r = CarryAlloc::NoMemory;
  for (const int64_t need : {full, doc}) {
    drop();
    r = CarryAlloc::Ok;
    for (void*& p : b.p)
      if (r == CarryAlloc::Ok) r = alloc(&p, need);
    if (r == CarryAlloc::Ok) {
      b.cap = need;
      b.doc = need < full;
    }
    if (r != CarryAlloc::NoMemory) break;
  }
  if (r != CarryAlloc::Ok) drop();
  return r;
}

}  // namespace fv
