// Which of the caller's buffers kernels may read and write in place (the entry points
// get bare pointers).  No CUDA types here: the rule is tested on the host.
#pragma once
#include <cstddef>
#include <cstdint>

namespace egpe {

// What the driver says of a pointer: the address under which kernels of the current
// device reach it (0: they do not, e.g. memory of a device without peer access, or host
// memory that is not registered), and the allocation it lies in.
struct PtrFacts {
  uint64_t device_ptr = 0, range_start = 0;
  size_t range_size = 0;
};

// Kernels take `bytes` at p as they are when they reach them under that address, in one
// allocation, aligned to an element.  Everything else goes through a copy, which the
// runtime makes from any memory and refuses where there is none.
inline bool in_place(const PtrFacts& f, uint64_t p, size_t bytes, size_t align) {
  return p != 0 && p % align == 0 && f.device_ptr == p && f.range_start != 0 && p >= f.range_start &&
         f.range_size >= bytes && p - f.range_start <= f.range_size - bytes;
}

}  // namespace egpe
