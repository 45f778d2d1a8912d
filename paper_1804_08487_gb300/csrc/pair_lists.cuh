// Lists of the same items, two to an array of `cap` places: list 2i from the
// front of array i, list 2i + 1 from its back.  Every item is in one list and
// an array has a place for each, so the two never meet.  Plain C++ apart from
// the qualifiers, so that it also compiles for the host.
#pragma once
#include <cstdint>

namespace cb {

__host__ __device__ inline int64_t pair_place(int list, int64_t i, int64_t cap) {
  return (list >> 1) * cap + ((list & 1) ? cap - 1 - i : i);
}

}  // namespace cb
