// Sorting a list of point indices by one thread, in place.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace vgicp {

__device__ __forceinline__ void insertion_sort(uint32_t* L, uint32_t c) {
  for (uint32_t a = 1; a < c; ++a) {
    const uint32_t x = L[a];
    int b = (int)a - 1;
    while (b >= 0 && L[b] > x) {
      L[b + 1] = L[b];
      --b;
    }
    L[b + 1] = x;
  }
}

// Lists of any length.  Roughly in order, they suit insertion while they are short; longer
// ones go through a heap, as insertion is quadratic and one thread's accesses follow one
// another (rebuild of a map whose points share a voxel: 4,000 points 201 -> 3.1 ms, 8,000
// 687 -> 6.8, 60,000 88 ms).
constexpr uint32_t kInsertionMax = 64;
static __device__ __noinline__ void sort_long(uint32_t* L, uint32_t c) {
  for (uint32_t built = c / 2, end = c; end > 1;) {
    uint32_t x, hole;
    if (built > 0) {  // the heap grows downwards to the root
      hole = --built;
      x = L[hole];
    } else {  // then gives its largest to the end
      x = L[--end];
      L[end] = L[0];
      hole = 0;
    }
    for (uint32_t child; (child = 2 * hole + 1) < end; hole = child) {
      uint32_t y = L[child];
      if (child + 1 < end && L[child + 1] > y) y = L[++child];
      if (y <= x) break;
      L[hole] = y;
    }
    L[hole] = x;
  }
}
__device__ __forceinline__ void sort_list(uint32_t* L, uint32_t c) {
  if (c <= kInsertionMax) insertion_sort(L, c);
  else sort_long(L, c);
}

}  // namespace vgicp
