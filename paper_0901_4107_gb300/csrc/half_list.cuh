// Places in the tessellation's list of half-faces.
#pragma once

#include <stdint.h>

namespace amm {
namespace vor {

// Where a run of m half-faces taken at count `at` lies in a list of cap places; -1: past
// its end.  The count runs on past the capacity (every run is added, so that the last
// value is the room the build needs), and a list may hold more than 2^32 half-faces:
// 15.6 a cell in 3D, n up to 2^30.  64 bits cannot wrap (2^30 cells of at most 64 + 64).
__host__ __device__ inline int64_t half_place(unsigned long long at, int m, int64_t cap) {
  return at + (unsigned long long)m <= (unsigned long long)cap ? (int64_t)at : -1;
}

// the capacity that a build with `used` half-faces is repeated with; 0: the list held them
inline int64_t half_more(unsigned long long used, int64_t cap) {
  return used <= (unsigned long long)cap ? 0 : (int64_t)used + 1024;
}

}  // namespace vor
}  // namespace amm
