// Threads of a plane (or of a 2D grid) walk its nodes, or node pairs, in one run,
// so that rows shorter than a block, or of a length that blocks do not divide,
// leave no threads idle.
#pragma once

#include <stdint.h>

namespace lbm {

// A row length and its reciprocal, floor(2^32 / n) (0 for n = 1).
struct RowLength {
  uint32_t n, inv;
};
inline RowLength row_length(int64_t n) {
  return RowLength{(uint32_t)n, n > 1 ? (uint32_t)(((uint64_t)1 << 32) / (uint64_t)n) : 0u};
}
// q / n, and the remainder
__device__ __forceinline__ uint32_t divide(uint32_t q, RowLength r, uint32_t& rest) {
  uint32_t d = r.inv ? __umulhi(q, r.inv) : q;
  rest = q - d * r.n;
  if (rest >= r.n) rest -= r.n, ++d;  // the reciprocal is rounded down
  return d;
}
// Entry q of the run: row y and position i in it; false past the last row.
__device__ __forceinline__ bool row_of(uint32_t q, RowLength r, int ny, int& i, int& y) {
  uint32_t rest;
  y = (int)divide(q, r, rest);
  i = (int)rest;
  return y < ny;
}

// The compiler does not know these values to be what they were: what it computed
// from them before is computed again after, instead of being kept in registers.
__device__ __forceinline__ void forget(int& x, int& y, int& z) { asm volatile("" : "+r"(x), "+r"(y), "+r"(z)); }
__device__ __forceinline__ void forget(int& x, int& y) { asm volatile("" : "+r"(x), "+r"(y)); }

}  // namespace lbm
