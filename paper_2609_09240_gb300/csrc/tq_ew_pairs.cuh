// tq_ew_pairs.cuh - which entries of the element-wise correction index are
// read as aligned 32-bit words (tq_ew.cu).
#pragma once
#include <cuda_runtime.h>

namespace tq {
namespace ew {

// Entry i of the index (16 bits) lies in half (i + odd) & 1 of word
// (i + odd) / 2, with odd = 1 where the index begins in the upper half of an
// aligned word.  The word of entry 0 then begins before the index, and the
// last entry's may end behind it: those halves may not be the caller's memory.
// Words hold the entries [odd, pairs_end) of `total`; a block's range is
// clamped into them (pairs_clamp), and the one or two other entries are read
// alone.  (The words of a clamped range lie wholly inside the index.)
__host__ __device__ __forceinline__ int pairs_end(int odd, int total) { return total - ((total + odd) & 1); }
__host__ __device__ __forceinline__ int pairs_clamp(int i, int odd, int end) {
  i = i > odd ? i : odd;
  return i < end ? i : end;
}
// Whether entry 0 (last: the last entry) is read alone.
__host__ __device__ __forceinline__ bool read_alone(bool last, int odd, int total) {
  return total > 0 && (last ? pairs_end(odd, total) < total : odd != 0);
}

}  // namespace ew
}  // namespace tq
