// A block-wide sort, one value per thread.
#pragma once

namespace xs {

// Sorts in descending order over the first n threads (rounded up to a power of
// two of at least 32; the others' values do not matter), a bitonic network
// through shuffles and, between warps, s_x ([blockDim]).  Every thread of the
// block calls it.  Returns the thread's value; s_x holds every thread's, for
// the whole block to read.
__device__ __forceinline__ unsigned long long block_sort_desc(unsigned long long v, int n,
                                                              unsigned long long *s_x) {
  const int tid = threadIdx.x;
  for (int k = 2; k < 2 * n || k <= 32; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      unsigned long long o;
      if (j >= 32) {
        __syncthreads();
        s_x[tid] = v;
        __syncthreads();
        o = s_x[tid ^ j];
      } else {
        o = __shfl_xor_sync(0xffffffffu, v, j);
      }
      const bool larger = ((tid & j) == 0) == ((tid & k) == 0);
      v = larger == (v > o) ? v : o;
    }
  }
  __syncthreads();  // a slower warp may still read what the last exchange left in s_x
  s_x[tid] = v;
  __syncthreads();
  return v;
}

}  // namespace xs
