// Sums over the 32 lanes of a warp of N values per lane (N a power of two).
//
// A butterfly per value costs 5 shuffles and 5 additions each, in every lane: 5 N of both.  Here the
// lanes halve the values they keep at every step (a lane keeps the half that its bit selects, sends
// the other half and adds what it receives): N/2 + N/4 + ... additions, and plain butterfly steps
// only once one value is left: 9 instead of 40 for N = 8, 62 instead of 320 for N = 64.  The additions
// of one value pair the lanes exactly as the butterfly does (xor 16, 8, 4, 2, 1), so the sums are
// bitwise the butterfly's.  It matters most in FP64, where a warp-wide addition takes 16 cycles of
// the SM's FP64 units.
#pragma once

#include <cuda_runtime.h>

namespace bddc {

// On return v[0 .. max(1, N / 32) - 1] holds the sums of the values lane_sum_index<N>(lane) + k; with
// N < 32 groups of 32 / N consecutive lanes hold the same sum (the first of them is the one to write).
template <int N, int OFF = 16, typename T>
__device__ __forceinline__ void lane_sums(T* v, int lane) {
  if constexpr (OFF > 0) {
    if constexpr (N > 1) {
      const bool up = (lane & OFF) != 0;
#pragma unroll
      for (int k = 0; k < N / 2; ++k) {
        const T send = up ? v[k] : v[k + N / 2];
        const T keep = up ? v[k + N / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
      }
      lane_sums<N / 2, OFF / 2>(v, lane);
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], OFF);
      lane_sums<1, OFF / 2>(v, lane);
    }
  }
}

template <int N>
__device__ __forceinline__ int lane_sum_index(int lane) {
  return N >= 32 ? lane * (N / 32) : lane / (32 / N);
}

template <int N>
__device__ __forceinline__ bool lane_sum_writer(int lane) {
  return N >= 32 || lane % (32 / N) == 0;
}

}  // namespace bddc
