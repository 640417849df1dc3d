// Transposed warp sums shared by the kernels that reduce several values per
// warp.
#pragma once
#include <cuda_runtime.h>

namespace h2 {

// Transposed warp sum: every lane holds N values (N a power of two no larger
// than G, the width of an aligned lane group, a power of two <= 32).  At
// xor-distance G/2, G/4, ... each lane keeps half of its remaining values
// and adds its partner's copies of them, then plain steps finish: lane l
// ends with the group sum of value tsum_index<N, G>(l), after N - 1 + the
// remaining plain shuffles (instead of N log2 G for N separate sums).
template <int N, int G, typename T>
__device__ __forceinline__ T tsum(const T (&v)[N]) {
  if constexpr (N == 1) {
    T x = v[0];
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  } else {
    const bool up = threadIdx.x & (G / 2);
    T w[N / 2];
#pragma unroll
    for (int q = 0; q < N / 2; ++q) {
      const T mine = up ? v[q + N / 2] : v[q], other = up ? v[q] : v[q + N / 2];
      w[q] = mine + __shfl_xor_sync(0xffffffffu, other, G / 2);
    }
    return tsum<N / 2, G / 2, T>(w);
  }
}
template <int N, int G>
__device__ __forceinline__ int tsum_index(int lane) {
  int idx = 0;
#pragma unroll
  for (int n = N, g = G; n > 1; n >>= 1, g >>= 1)
    if (lane & (g / 2)) idx += n / 2;
  return idx;
}
// lanes holding a distinct tsum result: the first lane of each group of
// G / N lanes with equal index
template <int N, int G>
__device__ __forceinline__ bool tsum_leader(int lane) {
  return (lane & (G / N - 1)) == 0;
}
// the first lane holding the sum of value v
template <int N, int G>
__host__ __device__ constexpr int tsum_lane(int v) {
  int lane = 0;
  for (int n = N, g = G; n > 1; n >>= 1, g >>= 1)
    if (v & (n / 2)) lane |= g / 2;
  return lane;
}

}  // namespace h2
