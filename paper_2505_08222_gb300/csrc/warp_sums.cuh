// Warp-level sums of many rows or columns at once.
#pragma once

#include <cuda_runtime.h>

namespace ut {

// Column sums of v[16] over the warp's 32 rows: lane i returns column i % 16
// (each exchange halves the columns a lane still carries: 16 shuffles instead
// of five per column).
__device__ __forceinline__ float colsum16(const float (&v)[16]) {
  const int lane = threadIdx.x & 31;
  float a[8], b[4], c[2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
    a[i] = ((lane & 8) ? v[i + 8] : v[i]) + __shfl_xor_sync(0xffffffffu, (lane & 8) ? v[i] : v[i + 8], 8);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    b[i] = ((lane & 4) ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, (lane & 4) ? a[i] : a[i + 4], 4);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    c[i] = ((lane & 2) ? b[i + 2] : b[i]) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? b[i] : b[i + 2], 2);
  const float d = ((lane & 1) ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, (lane & 1) ? c[0] : c[1], 1);
  return d + __shfl_xor_sync(0xffffffffu, d, 16);
}

// Sums over the lanes of N rows at once (8 or 16; v[i]: this lane's term of row
// i), each by the tree of warp_sum: the halves exchange at distances 16, 8, 4,
// 2, 1, and while more than one row is left a lane keeps half of them.  Lane
// row_lane<N>(i) returns row i's sum, bit for bit what warp_sum gives, for 16
// (N = 16) or 9 shuffles instead of 5 N; what follows per row (a reciprocal
// square root) is then done once per lane and handed back by one shuffle.
template <int N>
__host__ __device__ constexpr int row_lane(int i) {
  return N == 16 ? ((i >> 3 & 1) << 4 | (i >> 2 & 1) << 3 | (i >> 1 & 1) << 2 | (i & 1) << 1)
                 : ((i >> 2 & 1) << 4 | (i >> 1 & 1) << 3 | (i & 1) << 2);
}
template <int N>
__device__ __forceinline__ float row_sums(const float (&v)[N]) {
  static_assert(N == 8 || N == 16, "rows");
  const int lane = threadIdx.x & 31;
  float a[N / 2], b[N / 4], c[N / 8];
#pragma unroll
  for (int i = 0; i < N / 2; ++i)
    a[i] = ((lane & 16) ? v[i + N / 2] : v[i]) + __shfl_xor_sync(0xffffffffu, (lane & 16) ? v[i] : v[i + N / 2], 16);
#pragma unroll
  for (int i = 0; i < N / 4; ++i)
    b[i] = ((lane & 8) ? a[i + N / 4] : a[i]) + __shfl_xor_sync(0xffffffffu, (lane & 8) ? a[i] : a[i + N / 4], 8);
#pragma unroll
  for (int i = 0; i < N / 8; ++i)
    c[i] = ((lane & 4) ? b[i + N / 8] : b[i]) + __shfl_xor_sync(0xffffffffu, (lane & 4) ? b[i] : b[i + N / 8], 4);
  float d;
  if constexpr (N == 16)
    d = ((lane & 2) ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? c[0] : c[1], 2);
  else
    d = c[0] + __shfl_xor_sync(0xffffffffu, c[0], 2);
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}
// Row i's value from the lane that row_sums left it in.
template <int N>
__device__ __forceinline__ float row_get(float v, int i) {
  return __shfl_sync(0xffffffffu, v, row_lane<N>(i));
}

}  // namespace ut
