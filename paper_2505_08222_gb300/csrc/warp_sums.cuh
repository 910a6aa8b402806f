// Warp-level column sums of the tensor-core epilogues.
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

}  // namespace ut
