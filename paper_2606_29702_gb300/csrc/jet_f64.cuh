// Exact widening of FP32 sums for the FP64 sums across chunks.
#pragma once

#include <cuda_runtime.h>

namespace jet {

// Value-preserving float -> double on the integer pipe.  The FP64 pipe, which
// executes the conversion instruction, takes two lanes a clock per SM, and the
// weight gradients of every tile or chunk are converted; subnormals take the instruction.
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
  if (e == 0u && m != 0u) return (double)f;
  const unsigned ed = e == 0u ? 0u : e == 255u ? 2047u : e + 896u;
  return __hiloint2double((int)((b & 0x80000000u) | (ed << 20) | (m >> 3)), (int)(m << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

}  // namespace jet
