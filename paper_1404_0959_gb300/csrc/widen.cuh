// widen.cuh -- FP32 <-> FP64 conversions that stay off the FP64 pipe.
#pragma once
#include <cuda_runtime.h>

namespace fe {

// (double)v by integer operations: the conversion instruction takes the time of about five FP64
// operations here (the sums of k_diag at 256^3 went from 2.50 to 1.91 ms without it).  Zeros, subnormal
// and non-finite values take the instruction.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (double)v;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

}  // namespace fe
