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
// (float)v, rounded to nearest even, by integer operations for the same reason.  Values that are no
// normal FP32 number after rounding (zeros and subnormal ones, overflow, non-finite) take the
// instruction.
__device__ __forceinline__ float narrow(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  const unsigned long long r = b - (896ull << 52) + 0x0fffffffull + ((b >> 29) & 1ull);  // exponent rebased, rounded
  const unsigned f = (unsigned)(r >> 29);
  if (b < (897ull << 52) || r >= (255ull << 52)) return (float)v;
  return __uint_as_float(f | ((unsigned)__double2hiint(v) & 0x80000000u));
}

}  // namespace fe
