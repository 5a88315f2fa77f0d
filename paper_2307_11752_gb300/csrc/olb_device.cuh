// olb_device.cuh -- small device helpers shared by the fluid and the scalar kernels.
#pragma once

#include <cuda_runtime.h>

namespace olb {

// (double)v by integer instructions.  The conversion instruction runs on the FP64 pipe
// like an addition (16 cycles of an SM per warp), which bounded the readout kernels:
// reading 128^3 FP32 populations took 150 us with it and takes 95 (HBM: 72); 256^3 FP16
// 1180 and 630.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  // exponents of 8 and 11 bits, biases 127 and 1023; no branch that leads to the
  // conversion instruction (it would be issued for every value)
  const bool sub = (__float_as_uint(v) & 0x7f800000u) == 0u;
  const unsigned b = __float_as_uint(sub ? v * 18446744073709551616.0f : v);  // 2^64: exact, normal or zero
  unsigned base = sub ? 0x38000000u - (64u << 20) : 0x38000000u;
  if ((b & 0x7f800000u) == 0x7f800000u) base = 0x70000000u;  // infinite or NaN
  if ((b << 1) == 0u) base = 0u;                             // zero
  return __hiloint2double((int)((b & 0x80000000u) | (((b >> 3) & 0x0fffffffu) + base)), (int)(b << 29));
}

// n / d for 0 <= n < 2^31 by one high multiplication (T. Granlund, P. Montgomery,
// "Division by invariant integers using multiplication", PLDI 1994).
struct FastDiv {
  unsigned d, m;
  int s;
  FastDiv() = default;
  explicit FastDiv(unsigned d_) : d(d_), m(0), s(0) {
    while ((1ull << s) < d) ++s;
    m = (unsigned)(((1ull << (31 + s)) + d - 1) / d);
  }
  __device__ __forceinline__ unsigned div(unsigned n) const { return s == 0 ? n : __umulhi(n, m) >> (s - 1); }
};

}  // namespace olb
