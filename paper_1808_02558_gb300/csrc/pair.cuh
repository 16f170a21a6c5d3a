// Packed FP32 arithmetic on pairs of values in 64-bit registers (sm_100 and later).
#pragma once

namespace qp {

// d = a b + d
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

}  // namespace qp
