// Pivot key of the FP64 Gauss-Jordan eliminations: |x| rounded to FP32, as the
// bits of that number, which order as the numbers.  Both kernels compare this
// key (k_gj_cluster as a float), so that they take the same pivots.
#pragma once
#include <cstdint>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace dqmc {

// The key of the double with the bits b where |x| rounds to a normal FP32
// number or infinity (ok), in integer arithmetic: the conversion instruction
// would take the FP64 pipe.  Round to nearest, ties to even.
__host__ __device__ __forceinline__ uint32_t gj_key_bits(uint64_t b, bool& ok) {
  b &= 0x7FFFFFFFFFFFFFFFull;
  const uint32_t E = static_cast<uint32_t>(b >> 52);
  ok = E > 896u && E < 1151u;
  b -= 896ull << 52;
  return static_cast<uint32_t>((b + 0x0FFFFFFFull + ((b >> 29) & 1ull)) >> 29);
}

}  // namespace dqmc
