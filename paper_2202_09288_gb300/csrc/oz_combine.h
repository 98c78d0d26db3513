// oz_combine.h -- the exact integer combination of a tile entry's seven diagonal sums, for the FP64
// tensor-core kernels and, without CUDA, for its CPU test.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define OZ_HD __host__ __device__ __forceinline__
#else
#define OZ_HD inline
#endif

namespace chol {

// W = V_hi 2^17 + round(V_lo / 2^7) of the seven diagonals, V_hi = sum_{d<4} D_d 2^(8(3-d)),
// V_lo = sum_{d>=4} D_d 2^(8(6-d)) (|D_d| <= (d+1) 2^21 at K = 128, so |W| < 1.01 2^62).  Diagonals 2
// to 6 may exceed 2^22 and come as integers (oz_int), d_3 2^17 and d_2 2^25 as 32 x 32 -> 64-bit
// multiply-adds; 0 and 1 as offset bits f_d = 0x4B400000 + D_d, whose offsets are not subtracted one
// by one: f_1 2^33 + f_0 2^41 are in the high word alone, and kOzHiBias removes them (modulo 2^32).
constexpr uint32_t kOzHiBias = 0u - 0x4B400000u * 2u - 0x4B400000u * 512u;

OZ_HD long long oz_low(int d4, int d5, int d6) {
  long long v = (long long)d5 * 256 + (d6 + 64);
  v = (long long)d4 * 65536 + v;
  return v >> 7;  // round(V_lo / 2^7), half up
}

OZ_HD long long oz_high(long long lo, uint32_t f0, uint32_t f1, int d2, int d3) {
  long long w = (long long)d3 * 131072 + lo;
  w = (long long)d2 * 33554432 + w;
  return (long long)((unsigned long long)w + ((unsigned long long)(f1 * 2u + f0 * 512u + kOzHiBias) << 32));
}

}  // namespace chol
