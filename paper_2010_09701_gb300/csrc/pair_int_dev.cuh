// Conversions between FP64 and FP32 pairs (pair_dev.cuh) on the integer pipe. The conversion
// instructions and the FP64 subtraction of f2_from, and those of f2_to, issue at two results a clock
// per SM: four and three of them per value cost as much as 40 and 30 pair instructions.
#pragma once
#include "pair_dev.cuh"

namespace {

// x as a pair: h = x rounded to 24 bits, l the remainder rounded to 24 bits (the bits of f2_from)
__device__ __forceinline__ f2 f2_from_int(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  if (ex < 956 || ex > 1149) return ex == 0 ? f2{0.f, 0.f} : f2_from(x);   // l or h near the ends of FP32's range
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned top = (unsigned)((m + (1ull << 28) - 1 + ((m >> 29) & 1)) >> 29);   // 24 bits, ties to even (2^24 on a carry)
  const int rem = (int)((unsigned)m - (top << 29));                        // m - top 2^29, in [-2^28, 2^28]
  const unsigned sg = (unsigned)(b >> 32) & 0x80000000u;
  const float h = __uint_as_float(sg | ((((unsigned)ex - 896u) << 23) + (top - (1u << 23))));
  const float w = __uint_as_float(sg | ((unsigned)(ex - 948) << 23));      // 2^(ex - 1075) with the sign
  return f2{h, __fmul_rn(__int2float_rn(rem), w)};
}

__device__ __forceinline__ double widen_int(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xFF;
  if (e - 1u >= 254u) return (double)x;                                    // zero, subnormal, infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}
__device__ __forceinline__ double f2_to_int(f2 a) { return widen_int(a.h) + widen_int(a.l); }

}  // namespace
