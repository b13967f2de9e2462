// FP64 products on the FP16 tensor cores by exact splitting (the scheme of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with FP16 tensor
// products as in Mukunoki, Ozaki, Ogita and Imamura, ISC 2020).
//
// A row of an operand is scaled by a power of two to |y| < 1 and written as
// seven balanced base-256 digits, y = sum_i d_i 2^(-7-8i), |d_i| <= 128, i < 7:
// 55 bits below the row's largest entry (the 53 of FP64 and two guard bits at
// the top).  A digit is an integer that FP16 holds exactly, and a sum of fewer than 2^24 /
// 2^14 products of two digits is exact in the FP32 accumulators.  Digit
// products (i, j) of equal s = i + j < 7 share an accumulator; 128 K elements
// of up to seven products reach at most 7 * 128 * 2^14 < 2^24, after which the
// accumulators are drained into 64-bit integers.  The only roundings are the
// one of each operand entry at 2^-56 of its row's largest, the dropped
// products s >= 7 (of the same size) and the final conversion.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace {

constexpr int OZ_S = 7;          // digits per operand entry
constexpr int OZ_E_MAX = 400;    // largest |exponent| of a row scale; beyond it the FP64 kernels are used

// magnitude key of an FP64 value: orders like |x|, zero only for x = 0
__device__ __forceinline__ unsigned oz_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return ((unsigned)(b >> 32) & 0x7fffffffu) | ((unsigned)b != 0u ? 1u : 0u);
}
// exponent e with |x| < 2^e for every x whose key is at most `key` (0 for an
// all-zero row); *bad is set where the row holds Inf/NaN or its scale is out of range
__device__ __forceinline__ int oz_exponent(unsigned key, int* bad) {
  if (key == 0) return 0;
  const int e = (int)(key >> 20) - 1022;
  if (key >= 0x7ff00000u || e > OZ_E_MAX || e < -OZ_E_MAX) {
    *bad = 1;
    return 0;
  }
  return e;
}

// round(x 2^(55-e)) biased so that each byte of the result is a digit + 128
__device__ __forceinline__ unsigned long long oz_fixed(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
  int sh = ex - 1020 - e;   // at most 2 where |x| < 2^e
  if (sh > 2) sh = 2;       // only rows flagged out of range
  if (sh >= 0) {
    m <<= sh;
  } else {
    const int r = -sh > 62 ? 62 : -sh;
    m = (m + (1ull << (r - 1))) >> r;
  }
  const long long q = (long long)b < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)q + 0x80808080808080ull;
}

// digit i (0 = leading) of two entries as packed FP16; f from oz_fixed
__device__ __forceinline__ uint32_t oz_digit2(unsigned long long f0, unsigned long long f1, int i) {
  const int sh = 8 * (OZ_S - 1 - i);
  // the leading digit keeps the carry above its byte (128 at most)
  const uint32_t mask = i == 0 ? 0x1ffu : 0xffu;
  const uint32_t b0 = (uint32_t)(f0 >> sh) & mask, b1 = (uint32_t)(f1 >> sh) & mask;
  const uint32_t w = b0 | (b1 << 16) | 0x64006400u;   // FP16 1024 + digit + 128, exact
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w), __floats2half2_rn(1152.f, 1152.f));
  return *reinterpret_cast<const uint32_t*>(&d);
}

}  // namespace
