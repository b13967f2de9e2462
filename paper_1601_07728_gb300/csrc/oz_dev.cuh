// FP64 products on the FP16 tensor cores by exact splitting (the scheme of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with FP16 tensor
// products as in Mukunoki, Ozaki, Ogita and Imamura, ISC 2020).
//
// A row of an operand is scaled by a power of two to |y| < 1 and written as
// seven balanced base-256 digits, y = sum_i d_i 2^(-7-8i), |d_i| <= 128, i < 7:
// 55 bits below the row's largest entry (the 53 of FP64 and two guard bits at
// the top; eight digits: 2^-64 of the largest).  A digit is an integer that FP16 holds
// exactly, and a sum of fewer than 2^24 / 2^14 products of two digits is exact in
// the FP32 accumulators.  Digit
// products (i, j) of equal s = i + j share an accumulator; 128 K elements
// of up to seven products reach at most 7 * 128 * 2^14 < 2^24 (fewer products:
// more elements), after which the accumulators are drained into integers.
// Products of s = 7 are formed as well: of the rest, 2^-8 of that, none.  The
// only roundings are then the one of each operand entry at 2^-56 of its row's
// largest and the final conversion.
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

// f = round(x 2^(55-e)) + 0x80808080808080: each byte of f is a digit + 128 (the
// leading one with its carry above).  Integer arithmetic: at two FP64
// operations per SM and clock the FP64 pipe would take longer than HBM.  An
// entry far below the row's scale (every zero among them) shifts out to 0;
// e >= -960, or e = 0 for a row that counts as zero.
struct oz_fix {
  uint32_t lo, hi;
};
__device__ __forceinline__ oz_fix oz_fixed(double x, int e) {
  const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
  // |x| 2^(56-e) = (mantissa << 3) >> r with the leading bit of the mantissa at 52
  int r = 1022 + e - (int)((xh >> 20) & 0x7ffu);
  r = max(0, min(r, 63));   // below 0 only in rows flagged out of range
  uint32_t h = __funnelshift_l(xl, (xh & 0xfffffu) | 0x100000u, 3), l = xl << 3;
  if (r & 32) {
    l = h;
    h = 0;
  }
  l = __funnelshift_r(l, h, r);
  h >>= r & 31;
  // (v + 1 + 2 * 0x80808080808080) >> 1 rounds v / 2 to the nearest; with the
  // complement ~v = -v - 1 of a negative entry the same sum rounds -v / 2
  const uint32_t s = (uint32_t)((int)xh >> 31);
  const unsigned long long t = (((unsigned long long)(h ^ s) << 32) | (l ^ s)) + 0x0101010101010101ull;
  oz_fix f;
  f.lo = __funnelshift_r((uint32_t)t, (uint32_t)(t >> 32), 1);
  f.hi = (uint32_t)(t >> 32) >> 1;
  return f;
}

// |x| 2^-e as FP32, rounded down (0 below 2^-126): integer arithmetic as above
__device__ __forceinline__ float oz_unit(double x, int e) {
  const uint32_t xh = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  const int f = (int)(xh >> 20) - e - (1023 - 127);
  return f <= 0 ? 0.f : __uint_as_float(((uint32_t)min(f, 254) << 23) | ((xh & 0xfffffu) << 3));
}

__device__ __forceinline__ float oz_unit_square(double2 v, int e) {   // |v|^2 in units of 2^2e
  const float x = oz_unit(v.x, e), y = oz_unit(v.y, e);
  return x * x + y * y;
}
// (FP64 compares would run at 2 per SM and clock)
__device__ __forceinline__ bool oz_nonzero(double2 v) { return (oz_key(v.x) | oz_key(v.y)) != 0; }

// Which sums the digits may stand for.  With every entry held to 2^-56 of its
// row's scale, the error of a sum over k is about 0.58 * 2^-56 (|a|^2 + |b|^2)^1/2
// in units of the two scales (|.| the norms of the two rows there), whatever the
// sum itself is: where one row is large the other may be small throughout, and
// FP64 products keep the digits that are lost here.  So the magnitudes' sum
// S = sum |a_k| |b_k| is taken along from the leading digits (entries below
// 2^-8 of their row's scale count as zero, so that S is rather too small), and
// a sum is accepted where the error is below 2^-53 S, one rounding of it:
// S >= 0.0725 (|a|^2 + |b|^2)^1/2.  (With all K roundings of one sign it is at
// most K^1/2 2^-53 S, within the K 2^-53 S of an FP64 sum.)  The rest is summed
// on the FP64 pipe.  Rows
// of n normal random entries reach about 0.6 n / (r_a r_b) against a limit of
// 0.1 sqrt(n) (1 / r_a + 1 / r_b), r = 3..8 their scale over their deviation.
__device__ __forceinline__ bool oz_accept(float s, float norm_a, float norm_b) {
  return s >= 0.1f * (norm_a + norm_b);
}

// the same to 63 bits as eight digits, d[0] the leading one
__device__ __forceinline__ void oz_digits8(double x, int e, int* d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  // |x| 2^(63-e) = (mantissa << 10) >> r with the leading bit of the mantissa at 52
  const int r = max(0, 1022 + e - (int)((b >> 52) & 0x7ff));
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  long long v = r <= 10 ? (long long)(m << (10 - r)) : r < 73 ? (long long)((m + (1ull << (r - 11))) >> (r - 10)) : 0;
  if ((long long)b < 0) v = -v;
#pragma unroll
  for (int i = 7; i > 0; --i) {
    d[i] = (int)(signed char)(v & 0xff);
    v = (v - d[i]) >> 8;
  }
  d[0] = (int)v;
}

// digit i (0 = leading) of two entries as packed FP16: the bytes b become
// 0x6400 | b = 1024 + digit + 128, less 1152
__device__ __forceinline__ uint32_t oz_digit2(oz_fix f0, oz_fix f1, int i) {
  uint32_t w;
  if (i == 0) {
    w = (__byte_perm(f0.hi, f1.hi, 0x7632) & 0x01ff01ffu) | 0x64006400u;   // nine bits: 256 for the digit 128
  } else {
    const int b = OZ_S - 1 - i;   // byte of the 64-bit word
    const uint32_t sel = (uint32_t)((b & 3) * 0x1111 + 0x4400);
    w = (__byte_perm(b >= 4 ? f0.hi : f0.lo, b >= 4 ? f1.hi : f1.lo, sel) & 0x00ff00ffu) | 0x64006400u;
  }
  const uint32_t c = 0x64806480u;   // 1152 twice
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&c));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// block-wide maximum (blockDim.x <= 256); every thread returns it
__device__ unsigned block_max(unsigned v) {
  __shared__ unsigned wm[8];
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned m = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, wm[w]);
  return m;
}

// {norm, 2^1/2 of the number of entries} of a row from every thread's sum of
// squares and count (blockDim.x <= 256); for thread 0
__device__ float2 block_norm(float sq, int count) {
  __shared__ float ws[8];
  __shared__ int wc[8];
  for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
  count = __reduce_add_sync(0xffffffffu, count);
  if ((threadIdx.x & 31) == 0) {
    ws[threadIdx.x >> 5] = sq;
    wc[threadIdx.x >> 5] = count;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      sq += ws[w];
      count += wc[w];
    }
  return make_float2(sqrtf(sq), sqrtf(2.f * (float)count));
}

// a read-only load that stays where it is written: the compiler otherwise sinks
// the next block's loads behind the waits, to their use
__device__ __forceinline__ double2 load_in_place(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

}  // namespace
