// Integer slices of FP64 operands for the tensor-core FP64 contraction (tc_oz.cuh).
//
// The values of one operand row inside one chunk of 256 k share the scale 2^e, e the smallest
// exponent with max|x| < 2^e.  Each is rounded to the integer F = round(x 2^(63 - e)) (exact down
// to 2^-10 of the chunk's largest; fewer bits with fewer than the eight slices) and written in balanced base 256,
//   F = sum_{s=0..7} d_s 256^(7 - s),  |d_s| <= 128 (d_0: the remaining top part, |d_0| <= 128),
// each digit a BF16 number (integers up to 256 are exact).  Integer arithmetic throughout.
#pragma once
#include <stdint.h>

#include "oz_job.h"

namespace osv {
namespace oz {

__device__ __forceinline__ unsigned exp_field(double x) {
  return (unsigned)((__double_as_longlong(x) >> 52) & 0x7FF);
}

// BF16 bits of an integer |d| <= 128 (exact): the FP32 value by the 1.5 2^23 offset, its upper half.
__device__ __forceinline__ uint32_t bf16_of_int(int d) {
  return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f) >> 16;
}

// F of x for the chunk whose largest biased exponent field is emax (0 < emax < 2047).
__device__ __forceinline__ long long fixed63(double x, unsigned emax) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  if (ex == 0) return 0;
  const unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = 10 - ((int)emax - ex);          // |x| 2^(63-e) = mant 2^sh
  long long F;
  if (sh >= 0) F = (long long)(mant << sh);
  else if (sh > -54) F = (long long)((mant + (1ull << (-sh - 1))) >> -sh);
  else F = 0;
  return (bits >> 63) ? -F : F;
}

// Exponent code of a chunk from its largest exponent field.
__device__ __forceinline__ int chunk_exp(unsigned emax) {
  return emax == 0 ? EX_ZERO : (emax == 2047 ? EX_NAN : (int)emax - 1022);
}

// round(x 2^(T - e)) for NS slices, T = 7 + 8 (NS - 1) (63 for eight).  One place is left for the rounding before half
// a unit is added: F itself reaches 2^63 - 2^10, where that sum has no room.  The result 2^T has the top digit 128.
template <int NS>
__device__ __forceinline__ long long fixedn(double x, unsigned emax) {
  const long long F = fixed63(x, emax);
  constexpr int D = 8 * (NSL - NS);
  return D ? ((F >> (D > 0 ? D - 1 : 0)) + 1) >> 1 : F;
}

// Digit s (taken in the order s = NS - 1 .. 0) of two values, as a BF16 pair.
__device__ __forceinline__ uint32_t digit_pair(long long& f0, long long& f1, int s) {
  const int d0 = s ? (int)(signed char)(f0 & 255) : (int)f0, d1 = s ? (int)(signed char)(f1 & 255) : (int)f1;
  f0 = (f0 - d0) >> 8;
  f1 = (f1 - d1) >> 8;
  return bf16_of_int(d0) | (bf16_of_int(d1) << 16);
}

// The same for 32-bit fixed-point numbers (four slices).
__device__ __forceinline__ uint32_t digit_pair32(int& f0, int& f1, int s) {
  const int d0 = s ? (int)(signed char)(f0 & 255) : f0, d1 = s ? (int)(signed char)(f1 & 255) : f1;
  f0 = (f0 >> 8) + ((f0 >> 7) & 1);
  f1 = (f1 >> 8) + ((f1 >> 7) & 1);
  return bf16_of_int(d0) | (bf16_of_int(d1) << 16);
}

// One row-chunk held by a warp: lane l has elements k = 64 u + 2 l + {0, 1}, u = 0 .. 3 (zero past the
// end).  Writes the digits at dst + s * slice + k for k < kv and returns the exponent code.
template <int NS>
__device__ __forceinline__ int warp_slices(const double x[8], int kv, uint16_t* dst, size_t slice, int lane) {
  unsigned em = 0;
#pragma unroll
  for (int u = 0; u < 8; u++) em = max(em, exp_field(x[u]));
  em = __reduce_max_sync(0xffffffffu, em);
  const bool live = em != 0 && em != 2047;
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const int k = 64 * u + 2 * lane;
    if (k >= kv) continue;
    long long f0 = live ? fixedn<NS>(x[2 * u], em) : 0, f1 = live ? fixedn<NS>(x[2 * u + 1], em) : 0;
#pragma unroll
    for (int s = NS - 1; s >= 0; s--)   // k + 1 may be one past an odd K: still inside the padded row
      *reinterpret_cast<uint32_t*>(dst + s * slice + k) = digit_pair(f0, f1, s);
  }
  return chunk_exp(em);
}

}  // namespace oz
}  // namespace osv
