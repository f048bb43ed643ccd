// FP64 sums of products on the integer pipe.
//
// GB300 issues 2 FP64 FMAs per clock and SM against 27 32 x 32 -> 64-bit
// integer multiply-adds (measured: 0.60 against 7.9 T/s on one GPU), so the
// FP64 contractions here run in fixed point: a group of doubles is scaled by
// one power of two to integers X = x1 2^28 + x0 with |x0| <= 2^27 (centred
// digits), |X| < 2^57 (vectors) or < 2^59 (stored operators), and a product
// keeps three of its four digit products,
//   a x = a1 x1 2^56 + (a1 x0 + a0 x1) 2^28 + a0 x0,  |a0 x0| <= 2^54 dropped,
// each an exact 64-bit integer multiply-add: sums are exact (whatever their
// order) and rounded to a double once.  What is lost is the dropped term
// (2^-60 of the product of the two scales) and the operands' last bit (2^-57
// of their group's largest entry), below the 2^-53 that every single FP64
// addition of the same sum rounds off.
//
// Plain C++ apart from the decorations, so that a host test can compile it.
#pragma once

#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace mg {
namespace fx {

constexpr int kDigit = 28;      // bits of a low digit
constexpr int kVecBits = 57;    // |X| < 2^kVecBits for vectors
constexpr int kBadExp = 0x7ff;  // exponent field of Inf / NaN

FX_HD int64_t bits_of(double v) {
#if defined(__CUDA_ARCH__)
  return __double_as_longlong(v);
#else
  int64_t b;
  std::memcpy(&b, &v, 8);
  return b;
#endif
}

// exponent field (0 .. 2047) of a double: a value with field e < 2047 is
// below 2^(e - 1022)
FX_HD int exp_field(double v) { return (int)((bits_of(v) >> 52) & 0x7ff); }

// round toward zero of v 2^(BITS - (E - 1022)), BITS = 53 .. 62; |result| <
// 2^BITS for every v whose exponent field is at most E (1 <= E < 2047)
template <int BITS = kVecBits> FX_HD int64_t to_fixed(double v, int E) {
  const int64_t b = bits_of(v);
  int e = (int)((b >> 52) & 0x7ff);
  const uint64_t m = ((uint64_t)b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  if (e == 0) e = 1;
  // m 2^(e - E + BITS - 53): the mantissa left-aligned below the sign, then
  // one shift
  int s = E - e + 63 - BITS;
  if (s > 63) s = 63;
  const int64_t x = (int64_t)((m << 10) >> s);
  const int64_t sg = b >> 63;
  return (x ^ sg) - sg;
}

// centred digits of X: X = hi(X) 2^28 + lo(X), -2^27 <= lo < 2^27
FX_HD int digit_lo(int64_t X) { return (int)((uint32_t)X << 4) >> 4; }
FX_HD int digit_hi(int64_t X) { return (int)((X + (1 << (kDigit - 1))) >> kDigit); }

// the exponent u of a stored operator row's unit (entry = X 2^u): |X| < 2^58
// and sum |X| < 2^61 over the row's real and imaginary parts, so that a sum
// of a1 x1 over the row with |x1| <= 2^29 stays below 2^63
FX_HD int row_unit(int e_max, int e_sum) { return e_max - 58 > e_sum - 61 ? e_max - 58 : e_sum - 61; }

// acc + the middle digits' sum, rounded, in units of the high one
FX_HD int64_t fold(int64_t hi, int64_t mid) { return hi + ((mid + (1 << (kDigit - 1))) >> kDigit); }

#if defined(__CUDACC__)
// c + a b as one instruction (written out: as an expression the compiler
// reassociates chains of them into products and 64-bit additions)
__device__ __forceinline__ long long madw(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
#endif

}  // namespace fx
}  // namespace mg
