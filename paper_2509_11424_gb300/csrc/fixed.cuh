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
// order) and rounded to a double once.  What is lost of a sum of K products is
// the dropped term and the operands' rounding, at most K (2 x 2^-58 + 2^-60) of
// the product of the two groups' largest entries.  Where these meet, that is less
// than what FP64 additions round off (2^-53 of every partial sum).  Where they
// meet only small entries, or none, it is not: an entry 2^-k of its group's
// largest keeps 57 - k bits and below 2^-58 nothing.  So every kernel compares
// its sums (or the entries' exponents) with the scale, and forms those that are
// small against it in FP64.
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

// not +-0, on the integer pipe
FX_HD bool nonzero(double v) { return ((uint64_t)bits_of(v) << 1) != 0; }

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

// the same to nearest, BITS <= 61; |result| <= 2^BITS
template <int BITS = kVecBits> FX_HD int64_t to_nearest(double v, int E) {
  const int64_t b = bits_of(v);
  int e = (int)((b >> 52) & 0x7ff);
  const uint64_t m = ((uint64_t)b & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  if (e == 0) e = 1;
  int s = E - e + 63 - BITS;  // >= 2
  if (s > 64) s = 64;
  const int64_t x = (int64_t)((((m << 10) >> (s - 1)) + 1) >> 1);
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

// 2^e as a double, also outside the normal range
__device__ __forceinline__ double scaled(double v, int e) {
  return e > -1000 && e < 1000 ? v * __longlong_as_double((long long)(e + 1023) << 52) : scalbn(v, e);
}

// the sum over a warp of values some of which are Inf or NaN
__device__ __forceinline__ double warp_bad(double p) {
  const double inf = __longlong_as_double(0x7ff0000000000000ll);
  const bool pos = __any_sync(0xffffffffu, p == inf), neg = __any_sync(0xffffffffu, p == -inf);
  const bool nan = __any_sync(0xffffffffu, p != p) || (pos && neg);
  return nan ? __longlong_as_double(0x7ff8000000000000ll) : pos ? inf : -inf;
}

// ---- exact sums over a warp.  Every lane calls add() for value 0, 1, ... in
// turn; get() then gives lane v the sum of value v.
//
// FP32 lanes: integers of 51 bits in the unit of the largest lane's exponent,
// as two words whose 32-fold sums fit 32 bits.  Where bad() says so (in every
// lane), Inf or NaN were among the values: fix() for each of them, with the
// same arguments, before get().
struct WarpSumF {
  unsigned lo = 0;
  int hi = 0, e = 0;
  __device__ __forceinline__ void add(int v, float p) {
    const unsigned b = __float_as_uint(p);
    int x = (b >> 23) & 0xff;
    const int E = __reduce_max_sync(0xffffffffu, x);
    const unsigned m = (b & 0x7fffffu) | (x ? 0x800000u : 0u);
    x = x ? x : 1;
    const int s = min(max(E, 1) - x, 60);
    long long X = (long long)(((unsigned long long)m << 27) >> s);
    X = (int)b < 0 ? -X : X;
    const unsigned l = __reduce_add_sync(0xffffffffu, (unsigned)X & 0x3ffffffu);
    const int h = __reduce_add_sync(0xffffffffu, (int)(X >> 26));
    if ((int)(threadIdx.x & 31) == v) {
      lo = l;
      hi = h;
      e = E;
    }
  }
  __device__ __forceinline__ bool bad() const { return __any_sync(0xffffffffu, e == 0xff); }
  __device__ __forceinline__ void fix(int v, float p) {
    if (__shfl_sync(0xffffffffu, e, v) != 0xff) return;
    const float b = (float)warp_bad((p - p == 0.f) ? 0.0 : (double)p);
    if ((int)(threadIdx.x & 31) == v) lo = __float_as_uint(b);
  }
  __device__ __forceinline__ double get() const {
    const double d = scaled((double)(((long long)hi << 26) + lo), max(e, 1) - (127 + 23 + 27));
    return e == 0xff ? (double)__uint_as_float(lo) : d;
  }
};
// 64-bit integers in units of 2^unit (the same in every lane): three words.
constexpr int kSmallBits = 2 * kVecBits - 2 * kDigit - 5;
struct WarpSumI {
  unsigned w0 = 0, w1 = 0;
  int w2 = 0, e = 0;
  __device__ __forceinline__ void add(int v, long long X, int unit) {
    const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)X & 0x3ffffffu);
    const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(X >> 26) & 0x3ffffffu);
    const int c = __reduce_add_sync(0xffffffffu, (int)(X >> 52));
    if ((int)(threadIdx.x & 31) == v) {
      w0 = a;
      w1 = b;
      w2 = c;
      e = unit;
    }
  }
  // whether the lane's sum is between -2^kSmallBits and 2^kSmallBits
  __device__ __forceinline__ bool small() const {
    constexpr int t = 1 << (kSmallBits - 52);
    return (unsigned)(w2 + (int)(w1 >> 26) + t) < 2u * t;
  }
  __device__ __forceinline__ double get() const {
    return scaled(fma((double)w2, 0x1p52, (double)(((long long)w1 << 26) + w0)), e);
  }
};
// bit 2 j: pred holds in lanes 2 j and 2 j + 1
__device__ __forceinline__ unsigned ballot_pairs(bool pred) {
  const unsigned m = __ballot_sync(0xffffffffu, pred);
  return m & (m >> 1) & 0x55555555u;
}

__device__ __forceinline__ int warp_exp(int e) { return max(__reduce_max_sync(0xffffffffu, e), 1); }
// the sum over a warp's lanes of FP64 values, value v to lane v
struct WarpSumD : WarpSumI {
  double bad = 0.0;
  __device__ __forceinline__ void add(int v, double p) {
    const int E = max(__reduce_max_sync(0xffffffffu, exp_field(p)), 1);
    WarpSumI::add(v, to_fixed(p, min(E, kBadExp - 1)), E == kBadExp ? 1 << 20 : E - 1022 - kVecBits);
    if (E == kBadExp) {
      const double b = warp_bad(p);
      if ((int)(threadIdx.x & 31) == v) bad = b;
    }
  }
  __device__ __forceinline__ double get() const { return e == 1 << 20 ? bad : WarpSumI::get(); }
};
// the sum of n FP64 values by one warp, in lane 0: the 256 values of a step are
// added as integers in the unit of their largest (one by one in FP64, the 256
// partial sums of a reduction cost more than the reduction)
__device__ __forceinline__ double warp_total(const double *__restrict__ p, int n) {
  constexpr int U = 8;
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  for (int b = 0; b < n; b += 32 * U) {
    double x[U];
    int E = 1;
#pragma unroll
    for (int u = 0; u < U; ++u) x[u] = b + 32 * u + lane < n ? __ldcg(p + b + 32 * u + lane) : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) E = max(E, exp_field(x[u]));
    E = __reduce_max_sync(0xffffffffu, E);
    long long X = 0;  // 8 values below 2^kVecBits
#pragma unroll
    for (int u = 0; u < U; ++u) X += to_fixed(x[u], min(E, kBadExp - 1));
    WarpSumI ws;
    ws.add(0, X, E - 1022 - kVecBits);
    double d = ws.get();
    if (E == kBadExp) {
      double bad = 0.0;
#pragma unroll
      for (int u = 0; u < U; ++u) bad += exp_field(x[u]) == kBadExp ? x[u] : 0.0;
      d = warp_bad(bad);
    }
    t += d;
  }
  return t;
}
__device__ __forceinline__ int4 digits(double2 v, int E) {
  const long long a = to_nearest(v.x, E), b = to_nearest(v.y, E);
  return make_int4(digit_hi(a), digit_lo(a), digit_hi(b), digit_lo(b));
}
#endif

}  // namespace fx
}  // namespace mg
