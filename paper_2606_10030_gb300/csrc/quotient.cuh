// AVG = (double)SUM / (double)COUNT with integer operations: the quotient of a
// float64 (or an int64 rounded to float64) by a count of up to 32 bits, rounded
// to nearest, ties to even, as IEEE 754 defines it. GB300 issues few float64
// operations: the last pass of the sort strategy over 1.1 M groups took 24 us
// with the float64 division, 12 us with this one.
//
// The 53-bit significand, aligned to 64 bits, is divided by the count aligned
// to 32 bits, two 32-bit quotient digits at a time, with the reciprocal-based
// 2-by-1 division of Moeller and Granlund (Improved Division by Invariant
// Integers, IEEE Trans. Comput. 2011, algorithm 4): 64 or 65 quotient bits and
// a remainder, which decide the rounding exactly. Shared with a host build used
// by the unit tests.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define AGG_HDQ __host__ __device__ __forceinline__
#else
#define AGG_HDQ inline
#endif

namespace agg {

AGG_HDQ int lead_zeros64(uint64_t x) {  // x != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

// floor((2^64 - 1) / d) - 2^32 for d >= 2^31: one Newton step from a float32
// reciprocal (relative error 2^-23 -> 2^-45, at most one off), then settled
// by its residue.
AGG_HDQ uint32_t reciprocal32(uint32_t d) {
  const float f = 1.0f / (float)d;
  uint64_t x = (uint64_t)(f * 0x1p63f) << 1;  // about 2^64 / d, 33 bits
  int64_t e = (int64_t)(0ull - x * d);        // 2^64 - x d, below 2^42 in magnitude
  x += (uint64_t)(((e >> 12) * (int64_t)x) >> 52);
  e = (int64_t)(0ull - x * d);
  for (int k = 0; k < 2; ++k) {
    if (e <= 0) {
      --x;
      e += d;
    } else if (e > (int64_t)d) {
      ++x;
      e -= d;
    }
  }
  return (uint32_t)x;  // x - 2^32
}

// (u1:u0) / d for u1 < d, v = reciprocal32(d).
AGG_HDQ uint32_t div_2by1(uint32_t u1, uint32_t u0, uint32_t d, uint32_t v, uint32_t& rem) {
  const uint64_t q = (uint64_t)v * u1 + (((uint64_t)u1 << 32) | u0);
  uint32_t q1 = (uint32_t)(q >> 32) + 1u;
  uint32_t r = u0 - q1 * d;
  if (r > (uint32_t)q) {
    --q1;
    r += d;
  }
  if (r >= d) {
    ++q1;
    r -= d;
  }
  rem = r;
  return q1;
}

// Bits of the float64 with bits b divided by c (1 <= c < 2^32), or false for
// the cases left to a float64 division: a subnormal, infinite or NaN dividend,
// and a subnormal quotient.
AGG_HDQ bool quotient_bits(uint64_t b, uint32_t c, uint64_t* out) {
  const int e = (int)((b >> 52) & 0x7FF);
  const uint64_t sign = b & 0x8000000000000000ull;
  if ((b << 1) == 0) {
    *out = b;
    return true;
  }
  const int lz = lead_zeros64(c) - 32;
  const uint32_t d = c << lz;
  const uint64_t m = ((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  uint32_t m1 = (uint32_t)(m >> 32);
  const bool top = m1 >= d;  // the quotient has 65 bits
  if (top) m1 -= d;
  const uint32_t v = reciprocal32(d);
  uint32_t r, r2;
  const uint32_t q1 = div_2by1(m1, (uint32_t)m, d, v, r);
  const uint32_t q2 = div_2by1(r, 0u, d, v, r2);
  uint64_t q = ((uint64_t)q1 << 32) | q2;
  bool sticky = r2 != 0;
  if (top) {
    sticky = sticky || (q & 1u);
    q = (q >> 1) | 0x8000000000000000ull;
  }
  const int field = e + lz - 32 + (top ? 1 : 0);
  if (e == 0 || e == 0x7FF || field < 1) return false;
  uint64_t keep = q >> 11;  // 53 bits
  const uint32_t rest = (uint32_t)q & 0x7FFu;
  if (rest > 0x400u || (rest == 0x400u && (sticky || (keep & 1u)))) ++keep;
  // the implicit bit adds one to the exponent field (a carry out of it two)
  *out = sign | ((((uint64_t)field - 1) << 52) + keep);
  return true;
}

// Bits of (double)v for an int64, rounded to nearest, ties to even.
AGG_HDQ uint64_t float64_bits_of(int64_t v) {
  if (v == 0) return 0;
  const uint64_t sign = v < 0 ? 0x8000000000000000ull : 0ull;
  const uint64_t u = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
  const int lz = lead_zeros64(u);
  const uint64_t q = u << lz;
  uint64_t keep = q >> 11;
  const uint32_t rest = (uint32_t)q & 0x7FFu;
  if (rest > 0x400u || (rest == 0x400u && (keep & 1u))) ++keep;
  return sign | (((uint64_t)(1023 + 63 - lz - 1) << 52) + keep);
}

#ifdef __CUDACC__
// AVG of a group: the sum's float64 bits over the count.
__device__ __forceinline__ double average(unsigned long long sum, uint32_t count) {
  uint64_t q;
  if (quotient_bits(sum, count, &q)) return __longlong_as_double((long long)q);
  return __longlong_as_double((long long)sum) / (double)count;
}
#endif

}  // namespace agg
