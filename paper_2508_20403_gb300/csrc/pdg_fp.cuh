// Correctly rounded FP64 operations on the integer pipes.
//
// The recovery needs three floating-point operations per edge or vertex, each
// rounded once to nearest-even as IEEE 754 defines them:
//   r = fl(1/w)            step A1, the resistive weight of a tree edge (Eq. RT)
//   R = fl(D * 2^-S)       step A3, the exact fixed-point path sum to FP64
//   s = fl(w * R)          step A3, the stretch score (one hardware multiply)
// On this GPU the double-precision pipe is a small fraction of the integer and
// single-precision pipes; the reciprocal (a multi-step sequence on that pipe)
// and the conversion (which has no single hardware instruction) are computed
// from the bit patterns with integer arithmetic.  The results are bit-identical
// to the IEEE operations (the test-suite compares them with the oracle's C
// doubles); inputs outside the normal range of the fast path fall back to the
// hardware operation.
//
//   reciprocal: one step of Newton's iteration x <- x + x (1 - m x) for 1/m on
//     the 53-bit significand m, from the single-precision reciprocal of its top
//     bits (2^-22 -> 2^-44 relative), then the exact quotient floor(2^105 / m)
//     from the remainder, and the rounding bit from what remains (no ties:
//     2^106 / m is never an odd integer for a significand that is not a power
//     of two).  Five 64-bit products; the earlier form, two steps in 128-bit
//     fixed point, took 26 us of a recovery on 2.1 M tree edges.
//   fixed point to FP64: the leading bit of the integer fixes the exponent;
//     the 53 bits below it, rounded by the remainder, the significand.
#pragma once

#include <stdint.h>
#include <string.h>

namespace pdg {

#ifdef __CUDACC__
#define PDG_HD __host__ __device__ __forceinline__
#else
#define PDG_HD inline
#endif

constexpr uint64_t kMant = (1ull << 52) - 1;

PDG_HD int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// bits of 1/f to 2^-23 relative, for the bits of a float f in [1, 2)
PDG_HD uint32_t rcp_f32_bits(uint32_t f) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(f)));
  return __float_as_uint(y);
#else
  float x;
  memcpy(&x, &f, 4);
  x = 1.0f / x;
  memcpy(&f, &x, 4);
  return f;
#endif
}

// round(2^105 / m) for a significand 2^52 < m < 2^53; *ok is false if the
// bounded correction did not settle (it always does; the caller then falls
// back to a hardware division).  Residuals are taken modulo 2^64: each is known
// to be far smaller, so the low words of the products are enough.
PDG_HD uint64_t rcp_significand(uint64_t m, bool* ok) {
  // X = 2^84 / m as a 32-bit integer, to 2^-22 relative: the bits of a single-precision reciprocal of m's top 24
  // bits, built and taken apart without conversions (they run on a slow unit)
  const uint32_t y = rcp_f32_bits(0x3f800000u | ((uint32_t)(m >> 29) & 0x7fffffu));  // of [1, 2): in (1/2, 1]
  const uint32_t x = y >= 0x3f800000u ? 0xffffffffu : (y << 8) | 0x80000000u;
  // 2^105 / m = 2^21 (X + r / m) with r = 2^84 - m X, |r| <= 2^62, and r / m ~ r X / 2^84
  const int64_t r = (int64_t)(0 - m * (uint64_t)x);
  uint64_t q = ((uint64_t)x << 21) + (uint64_t)(((r >> 31) * (int64_t)(uint64_t)x) >> 32);
  // q is within a few hundred units now: the remainder fits 64 bits, and gives the rest
  int64_t rem = (int64_t)(0 - m * q);
  const int64_t d = ((rem >> 32) * (int64_t)(uint64_t)x) >> 52;
  q += (uint64_t)d;
  rem -= d * (int64_t)m;
  bool settled = false;
  for (int k = 0; k < 4; k++) {  // q = floor(2^105 / m): 0 <= rem < m
    if (rem < 0) {
      q--;
      rem += (int64_t)m;
    } else if (rem >= (int64_t)m) {
      q++;
      rem -= (int64_t)m;
    } else {
      settled = true;
      break;
    }
  }
  *ok = settled;
  return ((uint64_t)rem > m - (uint64_t)rem) ? q + 1 : q;  // 2 rem > m: round up
}

// IEEE bits of fl(1/w) for positive normal w whose reciprocal is normal;
// *ok is false when the caller must use a hardware division instead
PDG_HD uint64_t rcp_rn_bits(uint64_t wb, bool* ok) {
  const uint64_t e = wb >> 52;  // biased exponent (sign bit 0)
  const uint64_t f = wb & kMant;
  *ok = (e >= 1 && e <= 2044);
  if (f == 0) return (2046 - e) << 52;  // 1 / 2^(e-1023) exactly
  const uint64_t q = rcp_significand(f | (1ull << 52), ok);
  return ((2045 - e) << 52) | (q & kMant);  // q in (2^52, 2^53): 1/w = q 2^(1022 - (e-1023) - 52 - 52)
}

// IEEE bits of fl(x * 2^-S) for an integer 0 < x = hi 2^64 + lo < 2^115 (the
// exact path sums stay below 2^97) whose value is a normal double: every shift
// and mask stays within 64 bits.
PDG_HD uint64_t fixed_hl_to_bits(uint64_t hi, uint64_t lo, int S) {
  int p = hi ? 127 - clz64(hi) : 63 - clz64(lo);  // leading bit
  const int sh = p - 52;                          // at most 62
  uint64_t q;
  if (sh <= 0) {
    q = lo << (-sh);  // exact (hi is zero here)
  } else {
    q = (hi << (64 - sh)) | (lo >> sh);  // below 2^53: hi < 2^(p - 63)
    const uint64_t rem = lo & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (q & 1))) {
      q++;
      if (q >> 53) {
        q >>= 1;
        p++;
      }
    }
  }
  return ((uint64_t)(p - S + 1023) << 52) | (q & kMant);
}

}  // namespace pdg
