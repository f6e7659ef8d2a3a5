// mul64.h -- the correctly rounded binary64 product on the integer units.
//
// GB300 issues a warp's binary64 instruction every 76 cycles per SM
// sub-partition (64 for a fused multiply-add), its integer units one per cycle
// or two.  The parity form's sums acc = rn(acc + rn(a b)) are two binary64
// instructions per term, so forming the product from 32-bit integer multiplies
// (about 25 instructions) while the binary64 pipe does the additions halves
// what a term costs.
//
// Method: with the 53-bit significands shifted to 64 bits (A, B >= 2^63), the
// 128-bit product A B is formed from its four 32-bit partial products and
// normalised (its top bit is bit 127 or 126); the top 53 bits are kept and
// rounded to nearest even by the 11 bits below them and whether anything below
// those is set.  Operands whose product could leave the normal range are the
// caller's (mul64_safe).  There is no branch and no binary64 instruction: one
// that is predicated off for every lane still takes its turn in the pipe.
// Free of CUDA so that the host tests compile it.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define LAGP_M64 __device__ __host__ __forceinline__
#else
#define LAGP_M64 inline
#endif

namespace lagp {

// both words of a significand shifted to 64 bits, and the exponent (with the
// sign for `a`) in the place it has in the high word of a binary64
struct Mul64 {
  uint32_t lo, hi, e;
};

// operands within [2^-500, 2^500] in magnitude: neither they nor their product
// are zero, subnormal, infinite or NaN
LAGP_M64 bool mul64_safe(uint32_t hi_word) {
  return ((hi_word & 0x7fffffffu) - 0x20b00000u) < 0x3e800000u;
}

// the factor whose exponent word carries its sign, and the bias once
LAGP_M64 Mul64 mul64_a(uint32_t lo, uint32_t hi) {
  Mul64 m;
  m.lo = lo << 11;
  m.hi = (hi << 11 | lo >> 21) | 0x80000000u;
  m.e = (hi & 0xfff00000u) - (1024u << 20);
  return m;
}
// the positive factor (a correlation)
LAGP_M64 Mul64 mul64_b(uint32_t lo, uint32_t hi) {
  Mul64 m;
  m.lo = lo << 11;
  m.hi = (hi << 11 | lo >> 21) | 0x80000000u;
  m.e = hi & 0x7ff00000u;
  return m;
}

// the bits of rn(a b)
LAGP_M64 uint64_t mul64(const Mul64& a, const Mul64& b) {
  const uint64_t p = (uint64_t)a.lo * b.lo;
  const uint64_t t = (uint64_t)a.hi * b.lo + (p >> 32);
  const uint64_t u = (uint64_t)a.lo * b.hi + (uint32_t)t;
  uint64_t h = (uint64_t)a.hi * b.hi + (t >> 32) + (u >> 32);   // bits 64.. of A B
  uint32_t w = (uint32_t)u;                                      // bits 32..63
  const uint32_t top = (uint32_t)(h >> 63);
  if (!top) {
    h = (h << 1) | (w >> 31);
    w <<= 1;
  }
  const uint32_t low = (uint32_t)h;
  const uint32_t below = (w | (uint32_t)p) ? 1u : 0u;
  const uint32_t up = (((low & 0x7ffu) | below) + 0x3ffu + ((low >> 11) & 1u)) >> 11;
  return (h >> 11) + up + ((uint64_t)(a.e + b.e + (top << 20)) << 32);
}

}  // namespace lagp
