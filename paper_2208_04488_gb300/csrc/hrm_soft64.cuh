// FP64 products, quotients and square roots on the integer pipes.
//
// What bounds the FP64 kernels is the SM's one FP64 unit: measured on the GB300,
// it takes an add or a product of a warp every 19 cycles, whatever the number of
// active lanes, and one warp alone issues one only every 64 cycles, dependent or
// not. The integer pipes of the four schedulers are idle meanwhile. The functions
// below form the correctly rounded IEEE-754 result (to nearest, ties to even)
// from the encodings with integer arithmetic, so that a kernel can run part of
// its FP64 work beside the FP64 unit; every result has the bits of the FP64
// instruction, which the tests check. Measured with 16 warps per SM, in cycles of
// the SM per warp operation, against the FP64 unit's own: product 12.9 (16.7 with
// the checks of its operands) against 19, quotient 21 (27) against 137, square
// root 30 against 143.
//
// The quotient is a long division of the significands (digits of 23, 19 and 12
// bits from a reciprocal that is never too large, remainders exact), so its
// rounding needs no analysis of the approximation. This file also compiles as
// host C++, where the tests compare the functions with the machine's FP64
// arithmetic for every error that the reciprocal is allowed to have.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define HRM_SOFT __device__ __forceinline__
#else
#include <cstring>
#define HRM_SOFT static inline
#endif

namespace hrm {
namespace soft {

#ifdef __CUDACC__
HRM_SOFT uint32_t hi_of(double x) { return (uint32_t)__double2hiint(x); }
HRM_SOFT uint32_t lo_of(double x) { return (uint32_t)__double2loint(x); }
HRM_SOFT double pack(uint32_t hi, uint32_t lo) { return __hiloint2double((int)hi, (int)lo); }
HRM_SOFT uint32_t mul_hi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
HRM_SOFT uint32_t fsl(uint32_t lo, uint32_t hi, int s) { return __funnelshift_l(lo, hi, s); }
// bits of an approximate reciprocal, absolute error at most 2^-23 for 1 <= x <= 2
HRM_SOFT uint32_t rcp_bits(uint32_t x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(x)));
  return __float_as_uint(r);
}
HRM_SOFT uint32_t rsqrt_bits(uint32_t x) {  // 1 / sqrt(x), 1 <= x <= 4, relative error at most 2^-22.9
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(x)));
  return __float_as_uint(r);
}
#else
extern int rcp_error;  // units of 2^-24 that the test adds to the correctly rounded reciprocal
HRM_SOFT uint32_t hi_of(double x) { uint64_t u; std::memcpy(&u, &x, 8); return (uint32_t)(u >> 32); }
HRM_SOFT uint32_t lo_of(double x) { uint64_t u; std::memcpy(&u, &x, 8); return (uint32_t)u; }
HRM_SOFT double pack(uint32_t hi, uint32_t lo) { uint64_t u = (uint64_t)hi << 32 | lo; double x; std::memcpy(&x, &u, 8); return x; }
HRM_SOFT uint32_t mul_hi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
HRM_SOFT uint32_t fsl(uint32_t lo, uint32_t hi, int s) { return s ? hi << s | lo >> (32 - s) : hi; }
HRM_SOFT uint32_t rcp_bits(uint32_t x) {
  float f;
  std::memcpy(&f, &x, 4);
  f = 1.0f / f;
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return u + (uint32_t)rcp_error;
}
HRM_SOFT uint32_t rsqrt_bits(uint32_t x) {
  float f;
  std::memcpy(&f, &x, 4);
  f = (float)(1.0 / std::sqrt((double)f));
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return u + (uint32_t)rcp_error;
}
#endif

constexpr uint32_t kExp = 0x7ff00000u, kSign = 0x80000000u, kOne = 0x00100000u;  // exponent field, sign, unit of the exponent

// Product of two numbers that are each zero (ZERO) or normal, where a product
// that is not zero has a normal result. SIGN: they may be negative.
// The significands, one of them moved up by 11 bits, give a product whose upper
// 64 bits hold the 53-bit significand (or, below 2, one bit less) and whose
// lower 64 bits decide the rounding.
template <bool ZERO = true, bool SIGN = true>
HRM_SOFT double mul_in(double a, double b) {
  const uint32_t ah = hi_of(a), al = lo_of(a), bh = hi_of(b), bl = lo_of(b);
  const uint32_t ma = (ah & 0xfffffu) | kOne, mb = (bh & 0xfffffu) | kOne;
  const uint32_t b1 = fsl(bl, mb, 11), b0 = bl << 11;
  const uint64_t p = (uint64_t)al * b0;
  const uint64_t t = (uint64_t)ma * b0 + (p >> 32);
  const uint64_t u = (uint64_t)al * b1 + (uint32_t)t;
  const uint64_t h = (uint64_t)ma * b1 + (t >> 32) + (u >> 32);
  uint32_t h1 = (uint32_t)(h >> 32), h0 = (uint32_t)h, low = (uint32_t)u | ((uint32_t)p ? 1u : 0u);  // last bit: sticky
  const uint32_t two = (h1 >> 20) & 1u;  // the significands' product is at least 2
  if (!two) {
    h1 = fsl(h0, h1, 1);
    h0 = fsl(low, h0, 1);
    low <<= 1;
  }
  // exponents and signs add up in the upper word (h1 holds the leading bit)
  const uint32_t mask = SIGN ? 0xfff00000u : kExp;
  const uint32_t ex = (ah & mask) + (bh & mask) - (1024u << 20) + (two << 20);
  const uint64_t r = (uint64_t)low + 0x7fffffffu + (h0 & 1u);  // a carry out of 32 bits: round up
  const uint64_t m = ((uint64_t)(h1 + ex) << 32 | h0) + (r >> 32);
  uint32_t rh = (uint32_t)(m >> 32), rl = (uint32_t)m;
  if (ZERO) {
    const bool z = ((ah & kExp) == 0u) | ((bh & kExp) == 0u);
    rh = z ? (SIGN ? (ah ^ bh) & kSign : 0u) : rh;
    rl = z ? 0u : rl;
  }
  return pack(rh, rl);
}

// Quotient of two normal numbers with a normal result.
// ri is 2^76 / B for the 53-bit significand B, never too large and too small by
// at most 3 units of 2^-22 relative: with the remainder R of a digit step in
// units of B, the next digit is too small by at most R 3 2^-22 2^bits + 1, so
// the three remainders stay below 13.1 B, 6 B and 1.02 B (64 bits hold them)
// and one comparison completes the 54-bit quotient. A quotient of two 53-bit
// numbers never lies halfway between two others, so the bit below the last
// decides the rounding.
// EXP: the result times 2^EXP (exponents are added up in the upper word anyway).
template <int EXP = 0>
HRM_SOFT double div_in(double a, double b) {
  const uint32_t ah = hi_of(a), al = lo_of(a), bh = hi_of(b), bl = lo_of(b);
  const uint64_t A = (uint64_t)((ah & 0xfffffu) | kOne) << 32 | al;
  const uint64_t B = (uint64_t)((bh & 0xfffffu) | kOne) << 32 | bl;
  const uint32_t ri = rcp_bits(0x3f800001u + (fsl(bl, bh, 3) & 0x7fffffu)) - 0x3e800003u;
  const uint64_t nB = 0ull - B;
  const uint32_t n1 = (uint32_t)(nB >> 32), n0 = (uint32_t)nB;
  auto step = [&](uint64_t R, int bits, uint32_t d) -> uint64_t {  // R 2^bits - d B
    const uint64_t x = (uint64_t)d * n0 + (R << bits);
    return x + ((uint64_t)(d * n1) << 32);
  };
  const uint32_t d0 = mul_hi((uint32_t)(A >> 21), ri);
  uint64_t R = step(A, 23, d0);
  const uint32_t d1 = mul_hi((uint32_t)(R >> 25), ri);
  R = step(R, 19, d1);
  const uint32_t d2 = mul_hi((uint32_t)(R >> 25), ri) >> 7;
  R = step(R, 12, d2);
  uint64_t q = ((uint64_t)d0 << 31) + ((uint64_t)d1 << 12) + d2 + (R >= B ? 1u : 0u);
  const uint32_t one = (uint32_t)(q >> 54);  // A >= B
  q = (q + 1u + one) >> (1u + one);
  const uint32_t ex = (ah & 0xfff00000u) - (bh & 0xfff00000u) + ((uint32_t)(1021 + EXP) << 20) + (one << 20);
  return pack((uint32_t)(q >> 32) + ex, (uint32_t)q);
}

// Square root of a positive normal number. X, 54 bits, is the significand with
// an even exponent (m = X / 2^52 in [1, 4)) and the root the integer S with
// S^2 <= X 2^52 < (S + 1)^2. ri is 2^24 / sqrt(m), never too large and too small
// by at most 3.5 units of 2^-22 relative. The first digit (22 bits below the
// point) is m times it, the next two are half the exact remainder times it: too
// small by at most 8.01, 17.1 and 1.04 units (never too large: the remainder
// over 2 s is below the remainder over the sum of the roots), so that the
// remainders stay below 2^35.1, 2^48.1 and 2^54.1. One comparison completes S,
// and the final remainder compared with S decides the rounding: (S + 1/2)^2 is
// S^2 + S + 1/4.
HRM_SOFT double sqrt_in(double a) {
  const uint32_t ah = hi_of(a), al = lo_of(a);
  const uint32_t odd = ((ah >> 20) & 1u) ^ 1u;  // biased exponent even: true exponent odd, m in [2, 4)
  const uint64_t X = ((uint64_t)((ah & 0xfffffu) | kOne) << 32 | al) << odd;
  const uint32_t ri = rsqrt_bits(0x3f800001u + (fsl(al, ah, 3) & 0x7fffffu) + (odd << 23)) - 0x3e800004u;
  const uint32_t d0 = mul_hi((uint32_t)(X >> 22), ri);
  const uint64_t R0 = X - ((uint64_t)d0 * d0 << 8);                                               // units of 2^-52
  uint64_t S = ((uint64_t)d0 << 20) + (uint32_t)((uint64_t)(uint32_t)(R0 >> 4) * ri >> 31);       // of 2^-42
  const uint64_t R1 = (X << 32) - S * S;                                                          // of 2^-84
  S = (S << 10) + (mul_hi((uint32_t)(R1 >> 17), ri) >> 8);                                        // of 2^-52
  uint64_t R = (X << 52) - S * S;
  if (R > 2u * S) {
    R -= 2u * S + 1u;
    S += 1u;
  }
  S += R > S ? 1u : 0u;
  const uint32_t ex = ((ah >> 20) + 1023u) >> 1;
  return pack((uint32_t)(S >> 32) + ((ex - 1u) << 20), (uint32_t)S);
}

// a / b for any operands: the long division where both are normal and the
// quotient's exponent lies well inside the normal range; a zero a is a zero
// quotient; anything else is left to the FP64 instruction sequence.
HRM_SOFT double div(double a, double b) {
  const uint32_t ea = hi_of(a) & kExp, eb = hi_of(b) & kExp;
  const bool bn = eb - kOne < kExp - kOne;  // exponent field 1..2046
  if ((ea - kOne < kExp - kOne) & bn & (ea - eb + (1000u << 20) <= (2000u << 20))) return div_in(a, b);
  if (bn & (((hi_of(a) & ~kSign) | lo_of(a)) == 0u)) return pack((hi_of(a) ^ hi_of(b)) & kSign, 0u);
  return a / b;
}

// a b for any operands, likewise.
HRM_SOFT double mul(double a, double b) {
  const uint32_t ea = hi_of(a) & kExp, eb = hi_of(b) & kExp;
  // ea + eb - 1023 within 1..2044 (the sum of two fields fits 32 bits)
  if ((ea - kOne < kExp - kOne) & (eb - kOne < kExp - kOne) & (ea + eb - (1024u << 20) <= (2043u << 20)))
    return mul_in<false, true>(a, b);
  if ((ea < kExp) & (eb < kExp) &
      ((((hi_of(a) & ~kSign) | lo_of(a)) == 0u) | (((hi_of(b) & ~kSign) | lo_of(b)) == 0u)))
    return pack((hi_of(a) ^ hi_of(b)) & kSign, 0u);
  return a * b;
}

// a 2^EXP, EXP small: the exponent field of a normal number moves.
template <int EXP>
HRM_SOFT double scale(double a) {
  const uint32_t h = hi_of(a), e = h & kExp;
  if (e - (16u << 20) < (2000u << 20)) return pack(h + ((uint32_t)EXP << 20), lo_of(a));
  if (((h & ~kSign) | lo_of(a)) == 0u) return a;
  return a * (EXP < 0 ? 1.0 / (double)(1 << (EXP < 0 ? -EXP : 0)) : (double)(1 << (EXP > 0 ? EXP : 0)));
}

// Whether x is zero or of a magnitude within [2^LO, 2^HI).
template <int LO, int HI>
HRM_SOFT bool within(double x) {
  const uint32_t h = hi_of(x);
  return ((h & kExp) - ((uint32_t)(1023 + LO) << 20) < ((uint32_t)(HI - LO) << 20)) | (((h & ~kSign) | lo_of(x)) == 0u);
}

// sqrt(a) for any operand, likewise.
HRM_SOFT double root(double a) {
  if (hi_of(a) - kOne < kExp - kOne) return sqrt_in(a);  // positive and normal
  return ::sqrt(a);
}

}  // namespace soft
}  // namespace hrm
