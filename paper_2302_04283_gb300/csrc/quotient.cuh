// FP64 quotients on the integer and FP32 pipes.
//
// GB300 executes two FP64 lanes per SM and clock: an FP64 warp instruction
// occupies its SM's pipe for 16 cycles, in which the SM issues 64 others.  A
// quotient by the hardware's 20-bit approximation costs four FP64 operations
// (three to refine it, one to multiply); the digit recurrence below costs
// none.  With A and B the 53-bit significands, r an FP32 approximation of
// 1 / B (24-bit operand, one MUFU) and 21-bit digits,
//   W0 = A r,  R0 = 2^21 A - W0 B,  W1 = 2^21 R0 r,  R1 = 2^21 R0 - W1 B,
//   W2 = 2^21 R1 r,   A / B = W0 2^-21 + W1 2^-42 + W2 2^-63,
// where the remainders are exact 64-bit integers (they fit, so their low 64
// bits suffice).  r is within 2.5 2^-23 of 1 / B (truncated operand and MUFU),
// so a digit is within 2.3 of its value; W0 and W1 are taken 2 and 3 low, which
// keeps both remainders positive and below 2^56.  The quotient is good to
// 2^-61 before its one rounding: within 0.51 ulp.
#pragma once

#include <stdint.h>

namespace rad {

// A / B 2^63 (between 2^62 and 2^64) of two significands with the implicit bit
// at 52, given as words; no check of the operands.
__device__ __forceinline__ uint64_t quot_digits(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  const float bf = __uint_as_float((__funnelshift_l(bl, bh, 3) & 0x007fffffu) | 0x3f800000u);   // B 2^-52, truncated
  const float af = __uint_as_float((__funnelshift_l(al, ah, 3) & 0x007fffffu) | 0x3f800000u);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(bf));
  const uint64_t A = ((uint64_t)ah << 32) | al, B = ((uint64_t)bh << 32) | bl;
  // digits through the FP32 adder: 2^23 + x has x as its low bits
  const uint32_t w0 = __float_as_uint(__fmaf_rn(__fmul_rn(af, r), 0x1p21f, 0x1p23f - 2.0f)) - 0x4b000000u;
  const uint64_t r0 = (A << 21) - w0 * B;
  const float x0 = __uint2float_rn((uint32_t)(r0 >> 24));
  const uint32_t w1 = __float_as_uint(__fmaf_rn(x0, __fmul_rn(r, 0x1p-7f), 0x1p23f - 3.0f)) - 0x4b000000u;
  const uint64_t r1 = (r0 << 21) - w1 * B;
  const float x1 = __uint2float_rn((uint32_t)(r1 >> 24));
  const uint32_t w2 = __float_as_uint(__fmaf_rn(x1, __fmul_rn(r, 0x1p-9f), 0x1p23f)) - 0x4b000000u;   // in units of 4
  return ((uint64_t)w1 << 21) + (w2 << 2) + ((uint64_t)(w0 << 10) << 32);
}

// 1 / x; not a number for zero, subnormal, infinite or NaN x (as the refined
// hardware approximation gives; callers discard it) and where 1 / x is not normal
// (x above 2^1022).
__device__ __forceinline__ double rcp_digits(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t e = h & 0x7ff00000u;
  uint64_t q = quot_digits(0x00100000u, 0u, (h & 0x000fffffu) | 0x00100000u, l);
  const uint32_t top = (uint32_t)(q >> 63);             // significand of x is 1
  q = (q + (512u << top)) >> (10u + top);               // 53 bits, rounded
  const uint32_t hi = (uint32_t)(q >> 32) + 0x3ff00000u - e + ((1021u + top) << 20);
  // 1 / x is normal for exponents 1 .. 2044 (and for the power of two 2^1022)
  const bool ok = e - 0x00100000u < 0x7fc00000u;
  return __hiloint2double(ok ? (int)(hi | (h & 0x80000000u)) : 0x7ff80000, (int)(uint32_t)q);
}

// van Leer's half-slope dl dr / (dl + dr) where dl and dr have one sign, else
// 0: dl times the quotient dr / (dl + dr), which lies in (0, 1], formed from
// the quotient's 64 bits and dl's significand with one rounding (0.51 ulp;
// the refined reciprocal with its two products was within 1.5).  Differences
// below the normal range, and slopes that fall below it, count as zero; a
// sum that is not finite is returned as it is.
// Measured on GB300 (SM time per warp, eight warps per scheduler): 54.9 ns with
// the refined reciprocal (six FP64 operations), 15.3 with the digits; a
// reciprocal 35.6 -> 11.3 ns with its argument's addition.
__device__ __forceinline__ double van_leer_digits(double dl, double dr) {
  const double s = dl + dr;
  const uint32_t lh = (uint32_t)__double2hiint(dl), rh = (uint32_t)__double2hiint(dr), sh = (uint32_t)__double2hiint(s);
  const uint32_t el = lh & 0x7ff00000u, er = rh & 0x7ff00000u, es = sh & 0x7ff00000u;
  const uint64_t q = quot_digits((rh & 0x000fffffu) | 0x00100000u, (uint32_t)__double2loint(dr),
                                 (sh & 0x000fffffu) | 0x00100000u, (uint32_t)__double2loint(s));
  // times dl's significand (at bit 63): the top 64 bits of the product but for
  // the low halves' product, between 2^61 and 2^64
  const uint32_t ll = (uint32_t)__double2loint(dl), mh = (lh << 11) | (ll >> 21) | 0x80000000u, ml = ll << 11;
  const uint32_t qh = (uint32_t)(q >> 32), ql = (uint32_t)q;
  uint64_t t = (uint64_t)qh * mh + (((uint64_t)qh * ml) >> 32) + (((uint64_t)ql * mh) >> 32);
  const uint32_t z = (uint32_t)__clz((int)(t >> 32));    // 0 .. 2
  t = (t + (1024u >> z)) >> (11u - z);                  // 53 bits, rounded
  const int ex = (int)(el + er) - (int)es - (int)(z << 20);
  const uint32_t hi = (uint32_t)(t >> 32) + (uint32_t)ex;
  // exponent of the result: el + er - es + 1 - z biased, less the implicit bit
  const bool ok = (int)(lh ^ rh) >= 0 && er != 0u && el != 0u && ex > 0;
  const double v = __hiloint2double(ok ? (int)(hi | (lh & 0x80000000u)) : 0, ok ? (int)(uint32_t)t : 0);
  return es == 0x7ff00000u ? s : v;
}

}  // namespace rad
