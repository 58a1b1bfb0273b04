// Word-level modular arithmetic for the NTT primes: the 28-bit set (16p <
// 2^32, so lazily reduced residues up to 8p still fit a 32-bit register) and
// the 31-bit set (2p < 2^32: residues below 2p).
//
// Residues are kept "lazy": a value congruent to the residue but possibly a
// few multiples of p above it.  Every function states the range it accepts
// and the range it returns.
#pragma once
#include <stdint.h>

#include "internal.h"

namespace rosetta {

// Shoup multiplication by a constant w < p with companion ws = floor(w 2^32 / p):
// for any 32-bit y returns y*w mod p as a value in [0, 2p).
__device__ __forceinline__ uint32_t shoup_mul(uint32_t y, uint32_t w, uint32_t ws, uint32_t p) {
  const uint32_t q = __umulhi(y, ws);
  return y * w - q * p;
}

// Montgomery reduction with R = 2^32, p_inv = p^{-1} mod 2^32.
// For T < p * 2^32 returns a value in (0, 2p) congruent to T * 2^-32 mod p.
// The low words of T and m*p agree, so (T - m p) / 2^32 = hi(T) - hi(m p).
__device__ __forceinline__ uint32_t redc(uint64_t T, uint32_t p, uint32_t p_inv) {
  const uint32_t m = static_cast<uint32_t>(T) * p_inv;
  const uint32_t t = __umulhi(m, p);
  return static_cast<uint32_t>(T >> 32) - t + p;
}

// Quotient of the explicit CRT, round(sum_q y_q / p_q), from ysum = sum_q
// (y_q >> 2) with every y_q < 8 p_q.  The primes lie in (2^28 - 2^18, 2^28),
// so y / 2^28 undershoots y / p by less than 8 (2^28 - p) / 2^28 < 2^-7 per
// prime (the shift adds under 2^-26); the four together by less than 2^-5.
// The exact sum is an integer plus X / M with |X| <= 2^110 < M / 3.99 (the
// bound every accepted parameter set meets), so the estimate stays within
// 0.29 of that integer and rounds to it.
__device__ __forceinline__ uint32_t crt_quotient(uint32_t ysum) { return (ysum + (1u << 25)) >> 26; }

// The same for the three primes in (2^31 - 2^19, 2^31), from ysum = sum_q
// (y_q >> 3) with every y_q < 2 p_q < 2^32 (the sum stays below 2^31).
// y / 2^31 undershoots y / p by less than 2 (2^31 - p) / 2^31 < 2^-11 per
// prime (the shift adds under 2^-28); the three together by less than 2^-9.
// Only parameter sets whose exact integer value X obeys |X| <= 0.45 M take
// this prime set, so the estimate stays within 0.46 of the integer.
__device__ __forceinline__ uint32_t crt_quotient31(uint32_t ysum) { return (ysum + (1u << 27)) >> 28; }

// Worst case of the float transforms' estimate, in units of 2^-24 of the bound on |X|
// (derived in cfft.cuh).
constexpr double kCfftErr = 100.0;
static_assert(kCfftErr / 16777216.0 * (1ull << (kQfBits / 2)) * (1ull << (kQfBits - kQfBits / 2)) <
                  0.1 * kPrimeList[0] * kPrimeList[1] * kPrimeList[2],
              "the estimate of X / M3 is within 0.1 of its exact value");

// The quotient of three 28-bit primes where X may be many times their product
// M3: round(sum_q y_q / p_q - X / M3), from ysum = sum_q (y_q >> 17) and est =
// 2^kQfShift X / M3 as the float transforms give it, plus an offset of
// 2^(31 - kQfShift) that keeps it positive.  The primes lie in (2^28 - 2^18,
// 2^28): y / 2^28 undershoots y / p by less than 2^-7 per prime (the shift adds
// 2^-11), the three together by less than 2^-5.  est is within
// kCfftErr 2^-24 2^98 / 2^83.99 < 0.1 of its exact value (|X| <=
// 2^98), so the sum stays within 0.14 of an integer and rounds to it; |est|
// <= 2^30.02 fits the conversion.
__device__ __forceinline__ uint32_t qf_quotient(uint32_t ysum, float est) {
  static_assert(kQfShift > 11, "ysum counts units of 2^-11");
  return ((ysum << (kQfShift - 11)) + (1u << 31) + (1u << (kQfShift - 1)) -
          static_cast<uint32_t>(__float2int_rn(est))) >> kQfShift;
}

// y0 >> 17 in the low and y1 >> 17 in the high half (y < 2^31: three such words
// add without a carry between the halves).
__device__ __forceinline__ uint32_t qf_pack(uint32_t y0, uint32_t y1) {
  return (__byte_perm(y0, y1, 0x7632) >> 1) & 0x7FFF7FFFu;
}

// x in [0, 2b) -> [0, b) for a bound b: one subtraction when x >= b.
__device__ __forceinline__ uint32_t cond_sub(uint32_t x, uint32_t b) {
  return min(x, x - b);
}

// Balanced base-2^beta digits of a word rounded to its top beta * level bits,
// in closed form: the digits are the plain ones of the word plus dig_offset,
// each less 2^(beta-1).  (Rounding adds half the lowest kept unit; adding half a
// unit at every digit makes each carry happen where the digit-by-digit rule
// carries; the last carry falls off the word in both.)
__device__ __forceinline__ uint64_t dig_offset(uint32_t beta, uint32_t level) {
  const uint32_t bits = beta * level;
  uint64_t c = bits >= 64 ? 0 : 1ull << (63 - bits);
  for (uint32_t m = 1; m <= level; ++m) c += 1ull << (64 - m * beta + beta - 1);
  return c;
}

// The digit of level lev (0: most significant) plus 2^(beta-1), in [0, 2^beta),
// from w = word + dig_offset.
__device__ __forceinline__ uint32_t biased_digit(uint64_t w, uint32_t beta, uint32_t lev) {
  return static_cast<uint32_t>(w >> (64 - (lev + 1) * beta)) & ((1u << beta) - 1u);
}

}  // namespace rosetta
