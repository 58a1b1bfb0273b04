// Host-side precomputation: twiddle tables and CRT constants for a set of NTT
// primes (the four 28-bit primes, or the three 31-bit ones).  Runs once per
// context and set.
#include <cmath>
#include <vector>

#include "cfft.cuh"
#include "internal.h"

namespace rosetta {
namespace {

using u128 = unsigned __int128;

uint32_t powmod(uint64_t b, uint64_t e, uint32_t p) {
  uint64_t r = 1;
  b %= p;
  while (e) {
    if (e & 1) r = r * b % p;
    b = b * b % p;
    e >>= 1;
  }
  return static_cast<uint32_t>(r);
}

bool is_prime(uint32_t p) {
  if (p < 2) return false;
  for (uint32_t d = 2; (uint64_t)d * d <= p; ++d)
    if (p % d == 0) return false;
  return true;
}

// Smallest generator of Z_p^*: g^((p-1)/f) != 1 for every prime factor f.
uint32_t generator(uint32_t p) {
  std::vector<uint32_t> fac;
  uint32_t m = p - 1;
  for (uint32_t d = 2; (uint64_t)d * d <= m; ++d) {
    if (m % d == 0) {
      fac.push_back(d);
      while (m % d == 0) m /= d;
    }
  }
  if (m > 1) fac.push_back(m);
  for (uint32_t g = 2; g < p; ++g) {
    bool ok = true;
    for (uint32_t f : fac)
      if (powmod(g, (p - 1) / f, p) == 1) {
        ok = false;
        break;
      }
    if (ok) return g;
  }
  return 0;
}

uint32_t bitrev(uint32_t x, uint32_t bits) {
  uint32_t r = 0;
  for (uint32_t i = 0; i < bits; ++i) r |= ((x >> i) & 1u) << (bits - 1 - i);
  return r;
}

uint32_t shoup(uint32_t w, uint32_t p) { return static_cast<uint32_t>((static_cast<uint64_t>(w) << 32) / p); }

}  // namespace

bool build_tables(uint32_t logN, uint32_t primes, uint2 *tw_host, CrtConsts *cc, uint32_t use) {
  const uint32_t N = 1u << logN;
  if ((primes != kPrimes && primes != kPrimes31) || use > primes) return false;
  if (use == 0) use = primes;
  const uint32_t *list = primes == kPrimes ? kPrimeList : kPrime31List;
  // 28-bit set in (2^28 - 2^18, 2^28): lazy residues up to 16p fit 32 bits and
  // the CRT quotient may use 2^28 in place of p; 31-bit set in
  // (2^31 - 2^19, 2^31): residues below 2p fit, the quotient uses 2^31
  const uint32_t top = primes == kPrimes ? 28 : 31, gap = primes == kPrimes ? 18 : 19;
  *cc = CrtConsts{};
  u128 M = 1;
  for (uint32_t q = 0; q < use; ++q) M *= list[q];
  cc->M_mod64 = static_cast<uint64_t>(M);
  cc->qf_base = cc->M_mod64 << (31 - kQfShift);
  for (uint32_t q = 0; q < use; ++q) {
    const uint32_t p = list[q];
    if (tw_host) {
      if (!is_prime(p) || (p - 1) % (2 * N) != 0 || p >= (1u << top) || p <= (1u << top) - (1u << gap)) return false;
      const uint32_t g = generator(p);
      if (!g) return false;
      const uint32_t psi = powmod(g, (p - 1) / (2 * N), p);  // primitive 2N-th root of unity
      if (powmod(psi, N, p) != p - 1) return false;
      uint64_t w = 1;  // psi^i, i = bitrev(m)
      for (uint32_t i = 0; i < N; ++i) {
        tw_host[(size_t)q * N + bitrev(i, logN)] =
            make_uint2(static_cast<uint32_t>(w), shoup(static_cast<uint32_t>(w), p));
        w = w * psi % p;
      }
    }
    PrimeConsts &pc = cc->pr[q];
    pc.p = p;
    pc.p2 = 2 * p;
    pc.p8 = 8 * p;
    uint32_t inv = 1;  // Newton iteration for p^{-1} mod 2^32
    for (int it = 0; it < 5; ++it) inv *= 2u - p * inv;
    pc.p_inv = inv;
    const u128 Mq = M / p;
    const uint32_t Mq_mod_p = static_cast<uint32_t>(Mq % p);
    const uint32_t Mq_inv = powmod(Mq_mod_p, p - 2, p);
    const uint32_t N_inv = powmod(N, p - 2, p);
    pc.crt_c = static_cast<uint32_t>(static_cast<uint64_t>(Mq_inv) * N_inv % p);
    pc.crt_cs = shoup(pc.crt_c, p);
    const uint64_t r_mont = (static_cast<uint64_t>(1) << 32) % p;
    pc.key_scale = static_cast<uint32_t>(r_mont * pc.crt_c % p);
    pc.key_scale_s = shoup(pc.key_scale, p);
    pc.Mp_mod64 = static_cast<uint64_t>(Mq);
  }
  return true;
}

void build_cfft_tables(uint32_t logN, float4 *pass_tw, double2 *tw) {
  const uint32_t logC = logN - 1, C = 1u << logC;
  // group g of stage s splits X^len - w^2; exponents of w to the primitive
  // 2N-th root exp(i pi / N): the root node X^C - i has C/2, a node with
  // exponent e has children e/2 and e/2 + C (i times the first)
  std::vector<uint32_t> e(C);
  e[1] = C / 2;
  for (uint32_t m = 1; 2 * m < C; ++m) {
    e[2 * m] = e[m] / 2;
    e[2 * m + 1] = e[m] / 2 + C;
  }
  const double step = std::acos(-1.0) / (1u << logN);
  tw[0] = make_double2(1.0, 0.0);
  for (uint32_t m = 1; m < C; ++m) tw[m] = make_double2(std::cos(step * e[m]), std::sin(step * e[m]));
  for (uint32_t pass = 0; 2 * pass < logC; ++pass)
    for (uint32_t g = 0; g < (1u << (2 * pass)); ++g) {
      const double2 w1 = tw[(1u << (2 * pass)) + g], w2 = tw[(2u << (2 * pass)) + 2 * g];
      pass_tw[cfft_tw_offset(pass) + g] = make_float4(static_cast<float>(w1.x), static_cast<float>(w1.y),
                                                      static_cast<float>(w2.x), static_cast<float>(w2.y));
    }
}

}  // namespace rosetta
