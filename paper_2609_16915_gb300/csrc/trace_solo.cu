// RLWE trace for N = 2048 at full batches: one worker of 256 threads per
// ciphertext, three workers per SM, no cluster, the products by three 28-bit
// primes and a float quotient.
//
// Same steps and words as trace.cu; work split and arithmetic as in
// blind_rotate_solo.cu: worker thread tau owns coefficients tau + 256 e of both
// components, so digits stay in registers and residues end in the thread that
// needs them; only the automorphism's gather and the transforms' exchanges cross
// threads.  Per step and prime `level` forward and two inverse transforms, then the
// float estimate of X / M3 (X below level N 2^(base_log-1) 2^63 <= 2^98; cfft.cuh's
// rounding with `level` <= 4 products a sum: under 100 u).
//
// Bounded like blind_rotate_solo.cu by the shared-memory and integer-multiply pipes;
// the 64-bit words whose digits all three primes and the floats need cost 44
// bytes of spills at 80 registers.  Measured, gadget 2^16 x 4, 456 ciphertexts (a wave of
// three workers per SM): 480 us, the cluster kernel 603; with the level at run time
// and the float pairs in a loop 500 (152 bytes of spills).  912: 948 (1144); 1024 (912 here,
// the rest on clusters): 1142 (1264); 2000: 2143 (2480).
#include <stdint.h>

#include "cfft.cuh"
#include "internal.h"
#include "ntt.cuh"

namespace rosetta {

namespace {

constexpr int kTrLogN = 11;
constexpr uint32_t kTrN = 1u << kTrLogN, kTrT = kTrN / 8;  // threads of a worker
constexpr uint32_t kTrWorkers = 3;                         // per CTA (and SM)
constexpr uint32_t kTrTwF = 352;                           // float4 entries of the pass table (341, padded)
constexpr uint32_t kTrXbWords = 2 * NttShape<kTrLogN, 8>::XB_WORDS;
static_assert(kTrXbWords >= 4 * (kTrN / 2), "exchange buffer");

constexpr size_t tr_smem_bytes(uint32_t workers) {
  return kPrimesQf * kTrN * sizeof(uint2) + kTrTwF * sizeof(float4) +
         workers * (2 * kTrN * sizeof(uint64_t) + kTrXbWords * sizeof(uint32_t));
}

}  // namespace

// Shared memory: twiddles of the three primes uint2 [3][N], the float pass table
// float4 [352], then per worker acc uint64 [N][2] and the exchange buffer.
template <uint32_t PAIRS>
__global__ void __launch_bounds__(kTrWorkers *kTrT, 1) trace_solo_kernel(const __grid_constant__ TraceArgs a) {
  constexpr uint32_t N = kTrN, T = kTrT, TWO_N = 2 * N;
  constexpr int E = 8;
  extern __shared__ __align__(16) unsigned char smem[];
  uint2 *tw_all = reinterpret_cast<uint2 *>(smem);
  float4 *twf = reinterpret_cast<float4 *>(tw_all + kPrimesQf * N);
  const uint32_t worker = __shfl_sync(0xffffffffu, threadIdx.x / T, 0);  // (warp-uniform for the compiler)
  const uint32_t tau = threadIdx.x % T;
  ulonglong2 *acc = reinterpret_cast<ulonglong2 *>(twf + kTrTwF) + worker * (N + kTrXbWords / 4);
  uint32_t *xb = reinterpret_cast<uint32_t *>(acc + N);

  for (uint32_t m = threadIdx.x; m < kPrimesQf * N; m += blockDim.x)
    tw_all[m / N * N + split_tw_slot<kTrLogN>(m % N)] = a.tw[m];
  const float4 *twf_src = reinterpret_cast<const float4 *>(a.tw + kPrimesQf * N);
  for (uint32_t m = threadIdx.x; m < kTrTwF; m += blockDim.x) twf[m] = twf_src[m];
  __syncthreads();

  const uint32_t ct = blockIdx.x * (blockDim.x / T) + worker;
  if (ct >= a.batch) return;  // the whole worker; from here on it meets only its own barrier
  const GroupThreads th{worker + 1u, T};

  const uint64_t *gin = a.glwe_in + static_cast<size_t>(ct) * 2 * N;
  for (uint32_t j = tau; j < N; j += T) acc[j] = make_ulonglong2(gin[j], gin[N + j]);
  th.sync();

  const uint64_t dig_add = dig_offset(a.base_log, 2 * PAIRS);
  const uint32_t half = 1u << (a.base_log - 1);  // stored digits lie in [0, B): d = stored - B/2
  constexpr uint32_t kblk = PAIRS * 4 * N;  // words of one step's key block per prime

#pragma unroll 1
  for (uint32_t s = 0; s < kTrLogN; ++s) {
    const uint32_t k = (1u << (kTrLogN - s)) + 1u;
    uint32_t kinv = k;  // k^{-1} mod 2^32 (Newton), hence mod 2N
#pragma unroll
    for (int it = 0; it < 5; ++it) kinv *= 2u - k * kinv;
    const uint32_t *key = a.keys + static_cast<size_t>(s) * kPrimes * kblk;

    // ---- sigma_k(A) with the digit offsets, B + sigma_k(B) ----
    // coefficient j of a(X^k) is +-a[t] with t = j k^{-1} mod 2N (minus when t >= N)
    uint64_t w[E];
    {
      uint64_t b[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t t = ((tau + e * T) * kinv) & (TWO_N - 1);
        const ulonglong2 v = acc[t & (N - 1)];
        w[e] = (t >= N ? 0ull - v.x : v.x) + dig_add;
        b[e] = t >= N ? 0ull - v.y : v.y;
      }
      th.sync();
#pragma unroll
      for (int e = 0; e < E; ++e) acc[tau + e * T].y += b[e];
    }

    // ---- residues, one prime after the other ----
    uint32_t ysum[E];  // of component 0 in the low, of component 1 in the high half
    uint32_t q = worker;
#pragma unroll 1
    for (uint32_t n3 = 0; n3 < kPrimesQf; ++n3) {
      const uint32_t p = a.cc.pr[q].p, p_inv = a.cc.pr[q].p_inv;
      const NttPrime np(a.cc.pr[q]);
      const SplitTw<kTrLogN, 6> tw{tw_all + q * N, a.tw_lo[q]};
      const uint32_t dig_bias = p - half;
      uint32_t y[2][E];
#pragma unroll 1
      for (uint32_t P = 0; P < PAIRS; ++P) {
        uint32_t x[2][E];
#pragma unroll
        for (int pp = 0; pp < 2; ++pp)
#pragma unroll
          for (int e = 0; e < E; ++e) x[pp][e] = biased_digit(w[e], a.base_log, 2 * P + pp) + dig_bias;  // in (0, 2p)
        ntt_forward<kTrLogN, E, 2, 2>(x, tw, xb, tau, np, th);
        const uint4 *g = reinterpret_cast<const uint4 *>(key + q * kblk + 2 * P * 2 * N + E * tau);
#pragma unroll
        for (int pp = 0; pp < 2; ++pp)
#pragma unroll
          for (int e = 0; e < E; ++e) x[pp][e] = cond_sub(x[pp][e], np.p8);  // < 16p -> < 8p
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int h = 0; h < E / 4; ++h) {
            const uint4 va = __ldg(g + (c * N) / 4 + h), vb = __ldg(g + ((2 + c) * N) / 4 + h);
            const uint32_t ga[4] = {va.x, va.y, va.z, va.w}, gb[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const int e = 4 * h + m;
              const uint64_t prod = static_cast<uint64_t>(x[0][e]) * ga[m] + static_cast<uint64_t>(x[1][e]) * gb[m];
              const uint32_t rr = redc(prod, p, p_inv);  // (0, 2p)
              y[c][e] = P == 0 ? rr : cond_sub(y[c][e] + rr, 4 * p);
            }
          }
      }
      ntt_inverse<kTrLogN, E, 2, 2>(y, tw, xb, tau, np, th);  // < 8p, CRT-scaled through the keys
      const uint64_t mp = a.cc.pr[q].Mp_mod64;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t t = qf_pack(y[0][e], y[1][e]);
        ysum[e] = n3 == 0 ? t : ysum[e] + t;
        ulonglong2 v = acc[tau + e * T];
        v.x -= static_cast<uint64_t>(y[0][e]) * mp;
        v.y -= static_cast<uint64_t>(y[1][e]) * mp;
        acc[tau + e * T] = v;
      }
      q = q == kPrimesQf - 1 ? 0 : q + 1;
    }

    // ---- float estimate of the product, the multiple of M3 ----
    uint32_t o[4][4];
#pragma unroll
    for (uint32_t P = 0; P < PAIRS; ++P) {
      uint32_t z[4][4];  // coefficients j and j + N/2 (slots q and q + 4) make one complex value
#pragma unroll
      for (int m = 0; m < 16; ++m)
        z[m / 4][m % 4] = __float_as_uint(__int2float_rn(
            static_cast<int32_t>(biased_digit(w[m % 8], a.base_log, 2 * P + m / 8)) - static_cast<int32_t>(half)));
      cfft_forward<kTrLogN - 1>(z, twf, xb, tau, th);
      const float4 *g = reinterpret_cast<const float4 *>(key + kPrimesQf * kblk + 2 * P * 2 * N + E * tau);
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {  // two complex key words of both rows per 16-byte load
          const float4 va = __ldg(g + (c * N) / 4 + k2), vb = __ldg(g + ((2 + c) * N) / 4 + k2);
          const float gr[2][2] = {{va.x, va.z}, {vb.x, vb.z}}, gi[2][2] = {{va.y, va.w}, {vb.y, vb.w}};
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int e = 2 * k2 + h;
            float sr = P == 0 ? 0.0f : __uint_as_float(o[2 * c][e]);
            float si = P == 0 ? 0.0f : __uint_as_float(o[2 * c + 1][e]);
#pragma unroll
            for (int pp = 0; pp < 2; ++pp) {
              const float zr = __uint_as_float(z[2 * pp][e]), zi = __uint_as_float(z[2 * pp + 1][e]);
              sr = fmaf(-zi, gi[pp][h], fmaf(zr, gr[pp][h], sr));
              si = fmaf(zi, gr[pp][h], fmaf(zr, gi[pp][h], si));
            }
            o[2 * c][e] = __float_as_uint(sr);
            o[2 * c + 1][e] = __float_as_uint(si);
          }
        }
    }
    cfft_inverse<kTrLogN - 1>(o, twf, xb, tau, th);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t u0 = qf_quotient(ysum[e] & 0xFFFFu, __uint_as_float(o[e / 4][e % 4]));
      const uint32_t u1 = qf_quotient(ysum[e] >> 16, __uint_as_float(o[2 + e / 4][e % 4]));
      ulonglong2 v = acc[tau + e * T];
      v.x += static_cast<uint64_t>(u0) * a.cc.M_mod64 - a.cc.qf_base;
      v.y += static_cast<uint64_t>(u1) * a.cc.M_mod64 - a.cc.qf_base;
      acc[tau + e * T] = v;
    }
    th.sync();
  }

  uint64_t *gout = a.glwe_out + static_cast<size_t>(ct) * 2 * N;
  for (uint32_t j = tau; j < N; j += T) {
    const ulonglong2 v = acc[j];
    gout[j] = v.x;
    gout[N + j] = v.y;
  }
}

bool trace_solo_supported(uint32_t logN, uint32_t base_log, uint32_t level) {
  if (logN != kTrLogN || base_log > 24 || (level != 2 && level != 4)) return false;
  uint32_t e = 0;
  while ((1u << e) < level * kTrN) ++e;
  return 63 + (base_log - 1) + e <= 98;
}

cudaError_t launch_trace_solo(const TraceArgs &a, uint32_t workers, cudaStream_t s) {
  if (workers < 1 || workers > kTrWorkers) return cudaErrorInvalidValue;
  const size_t smem = tr_smem_bytes(workers);
  const auto kern = a.level == 2 ? trace_solo_kernel<1> : trace_solo_kernel<2>;
  cudaError_t e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  kern<<<(a.batch + workers - 1) / workers, workers * kTrT, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace rosetta
