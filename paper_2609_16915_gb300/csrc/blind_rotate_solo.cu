// Blind rotation for N = 2048 and one gadget level at full batches: one worker
// of 256 threads per ciphertext, three workers per SM, no cluster.
//
// Same construction as the cluster kernel (blind_rotate.cu), whose four CTAs
// spend a quarter of their multiply-pipe work on the fourth 28-bit prime: the
// product X needs 98 bits, three primes hold 84.  Here the exact residues come
// from three primes only, and the missing multiple of their product M3 from
// an estimate of X / M3 by single-precision complex transforms (cfft.cuh),
// whose worst-case error stays below 0.1 of M3 for every accepted set.  The
// words are those of the exact product.  The float transforms need half the
// points, run mostly on the float pipe that the integer butterflies leave
// idle, and cost about a third of a prime.
//
// Work split.  Worker thread tau (0 .. 255) owns coefficients tau + 256 e of
// both components: the transforms' first-pass slots.  So a step's digits stay
// in registers, every residue ends in the thread that needs it, and the only
// words that cross threads are the rotated accumulator's and the transforms'
// exchanges; all barriers are the worker's own (256 threads).  Per step: digits
// of X^{a~} ACC - ACC; the float estimate; then per prime two forward
// transforms, the products with BSK_i, two inverse transforms, and
// acc += y (M3 / p) in place.  The workers take the primes in different
// orders and share one copy of the twiddle tables; the float transforms come
// last, when the digits' registers are free.
//
// What bounds it: at three workers (24 warps, 80 registers, no spills) the
// shared-memory pipe, the integer-multiply pipe and the issue slots are each about
// two thirds busy.  Hence the layouts: both polynomials of a transform cross the
// exchange buffer as 8-byte pairs, all four float planes as 16-byte elements,
// both components of an accumulator word lie together, and the first six
// stages' twiddles come from the constant bank.  Measured, n = 742, batch 4096:
// 235.9 ms with the cluster kernel; here 219.3 with the float transforms
// first and spills (172 bytes), 190.1 without, 184.5 with the paired exchanges,
// 171 with 2p and 8p loaded as values (NttPrime: 6079 -> 5470 instructions a step;
// 456 ciphertexts, one wave: 28.8, 24.5, 21.2, 20.6, 19.1 ms).  Two workers with 128
// registers: 14.9 ms per 304.  The float quotient as the fourth CTA of a
// cluster gained 1.6 % only: a cluster moves at the pace of its most loaded SM.
#include <stdint.h>

#include "cfft.cuh"
#include "check.cuh"
#include "internal.h"
#include "ntt.cuh"

namespace rosetta {

namespace {

constexpr int kLogN = 11;
constexpr uint32_t kN = 1u << kLogN, kT = kN / 8;   // threads of a worker
constexpr uint32_t kWorkers = 3;                    // per CTA (and SM)
constexpr uint32_t kTwF = 352;                      // float4 entries of the pass table (341, padded)
constexpr uint32_t kXbWords = 2 * NttShape<kLogN, 8>::XB_WORDS;  // two integer polynomials; four float ones
static_assert(kXbWords >= 4 * (kN / 2), "exchange buffer");

__host__ __device__ constexpr size_t solo_worker_bytes(uint32_t n) {
  return 2 * kN * sizeof(uint64_t) + kXbWords * sizeof(uint32_t) + (((n + 1) * sizeof(uint16_t) + 15) & ~size_t(15));
}
__host__ __device__ constexpr size_t solo_table_bytes() {
  return kPrimesQf * kN * sizeof(uint2) + kTwF * sizeof(float4);
}

}  // namespace

// acc[e T] += y[.][e] mp, both components
__device__ __forceinline__ void add_residues(ulonglong2 *acc, const uint32_t (&y)[2][8], uint64_t mp) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    ulonglong2 v = acc[e * kT];
    v.x += static_cast<uint64_t>(y[0][e]) * mp;
    v.y += static_cast<uint64_t>(y[1][e]) * mp;
    acc[e * kT] = v;
  }
}

// Shared memory: twiddles of the three primes uint2 [3][N], the float pass
// table float4 [352], then per worker acc uint64 [N][2], the exchange buffer,
// the switched mask and body uint16 [n+1].
__global__ void __launch_bounds__(kWorkers *kT, 1) blind_rotate_solo_kernel(const __grid_constant__ BrArgs a) {
  constexpr uint32_t N = kN, T = kT, TWO_N = 2 * N;
  constexpr int E = 8;
  extern __shared__ __align__(16) unsigned char smem[];
  uint2 *tw_all = reinterpret_cast<uint2 *>(smem);
  float4 *twf = reinterpret_cast<float4 *>(tw_all + kPrimesQf * N);
  const uint32_t worker = __shfl_sync(0xffffffffu, threadIdx.x / T, 0);  // (warp-uniform for the compiler)
  const uint32_t tau = threadIdx.x % T;
  unsigned char *own = smem + solo_table_bytes() + worker * solo_worker_bytes(a.n);
  ulonglong2 *acc = reinterpret_cast<ulonglong2 *>(own);  // [N], both components of a coefficient together
  uint32_t *xb = reinterpret_cast<uint32_t *>(acc + N);
  uint16_t *atil = reinterpret_cast<uint16_t *>(xb + kXbWords);

  for (uint32_t m = threadIdx.x; m < kPrimesQf * N; m += blockDim.x) {
    const uint32_t q = m / N, idx = m % N;
    tw_all[q * N + split_tw_slot<kLogN>(idx)] = a.tw[m];
  }
  const float4 *twf_src = reinterpret_cast<const float4 *>(a.tw + kPrimesQf * N);
  for (uint32_t m = threadIdx.x; m < kTwF; m += blockDim.x) twf[m] = twf_src[m];
  __syncthreads();

  const uint32_t ct = blockIdx.x * (blockDim.x / T) + worker;
  if (ct >= a.batch) return;  // the whole worker; from here on it meets only its own barrier
  const GroupThreads th{worker + 1u, T};

  const uint64_t *lwe = a.lwe_in + static_cast<size_t>((a.lwe_first + ct) % a.lwe_count) * (a.n + 1);
  constexpr uint32_t SH = 63 - kLogN;  // 64 - log2(2N)
  for (uint32_t i = tau; i <= a.n; i += T)
    atil[i] = static_cast<uint16_t>(((lwe[i] + (1ull << (SH - 1))) >> SH) & (TWO_N - 1));
  th.sync();
  {
    const uint32_t btil = atil[a.n];
    if (a.glwe_in) {
      // encrypted test polynomial: ACC = X^{-b~} (A, B) for this ciphertext
      const uint64_t *gin = a.glwe_in + static_cast<size_t>(ct) * 2 * N;
      for (uint32_t j = tau; j < N; j += T) {
        const uint32_t e = (j + btil) & (TWO_N - 1);
        const uint64_t v0 = gin[e & (N - 1)], v1 = gin[N + (e & (N - 1))];
        acc[j] = e >= N ? make_ulonglong2(0ull - v0, 0ull - v1) : make_ulonglong2(v0, v1);
      }
    } else {
      // trivial GLWE (0, X^{-b~} v) of the test polynomial of this ciphertext's LUT
      uint32_t li = 0;
      if (a.lut_index) {
        li = a.lut_index[ct];
        if (li >= a.num_luts) {  // never read outside the LUT array
          if (tau == 0 && a.err_flag) atomicExch(a.err_flag, 1u);
          li = 0;
        }
      }
      const uint64_t *lut = a.lut + (static_cast<size_t>(li) << a.msg_bits);
      const uint32_t box = N >> a.msg_bits, h = box >> 1;
      for (uint32_t j = tau; j < N; j += T) {
        // (X^{2N - b~} v)[j] = +-v[t], t = (j + b~) mod 2N folded into [0, N)
        const uint32_t e = (j + btil) & (TWO_N - 1);
        const uint32_t t = e & (N - 1);
        const uint64_t v = (t < N - h) ? lut[(t + h) / box] : (0ull - lut[0]);
        acc[j] = make_ulonglong2(0ull, (e >= N) ? 0ull - v : v);
      }
    }
  }
  th.sync();

  // one level: the digit of a word is its top base_log bits, rounded, as a
  // signed number (base_log <= 24: they lie in the upper half)
  const uint64_t round_add = 1ull << (63 - a.base_log);
  const uint32_t dig_sh = 32 - a.base_log;
  constexpr uint32_t kblk = 2 * 2 * N;  // words of one step's key block per prime

#pragma unroll 1
  for (uint32_t i = 0; i < a.n; ++i) {
    const uint32_t at = atil[i];
    if (at == 0) continue;  // X^0 ACC - ACC = 0: the step adds nothing
    const uint32_t *key = a.bsk + static_cast<size_t>(i) * kPrimes * kblk;
    const bool key_ok =
        dbg_ok(a.bsk_words == 0 || (static_cast<size_t>(i) + 1) * kPrimes * kblk <= a.bsk_words, a.err_flag);

    // ---- digits of the rotated difference, (X^a P)[j] = +-P[(j - a) mod 2N] ----
    int32_t d[2][E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t j = tau + e * T;
      const uint32_t t = (j + TWO_N - at) & (TWO_N - 1);
      const ulonglong2 v = acc[t & (N - 1)], o = acc[j];
      const uint64_t d0 = (t >= N ? 0ull - v.x : v.x) - o.x + round_add;
      const uint64_t d1 = (t >= N ? 0ull - v.y : v.y) - o.y + round_add;
      d[0][e] = static_cast<int32_t>(d0 >> 32) >> dig_sh;
      d[1][e] = static_cast<int32_t>(d1 >> 32) >> dig_sh;
    }

    // ---- residues, one prime after the other ----
    uint32_t ysum[E];  // of component 0 in the low, of component 1 in the high half
    uint32_t y[2][E];
    uint32_t q = worker;
#pragma unroll 1
    for (uint32_t k = 0; k < kPrimesQf; ++k) {
      if (k > 0) {
        // add the previous prime's share before its residues are overwritten
        add_residues(acc + tau, y, a.cc.pr[q].Mp_mod64);
        q = q == kPrimesQf - 1 ? 0 : q + 1;
      }
      const uint32_t p = a.cc.pr[q].p, p_inv = a.cc.pr[q].p_inv;
      const NttPrime np(a.cc.pr[q]);
      const SplitTw<kLogN, 6> tw{tw_all + q * N, a.tw_lo[q]};
      uint32_t x[2][E];
#pragma unroll
      for (int pp = 0; pp < 2; ++pp)
#pragma unroll
        for (int e = 0; e < E; ++e) x[pp][e] = static_cast<uint32_t>(d[pp][e]) + p;  // in (0, 2p)
      ntt_forward<kLogN, E, 2, 2>(x, tw, xb, tau, np, th);
      const uint4 *g = reinterpret_cast<const uint4 *>(key + q * kblk + E * tau);
#pragma unroll
      for (int pp = 0; pp < 2; ++pp)
#pragma unroll
        for (int e = 0; e < E; ++e) x[pp][e] = cond_sub(x[pp][e], np.p8);  // < 16p -> < 8p
#pragma unroll
      for (int h = 0; h < E / 4; ++h) {
        uint4 w[2][2];  // [component][row]
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int pp = 0; pp < 2; ++pp)
            w[c][pp] = key_ok ? __ldg(g + ((2 * pp + c) * N) / 4 + h) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint32_t ga[4] = {w[c][0].x, w[c][0].y, w[c][0].z, w[c][0].w};
          const uint32_t gb[4] = {w[c][1].x, w[c][1].y, w[c][1].z, w[c][1].w};
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            // forward outputs < 8p, BSK words < p in Montgomery form: the pair
            // sum stays below 16 p^2 < p * 2^32
            const int e = 4 * h + m;
            const uint64_t prod = static_cast<uint64_t>(x[0][e]) * ga[m] + static_cast<uint64_t>(x[1][e]) * gb[m];
            y[c][e] = redc(prod, p, p_inv);  // (0, 2p)
          }
        }
      }
      ntt_inverse<kLogN, E, 2, 2>(y, tw, xb, tau, np, th);  // < 8p, CRT-scaled through the keys
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t t = qf_pack(y[0][e], y[1][e]);
        ysum[e] = k == 0 ? t : ysum[e] + t;
      }
    }

    // ---- float estimate of the product ----
    {
      uint32_t z[4][4];  // coefficients j and j + N/2 (slots q and q + 4) make one complex value
#pragma unroll
      for (int m = 0; m < 16; ++m)
        z[m / 4][m % 4] = __float_as_uint(__int2float_rn(d[m / 8][m % 8]));
      cfft_forward<kLogN - 1>(z, twf, xb, tau, th);
      const float4 *g = reinterpret_cast<const float4 *>(key + kPrimesQf * kblk + E * tau);
      uint32_t o[4][4];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k) {  // two complex key words of both rows per 16-byte load
          const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          const float4 va = key_ok ? __ldg(g + (c * N) / 4 + k) : zero;
          const float4 vb = key_ok ? __ldg(g + ((2 + c) * N) / 4 + k) : zero;
          const float gr[2][2] = {{va.x, va.z}, {vb.x, vb.z}}, gi[2][2] = {{va.y, va.w}, {vb.y, vb.w}};
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int e = 2 * k + h;
            float sr = 0.0f, si = 0.0f;
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
      cfft_inverse<kLogN - 1>(o, twf, xb, tau, th);

      // ---- the last prime's share and the multiple of M3 ----
      const uint64_t mp = a.cc.pr[q].Mp_mod64;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const uint32_t u0 = qf_quotient(ysum[e] & 0xFFFFu, __uint_as_float(o[e / 4][e % 4]));
        const uint32_t u1 = qf_quotient(ysum[e] >> 16, __uint_as_float(o[2 + e / 4][e % 4]));
        ulonglong2 v = acc[tau + e * T];
        v.x += a.cc.qf_base + static_cast<uint64_t>(y[0][e]) * mp - static_cast<uint64_t>(u0) * a.cc.M_mod64;
        v.y += a.cc.qf_base + static_cast<uint64_t>(y[1][e]) * mp - static_cast<uint64_t>(u1) * a.cc.M_mod64;
        acc[tau + e * T] = v;
      }
    }
    th.sync();
  }

  if (a.glwe_out) {
    // ---- the rotated accumulator itself ----
    uint64_t *gout = a.glwe_out + static_cast<size_t>(ct) * 2 * N;
    for (uint32_t j = tau; j < N; j += T) {
      const ulonglong2 v = acc[j];
      gout[j] = v.x;
      gout[N + j] = v.y;
    }
  } else {
    // ---- sample extraction of the constant coefficient ----
    uint64_t *out = a.lwe_big_out + static_cast<size_t>(ct) * (N + 1);
    for (uint32_t j = tau; j < N; j += T) out[j == 0 ? 0 : N - j] = (j == 0) ? acc[j].x : 0ull - acc[j].x;
    if (tau == 0) out[N] = acc[0].y;
  }
}

bool br_solo_supported(uint32_t logN, uint32_t level, uint32_t base_log) {
  return logN == kLogN && level == 1 && base_log <= 24;
}

size_t br_solo_smem_bytes(uint32_t n, uint32_t workers) { return solo_table_bytes() + workers * solo_worker_bytes(n); }

cudaError_t launch_blind_rotate_solo(const BrArgs &a, uint32_t workers, cudaStream_t s) {
  if (workers < 1 || workers > kWorkers) return cudaErrorInvalidValue;
  const size_t smem = br_solo_smem_bytes(a.n, workers);
  cudaError_t e = allow_dynamic_smem(blind_rotate_solo_kernel);
  if (e != cudaSuccess) return e;
  blind_rotate_solo_kernel<<<(a.batch + workers - 1) / workers, workers * kT, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace rosetta
