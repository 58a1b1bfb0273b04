// Plaintext x ciphertext polynomial products (k = 1): (P * A, P * B + Q) in
// Z_{2^64}[X]/(X^N + 1) for every ciphertext of a batch, the linear mapping
// a_s(X) [[x]] + b_s(X) of the lookup protocol (Cryptographic Lookup Protocol,
// Steps 2 and 3), P any int64 polynomial.
//
// Each 64-bit word is two balanced base-2^32 digits, w = D1 2^32 + D0, and the
// product D1 * (P 2^32) + D0 * P with centred 64-bit P words stays below
// 2 N 2^31 2^63 <= 2^107 in magnitude, within the four 28-bit primes (product
// > 2^111.99).  So a component takes two forward and one inverse transform per
// prime, against the plaintext's two transformed rows.
//
// One CTA of N/8 threads per plaintext, ciphertext and component, no cluster: thread tau
// owns coefficients tau + e N/8, which are the transforms' first-pass slots, so
// words are read and written once, straight between global memory and registers,
// and nothing but the exchanges crosses threads.  The twiddles of one prime at a
// time lie in shared memory.  80 registers: 24 warps per SM at N = 2048.
// Launched behind the transform of its rows (rosetta_plaintext_mul_batch) it starts
// while that runs and waits for it only before the first product.
// Measured, N = 2048, 512 ciphertexts, the whole call with its host-side rows:
// 198 us with the trace kernel's one-step mode (base 2^16 digits, eight rows whose
// cross-component half was zero); 111 with one CTA of 128 registers for both
// components (71 us of it the kernel: 1.7 waves of long CTAs); 100 with these (64 us
// the kernel, 2.2 waves at the transforms' own rate of 10 butterflies per clock
// and SM); 95 with the early start.
#include <stdint.h>

#include "internal.h"
#include "ntt.cuh"

namespace rosetta {

// Words that the kernel before this one may still be writing when this one starts:
// an ordinary load that stays behind the wait (a read-only one, __ldg, may be moved before it).
__device__ __forceinline__ uint4 ld_row(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 8, LOGN >= 12 ? 1 : LOGN == 8 ? 20 : 3 * (2048 >> LOGN))
    plain_mul_kernel(const __grid_constant__ PlainMulArgs a) {
  constexpr uint32_t N = 1u << LOGN, T = N / 8;
  constexpr int E = 8;
  extern __shared__ __align__(16) unsigned char smem[];
  uint2 *tw_s = reinterpret_cast<uint2 *>(smem);
  uint32_t *xb = reinterpret_cast<uint32_t *>(tw_s + N);
  const uint32_t tau = threadIdx.x;
  const uint32_t which = blockIdx.x / (2 * a.batch);           // plaintext
  const size_t poly = blockIdx.x - which * (2 * a.batch);      // 2 ciphertext + component
  const uint64_t *gin = a.glwe_in + poly * N + tau;
  const uint64_t *add = (poly & 1u) != 0 && a.plain_add ? a.plain_add + static_cast<size_t>(which) * N : nullptr;

  uint64_t w[E], s[E];
  uint32_t ysum[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    w[e] = gin[e * T] + ((1ull << 63) + (1ull << 31));  // both digits plus 2^31
    s[e] = add ? add[tau + e * T] : 0ull;
    ysum[e] = 0;
  }

#pragma unroll 1
  for (uint32_t q = 0; q < kPrimes; ++q) {
    const uint32_t p = a.cc.pr[q].p, p_inv = a.cc.pr[q].p_inv;
    const NttPrime np(a.cc.pr[q]);
    // digit u - 2^31 mod p: u = (u >> 28) 2^28 + .., 2^28 = p + g with g < 2^18;
    // 2^31 = 8p + 8g
    const uint32_t bias = p - 8 * ((1u << 28) - p);
    __syncthreads();  // the previous prime's twiddles and exchanges are done with
    for (uint32_t m = tau; m < N; m += T) tw_s[split_tw_slot<LOGN>(m)] = a.tw[q * N + m];
    __syncthreads();
    const SplitTw<LOGN, 3> tw{tw_s, a.tw_lo[q]};
    uint32_t x[2][E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t hi = static_cast<uint32_t>(w[e] >> 32), lo = static_cast<uint32_t>(w[e]);
      x[0][e] = cond_sub(hi - (hi >> 28) * p, p) + bias;  // < 2p
      x[1][e] = cond_sub(lo - (lo >> 28) * p, p) + bias;
    }
    ntt_forward<LOGN, E, 2, 2>(x, tw, xb, tau, np, CtaPairs());
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the plaintext's rows are there (key_pending)
    const uint4 *g = reinterpret_cast<const uint4 *>(a.keys + (static_cast<size_t>(which) * kPrimes + q) * 2 * N + E * tau);
    uint32_t o[1][E];
#pragma unroll
    for (int k = 0; k < E / 4; ++k) {
      const uint4 v0 = ld_row(g + k), v1 = ld_row(g + N / 4 + k);
      const uint32_t k0[4] = {v0.x, v0.y, v0.z, v0.w}, k1[4] = {v1.x, v1.y, v1.z, v1.w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int e = 4 * k + m;
        const uint64_t prod = static_cast<uint64_t>(cond_sub(x[0][e], np.p8)) * k0[m] +
                              static_cast<uint64_t>(cond_sub(x[1][e], np.p8)) * k1[m];
        o[0][e] = redc(prod, p, p_inv);
      }
    }
    // the exchange buffer changes from pairs to single words, whose warp-local
    // parts lie elsewhere: every forward read first
    __syncthreads();
    ntt_inverse<LOGN, E, 1, 1>(o, tw, xb, tau, np, CtaThreads());  // < 8p, CRT-scaled through the keys
    const uint64_t mp = a.cc.pr[q].Mp_mod64;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      s[e] += static_cast<uint64_t>(o[0][e]) * mp;
      ysum[e] += o[0][e] >> 2;
    }
  }
  uint64_t *gout = a.glwe_out + static_cast<size_t>(blockIdx.x) * N + tau;
#pragma unroll
  for (int e = 0; e < E; ++e) gout[e * T] = s[e] - static_cast<uint64_t>(crt_quotient(ysum[e])) * a.cc.M_mod64;
}

template <int LOGN>
static cudaError_t launch_pm_t(const PlainMulArgs &a, cudaStream_t s) {
  constexpr size_t N = size_t(1) << LOGN;
  const size_t smem = N * sizeof(uint2) + 2 * (N + N / 8) * sizeof(uint32_t);
  auto kern = plain_mul_kernel<LOGN>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * a.batch * a.polys, 1, 1);
  cfg.blockDim = dim3(N / 8, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.key_pending ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

cudaError_t launch_plaintext_mul(const PlainMulArgs &a, uint32_t logN, cudaStream_t s) {
  switch (logN) {
    case 8: return launch_pm_t<8>(a, s);
    case 9: return launch_pm_t<9>(a, s);
    case 10: return launch_pm_t<10>(a, s);
    case 11: return launch_pm_t<11>(a, s);
    case 12: return launch_pm_t<12>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rosetta
