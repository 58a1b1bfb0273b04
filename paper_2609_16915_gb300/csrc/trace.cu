// RLWE trace of a batch of GLWE ciphertexts (k = 1), one 4-CTA cluster per
// ciphertext.
//
// The paper isolates the constant coefficient of an RLWE ciphertext with a
// trace: a logarithmic sequence of Galois automorphisms and additions under
// which every other coefficient cancels (Background, "Scheme Conversion and
// Other Primitives", RLWE Trace Computation; used after each blind rotation
// of the Cryptographic Lookup Protocol).  Step s (s = 0 .. log2 N - 1) uses
// the automorphism X -> X^k, k = 2^(log2 N - s) + 1:
//     c <- c + KS_s(sigma_k(c)),  KS_s(A', B') = (0, B') - sum_l D_l(A') * key_s[l]
// where key_s[l] encrypts sigma_k(S) 2^(64 - l beta) under S.  After all steps
// the phase is N times the input's constant coefficient (N has no inverse on
// the torus Z_{2^64}; the factor stays).
//
// The products sum_l D_l * key_s[l][c] are computed exactly with the same
// four-prime NTT + explicit CRT machinery as blind rotation, split the same
// way: CTA r of the cluster transforms for prime r and owns coefficients
// [rN/4, (r+1)N/4).  Per step:
//   1. owners gather sigma_k(A), sigma_k(B) for their quarter (distributed
//      shared memory), write the digits of sigma_k(A) and, after the barrier,
//      add sigma_k(B) to B;
//   2. prime-CTAs transform digit pairs, multiply by key_s, inverse-transform
//      and leave the CRT-scaled residues in their exchange buffer;
//   3. owners read them: (A, B) -= (X_0, X_1).
// Digits and residues travel in packed groups and the barriers order shared
// memory only, as in the blind rotation; the transforms exchange pairs; four
// CTAs fit an SM at N = 2048.  Measured, N = 2048, gadget 2^16 x 4, 1024
// ciphertexts: 1.84 ms with single-word exchanges, pushed residues and plain
// barriers, 1.38 ms with these, 1.25 with 2p and 8p loaded as values (NttPrime).  At N = 2048
// most of a large batch goes to trace_solo.cu.
#include <cooperative_groups.h>

#include "dsmem.cuh"
#include "internal.h"
#include "ntt.cuh"

namespace rosetta {
namespace cg = cooperative_groups;

template <int LOGN>
struct TrShape {
  static constexpr int N = 1 << LOGN;
  static constexpr int E = 8;
  static constexpr int T = N / E;
  static constexpr int Q = N / 4;
  // resident CTAs per SM the register allocation must allow (4 x 46-50 KB of
  // shared memory at N = 2048, 2 x 92-100 KB at 4096, four levels of 16- or 32-bit digits)
  static constexpr int MIN_CTAS = LOGN == 11 ? 4 : (LOGN == 12 ? 2 : 1);
  static constexpr int XB_WORDS = 2 * (N + N / 8);  // pairs of words; the outgoing residues (2N) afterwards
};

template <int LOGN, bool DIG16>
__global__ void __launch_bounds__(TrShape<LOGN>::T, TrShape<LOGN>::MIN_CTAS) trace_kernel(
    const __grid_constant__ TraceArgs a) {
  using B = TrShape<LOGN>;
  constexpr uint32_t N = B::N, T = B::T, Q = B::Q, TWO_N = 2 * N;
  constexpr int E = B::E;

  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = cluster.block_rank();
  const uint32_t ct = blockIdx.x / 4;
  const uint32_t tau = threadIdx.x;

  extern __shared__ __align__(16) unsigned char smem[];
  uint2 *tw_s = reinterpret_cast<uint2 *>(smem);              // [N]
  uint64_t *acc = reinterpret_cast<uint64_t *>(tw_s + N);     // [2][Q]
  uint32_t *xb = reinterpret_cast<uint32_t *>(acc + 2 * Q);
  uint32_t *dig = xb + B::XB_WORDS;                           // [level / 2][T][2 rows][2 slots], 16- or 32-bit

  const uint32_t p = a.cc.pr[rank].p;
  const NttPrime np(a.cc.pr[rank]);
  const uint32_t p_inv = a.cc.pr[rank].p_inv;

  for (uint32_t m = tau; m < N; m += T) tw_s[split_tw_slot<LOGN>(m)] = a.tw[rank * N + m];
  const SplitTw<LOGN, 3> tw{tw_s, a.tw_lo[rank]};
  const uint64_t *gin = a.glwe_in + static_cast<size_t>(ct) * 2 * N;
#pragma unroll
  for (int m = 0; m < 4; ++m) {  // thread tau owns local coefficients tau and tau + T of both components
    const uint32_t c = m / 2, jl = tau + (m % 2) * T;
    acc[c * Q + jl] = gin[c * N + rank * Q + jl];
  }
  cluster.sync();

  const uint32_t acc_s = smem_addr(acc), xb_s = smem_addr(xb);
  constexpr uint32_t GRP_BYTES = DIG16 ? 8 : 16;
  const uint32_t dig_t = smem_addr(dig) + tau * GRP_BYTES;
  const uint32_t res_t = xb_s + (rank * T + tau) * 16u;  // this owner's group in every prime-CTA
  const uint64_t dig_add = dig_offset(a.base_log, a.level);
  const uint32_t dig_bias = p - (1u << (a.base_log - 1));  // stored digits lie in [0, B): d + p = stored + bias
  const uint32_t pairs = a.level / 2;

#pragma unroll 1
  for (uint32_t s = 0; s < LOGN; ++s) {
    const uint32_t k = (1u << (LOGN - s)) + 1u;
    uint32_t kinv = k;  // k^{-1} mod 2^32 (Newton), hence mod 2N
#pragma unroll
    for (int it = 0; it < 5; ++it) kinv *= 2u - k * kinv;

    // ---- phase 1: gather sigma_k(c) for the owned quarter, digits of sigma_k(A) ----
    // coefficient j of a(X^k) is +-a[t] with t = j k^{-1} mod 2N (minus when t >= N)
    uint64_t v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t c = m / 2, j = rank * Q + tau + (m % 2) * T;
      const uint32_t t = (j * kinv) & (N - 1);
      v[m] = dsmem_ld_u64(dsmem_map(acc_s + (c * Q + (t % Q)) * 8u, t / Q));
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t j = rank * Q + tau + (m % 2) * T;
      if (((j * kinv) & (TWO_N - 1)) >= N) v[m] = 0ull - v[m];
    }
    v[0] += dig_add;
    v[1] += dig_add;
    for (uint32_t P = 0; P < pairs; ++P) {
      const uint32_t d00 = biased_digit(v[0], a.base_log, 2 * P), d01 = biased_digit(v[1], a.base_log, 2 * P);
      const uint32_t d10 = biased_digit(v[0], a.base_log, 2 * P + 1), d11 = biased_digit(v[1], a.base_log, 2 * P + 1);
      if constexpr (DIG16)
        *reinterpret_cast<uint2 *>(dig + (P * T + tau) * 2) = make_uint2(d00 | (d01 << 16), d10 | (d11 << 16));
      else
        *reinterpret_cast<uint4 *>(dig + (P * T + tau) * 4) = make_uint4(d00, d01, d10, d11);
    }
    cluster_sync_shared();
    // the remote reads are over: B + sigma_k(B) in place
    acc[Q + tau] += v[2];
    acc[Q + tau + T] += v[3];

    // ---- phase 2: digits x key_s for prime `rank` ----
    uint32_t oh[2][E];
    const uint32_t *kbase =
        a.keys + (static_cast<size_t>(s) * kPrimes + rank) * (static_cast<size_t>(a.level) * 2 * N);
#pragma unroll 1
    for (uint32_t P = 0; P < pairs; ++P) {
      // first-pass slot q of thread tau is coefficient tau + q N/8 of owner q / 2
      uint32_t x[2][E];
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const uint32_t ad = dsmem_map(dig_t, o) + P * T * GRP_BYTES;
        if constexpr (DIG16) {
          const uint2 w = dsmem_ld_v2_u32(ad);
          x[0][2 * o] = (w.x & 0xFFFFu) + dig_bias;
          x[0][2 * o + 1] = (w.x >> 16) + dig_bias;
          x[1][2 * o] = (w.y & 0xFFFFu) + dig_bias;
          x[1][2 * o + 1] = (w.y >> 16) + dig_bias;
        } else {
          const uint4 w = dsmem_ld_v4_u32(ad);
          x[0][2 * o] = w.x + dig_bias;
          x[0][2 * o + 1] = w.y + dig_bias;
          x[1][2 * o] = w.z + dig_bias;
          x[1][2 * o + 1] = w.w + dig_bias;
        }
      }
      ntt_forward<LOGN, E, 2, 2>(x, tw, xb, tau, np, CtaPairs());
      const uint4 *g = reinterpret_cast<const uint4 *>(kbase + static_cast<size_t>(2 * P) * 2 * N + E * tau);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t ga[E], gb[E];
#pragma unroll
        for (int kk = 0; kk < E / 4; ++kk) {
          const uint4 va = __ldg(g + (c * N) / 4 + kk), vb = __ldg(g + ((2 + c) * N) / 4 + kk);
          ga[4 * kk] = va.x; ga[4 * kk + 1] = va.y; ga[4 * kk + 2] = va.z; ga[4 * kk + 3] = va.w;
          gb[4 * kk] = vb.x; gb[4 * kk + 1] = vb.y; gb[4 * kk + 2] = vb.z; gb[4 * kk + 3] = vb.w;
        }
        if (c == 0) {
#pragma unroll
          for (int pp = 0; pp < 2; ++pp)
#pragma unroll
            for (int e = 0; e < E; ++e) x[pp][e] = cond_sub(x[pp][e], np.p8);
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const uint64_t prod = static_cast<uint64_t>(x[0][e]) * ga[e] + static_cast<uint64_t>(x[1][e]) * gb[e];
          const uint32_t rr = redc(prod, p, p_inv);
          oh[c][e] = (P == 0) ? rr : cond_sub(oh[c][e] + rr, 4 * p);
        }
      }
    }
    ntt_inverse<LOGN, E, 2, 2>(oh, tw, xb, tau, np, CtaPairs());
    __syncthreads();  // every exchange read done: the buffer takes the outgoing residues
    // (< 8p, CRT-scaled through the keys), one packed group (component, slot) per owner
#pragma unroll
    for (int o = 0; o < 4; ++o)
      *reinterpret_cast<uint4 *>(xb + (o * T + tau) * 4) =
          make_uint4(oh[0][2 * o], oh[0][2 * o + 1], oh[1][2 * o], oh[1][2 * o + 1]);
    cluster_sync_shared();

    // ---- phase 3: c <- c + (0, sigma_k(B)) - X on the owned quarter ----
    uint32_t yq[kPrimes][4];
#pragma unroll
    for (int pq = 0; pq < kPrimes; ++pq) {
      const uint4 w = dsmem_ld_v4_u32(dsmem_map(res_t, pq));
      yq[pq][0] = w.x;
      yq[pq][1] = w.y;
      yq[pq][2] = w.z;
      yq[pq][3] = w.w;
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      uint64_t sum = 0;
      uint32_t ysum = 0;
#pragma unroll
      for (int pq = 0; pq < kPrimes; ++pq) {
        const uint32_t y = yq[pq][m];
        sum += static_cast<uint64_t>(y) * a.cc.pr[pq].Mp_mod64;
        ysum += y >> 2;
      }
      const uint32_t u = crt_quotient(ysum);
      acc[(m / 2) * Q + tau + (m % 2) * T] -= sum - static_cast<uint64_t>(u) * a.cc.M_mod64;
    }
    cluster_sync_shared();
  }

  uint64_t *gout = a.glwe_out + static_cast<size_t>(ct) * 2 * N;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const uint32_t c = m / 2, jl = tau + (m % 2) * T;
    gout[c * N + rank * Q + jl] = acc[c * Q + jl];
  }
  cluster.sync();
}

static size_t trace_smem_bytes(uint32_t logN, uint32_t level, uint32_t base_log) {
  const size_t N = size_t(1) << logN, Q = N / 4;
  size_t b = N * sizeof(uint2) + 2 * Q * sizeof(uint64_t) + 2 * (N + N / 8) * sizeof(uint32_t) +
             level * Q * (base_log <= 16 ? sizeof(uint16_t) : sizeof(uint32_t));
  return (b + 15) & ~size_t(15);
}

template <int LOGN, bool DIG16>
static cudaError_t launch_trace_t(const TraceArgs &a, cudaStream_t s) {
  auto kern = trace_kernel<LOGN, DIG16>;
  const size_t smem = trace_smem_bytes(LOGN, a.level, a.base_log);
  cudaError_t e = allow_dynamic_smem(kern);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(4 * a.batch, 1, 1);
  cfg.blockDim = dim3(TrShape<LOGN>::T, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 4;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
  attr[1].val.clusterSchedulingPolicyPreference = br_cluster_policy(kern, TrShape<LOGN>::T, smem, cfg.gridDim.x);
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int LOGN>
static cudaError_t launch_trace_n(const TraceArgs &a, cudaStream_t s) {
  return a.base_log <= 16 ? launch_trace_t<LOGN, true>(a, s) : launch_trace_t<LOGN, false>(a, s);
}

cudaError_t launch_trace(const TraceArgs &a, uint32_t logN, cudaStream_t s) {
  switch (logN) {
    case 8: return launch_trace_n<8>(a, s);
    case 9: return launch_trace_n<9>(a, s);
    case 10: return launch_trace_n<10>(a, s);
    case 11: return launch_trace_n<11>(a, s);
    case 12: return launch_trace_n<12>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

// R <- (first ? 0 : R) + sum_i X^(e0 + i step) r_i over `polys` blocks r_i of
// `words` words (0 <= every exponent < N): coefficient j of X^e r is r[j - e] for
// j >= e and -r[j - e + N] below.
__global__ void __launch_bounds__(256) monomial_acc_kernel(uint64_t *__restrict__ R, const uint64_t *__restrict__ r,
                                                          size_t words, uint32_t logN, uint32_t polys, uint32_t e0,
                                                          uint32_t step, bool first) {
  const uint32_t N = 1u << logN;
  const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
  for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < words; i += stride) {
    const uint32_t j = static_cast<uint32_t>(i) & (N - 1);
    const size_t row = i - j;
    uint64_t v = first ? 0ull : R[i];
    uint32_t e = e0;
    for (uint32_t k = 0; k < polys; ++k, e += step) {
      const uint64_t *p = r + k * words + row;
      v += j >= e ? p[j - e] : 0ull - p[j - e + N];
    }
    R[i] = v;
  }
}

cudaError_t launch_monomial_acc(uint64_t *R, const uint64_t *r, uint32_t count, uint32_t logN, uint32_t polys, uint32_t e0,
                                uint32_t step, bool first, cudaStream_t s) {
  const size_t words = static_cast<size_t>(count) << logN;
  if (words == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  size_t blocks = (words + 255) / 256;
  const size_t cap = static_cast<size_t>(sms > 0 ? sms : 1) * 8;
  if (blocks > cap) blocks = cap;
  monomial_acc_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(R, r, words, logN, polys, e0, step, first);
  return cudaGetLastError();
}

}  // namespace rosetta
