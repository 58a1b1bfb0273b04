// Blind rotation for small batches, where a step's latency counts and SMs are
// idle: a cluster of two CTAs per prime for each ciphertext, one per component.
//
// Same construction and words as blind_rotate.cu / blind_rotate3.cu, with half
// the work per CTA and step.  CTA (q, c) works modulo prime q on component c: it
// keeps the whole component of the accumulator, cuts its digits, transforms its
// rows, multiplies them by both components of the key, sends its partner (q, 1-c)
// the half that belongs there, transforms the sum back, sends the residues to the
// other primes' CTAs of component c and does the CRT of all its coefficients
// (once per prime, where the other kernels do it once).  Thread tau owns
// coefficients tau + e N/8, which are the transforms' first-pass slots, so
// rotated words and digits never leave the CTA.  The next step's key words are
// requested a step ahead (registers are plentiful with few CTAs per SM).
//
// There is no cluster barrier in a step.  Partial products and residues are
// stored straight into the receiver's shared memory (st.async), each store
// counted by an mbarrier there.  Both may arrive a step early, never two: the
// sender of a step's partial products (residues) has received this CTA's of the
// step before, and this CTA sent those after it had waited for and read what it
// got two steps back.  So each kind has two buffers and two mbarriers, by step
// parity, and a phase of an mbarrier only ever counts one step's bytes.
// Measured, n = 742, N = 2048, one ciphertext: 3.78 ms with four CTAs and three
// cluster barriers per step (blind_rotate.cu); 3.92 with the whole accumulator in
// every one of four CTAs and one barrier (the arithmetic, not the barriers, is
// most of a step); 2.85 with two CTAs per prime and two barriers; 2.54 with
// st.async, 2.42 with 2p and 8p loaded as values (NttPrime).
//
// Every wait gives up after about two seconds and raises the error flag.  The CTA
// then finishes the step with what it has, all threads leave the loop after it (no
// further words are sent; the next step's mbarriers are armed once, to count what still
// comes), and nothing is written out.  Its peers miss its words in the next step and leave the same way, so every CTA
// comes to the cluster barrier at the end; the CTA that gave up then waits, with a limit,
// for the words that were still on their way to it: the rest of its last step's and, a
// step early, those of the next.
#include <cooperative_groups.h>

#include <type_traits>

#include "check.cuh"
#include "dsmem.cuh"
#include "internal.h"
#include "ntt.cuh"
#include "tcgen.cuh"

namespace rosetta {
namespace cg = cooperative_groups;

namespace {

// A load that stays where it is written (the next step's key words).
__device__ __forceinline__ uint4 ld_key(const uint32_t *p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Key words of NP rows at a thread's 8 positions: [row][own, partner's component][half].
template <int NP>
struct RowKeys {
  uint4 w[NP][2][2];
  __device__ __forceinline__ void load(const uint32_t *own, const uint32_t *other, uint32_t row_words, bool ok,
                                       uint32_t rows = NP) {
#pragma unroll
    for (int r = 0; r < NP; ++r)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool there = ok && static_cast<uint32_t>(r) < rows;
        w[r][0][k] = there ? ld_key(own + r * row_words + 4 * k) : make_uint4(0u, 0u, 0u, 0u);
        w[r][1][k] = there ? ld_key(other + r * row_words + 4 * k) : make_uint4(0u, 0u, 0u, 0u);
      }
  }
};

__device__ __forceinline__ uint32_t word(const uint4 &v, int m) { return m == 0 ? v.x : m == 1 ? v.y : m == 2 ? v.z : v.w; }

// o[e] (+)= sum_r x[r][e] key[r][side]
template <bool P31, int NP>
__device__ __forceinline__ void mac(uint32_t (&o)[8], const uint32_t (&x)[NP][8], const RowKeys<NP> &key, int side,
                                    bool first, uint32_t p, uint32_t p_inv) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    uint64_t prod = static_cast<uint64_t>(x[0][e]) * word(key.w[0][side][e / 4], e % 4);
    if constexpr (NP == 2) prod += static_cast<uint64_t>(x[1][e]) * word(key.w[1][side][e / 4], e % 4);
    const uint32_t rr = redc(prod, p, p_inv);  // (0, 2p)
    if (first)
      o[e] = rr;
    else
      o[e] = P31 ? cond_sub(o[e], p) + cond_sub(rr, p) : cond_sub(o[e] + rr, 4 * p);
  }
}

template <int LOGN, int LEV>
struct BrsShape {
  static constexpr int N = 1 << LOGN, T = N / 8;
  // one polynomial at a time with one level, else pairs
  static constexpr int XB_WORDS = (LEV == 1 ? 1 : 2) * (N + N / 8);
};

__host__ __device__ constexpr size_t brs_smem(size_t N, bool single, size_t n, size_t primes) {
  return (6 * sizeof(uint64_t) + N * sizeof(uint2) + N * sizeof(uint64_t) + (single ? 1 : 2) * (N + N / 8) * sizeof(uint32_t) +
          2 * N * sizeof(uint32_t) + 2 * (primes - 1) * N * sizeof(uint32_t) + (n + 1) * sizeof(uint16_t) + 15) & ~size_t(15);
}

}  // namespace

// PRIMES: 4 (28-bit set) or 3 (31-bit set).  LEV > 0: levels known at compile
// time; 0: from the arguments.  Shared memory, all of it dynamic, so that
// brs_smem is the whole of what a CTA takes: mbarriers uint64 [4] (partial
// products, residues of even steps; of odd ones), a word raised when a wait gives up (and
// padding to 16 bytes), twiddles of prime q uint2 [N], acc uint64 [N], exchange buffer, received
// partial products uint32 [2 steps][2][T][4], received
// residues uint32 [2 steps][PRIMES - 1][2][T][4], switched mask and body uint16 [n+1].
template <int LOGN, int LEV, int PRIMES>
__global__ void __launch_bounds__(BrsShape<LOGN, LEV>::T, LOGN == 11 ? 2 : 1)
    blind_rotate_small_kernel(const __grid_constant__ BrArgs a) {
  using B = BrsShape<LOGN, LEV>;
  constexpr uint32_t N = B::N, T = B::T, TWO_N = 2 * N;
  constexpr int E = 8;
  constexpr bool P31 = PRIMES == kPrimes31;
  constexpr uint16_t kStopped = 0xFFFF;  // in place of a switched mask word (below 2N)

  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = cluster.block_rank();
  const uint32_t q = rank / 2, comp = rank % 2;
  const uint32_t ct = blockIdx.x / (2 * PRIMES);
  const uint32_t tau = threadIdx.x;
  if (!dbg_ok(ct < a.batch, a.err_flag)) return;  // the whole cluster shares ct

  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  volatile uint32_t *stop = reinterpret_cast<uint32_t *>(bars + 4);
  uint2 *tw_s = reinterpret_cast<uint2 *>(bars + 6);
  uint64_t *acc = reinterpret_cast<uint64_t *>(tw_s + N);
  uint32_t *xb = reinterpret_cast<uint32_t *>(acc + N);
  uint4 *part = reinterpret_cast<uint4 *>(xb + B::XB_WORDS);
  uint4 *res = part + 4 * T;
  uint16_t *atil = reinterpret_cast<uint16_t *>(res + 2 * (PRIMES - 1) * 2 * T);

  const uint32_t p = a.cc.pr[q].p;
  const NttPrime npr(a.cc.pr[q]);
  const uint32_t p_inv = a.cc.pr[q].p_inv;
  const uint32_t level = LEV > 0 ? static_cast<uint32_t>(LEV) : a.level;

  if (tau == 0) {
    *stop = 0u;
    for (int b = 0; b < 4; ++b) mbar_init(smem_addr(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (uint32_t m = tau; m < N; m += T) tw_s[split_tw_slot<LOGN>(m)] = a.tw[q * N + m];
  const SplitTw<LOGN, 3> tw{tw_s, a.tw_lo[q]};
  const uint64_t *lwe = a.lwe_in + static_cast<size_t>((a.lwe_first + ct) % a.lwe_count) * (a.n + 1);
  constexpr uint32_t SH = 63 - LOGN;  // 64 - log2(2N)
  for (uint32_t i = tau; i <= a.n; i += T)
    atil[i] = static_cast<uint16_t>(((lwe[i] + (1ull << (SH - 1))) >> SH) & (TWO_N - 1));
  __syncthreads();
  {
    const uint32_t btil = atil[a.n];
    if (a.glwe_in) {
      // encrypted test polynomial: ACC = X^{-b~} (A, B) for this ciphertext
      const uint64_t *gin = a.glwe_in + (static_cast<size_t>(ct) * 2 + comp) * N;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const uint32_t j = tau + m * T, e = (j + btil) & (TWO_N - 1);
        const uint64_t v = gin[e & (N - 1)];
        acc[j] = e >= N ? 0ull - v : v;
      }
    } else {
      // trivial GLWE (0, X^{-b~} v) of the test polynomial of this ciphertext's LUT
      uint32_t li = 0;
      if (a.lut_index) {
        li = a.lut_index[ct];
        if (li >= a.num_luts) {  // never read outside the LUT array
          if (tau == 0 && rank == 0 && a.err_flag) atomicExch(a.err_flag, 1u);
          li = 0;
        }
      }
      const uint64_t *lut = a.lut + (static_cast<size_t>(li) << a.msg_bits);
      const uint32_t box = N >> a.msg_bits, h = box >> 1;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        // (X^{2N - b~} v)[j] = +-v[t], t = (j + b~) mod 2N folded into [0, N)
        const uint32_t j = tau + m * T, e = (j + btil) & (TWO_N - 1), t = e & (N - 1);
        const uint64_t v = (t < N - h) ? lut[(t + h) / box] : (0ull - lut[0]);
        acc[j] = comp == 0 ? 0ull : (e >= N ? 0ull - v : v);
      }
    }
  }
  cluster.sync();  // the peers have started and their mbarriers are ready

  const uint64_t dig_add = dig_offset(a.base_log, level);
  const uint32_t dig_bias = p - (1u << (a.base_log - 1));
  const uint32_t bar0 = smem_addr(bars), part_s = smem_addr(part), res_s = smem_addr(res);
  const uint32_t part_to = dsmem_map(part_s + tau * 16u, rank ^ 1u), part_bar_to = dsmem_map(bar0, rank ^ 1u);
#ifdef ROSETTA_DEBUG
  const long long wait_cycles = a.wait_cycles ? a.wait_cycles : kWaitCycles;
#else
  constexpr long long wait_cycles = kWaitCycles;
#endif
  const size_t kblk = static_cast<size_t>(2 * level) * 2 * N;  // words of one step's key block per prime
  // this thread's words of the first row of component comp, own and partner's column
  const uint32_t *key_own = a.bsk + q * kblk + (static_cast<size_t>(comp) * level * 2 + comp) * N + E * tau;
  const uint32_t *key_oth = a.bsk + q * kblk + (static_cast<size_t>(comp) * level * 2 + (comp ^ 1u)) * N + E * tau;
  const auto step_off = [&](uint32_t i) { return static_cast<size_t>(i) * PRIMES * kblk; };
  const auto key_ok = [&](uint32_t i) {
    return dbg_ok(a.bsk_words == 0 || (static_cast<size_t>(i) * PRIMES + q + 1) * kblk <= a.bsk_words, a.err_flag);
  };
  constexpr int NP0 = LEV == 1 ? 1 : 2;  // rows transformed together
  RowKeys<NP0> key;                      // of the first rows of the coming step
  const auto load_first = [&](uint32_t i) {
    key.load(key_own + step_off(i), key_oth + step_off(i), 2 * N, key_ok(i), level);
  };
  // next step to run; a step with a~ = 0 adds nothing
  const auto next_step = [&](uint32_t i) {
    while (i < a.n && atil[i] == 0) ++i;
    return i;
  };
  uint32_t i = next_step(0), step = 0;
  if (i < a.n) load_first(i);
#pragma unroll 1
  while (i < a.n) {
    const uint32_t at = atil[i];
    const uint32_t odd = step & 1u, phase = (step >> 1) & 1u;
    const uint32_t part_bar = bar0 + 16u * odd, res_bar = part_bar + 8u;
    if (tau == 0) {
      expect_tx(part_bar, N * 4u);
      expect_tx(res_bar, (PRIMES - 1) * N * 4u);
    }
    // A wait of the last step gave up: the same for all threads, as it was written before that
    // step's last barrier and is not again before this one's first.  (The word is needed
    // anyway; a flag of its own, or a barrier that reduces the threads', cost 1 to 3 %.)
    if (at == kStopped) break;
    // ---- rotated difference, (X^a P)[j] = +-P[(j - a) mod 2N], digit offsets added ----
    uint64_t w[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t j = tau + e * T, t = (j + TWO_N - at) & (TWO_N - 1);
      const uint64_t v = acc[t & (N - 1)];
      w[e] = (t >= N ? 0ull - v : v) - acc[j] + dig_add;
    }
    const uint32_t next = next_step(i + 1);
    const auto wait = [&](uint32_t bar, uint32_t parity) {
      if (!mbar_wait_cluster(bar, parity, wait_cycles)) {
        *stop = 1u;
        if (next < a.n) atil[next] = kStopped;
        if (a.err_flag) atomicExch(a.err_flag, 2u);
      }
    };

    // ---- forward transforms, products with both components of the key ----
    uint32_t own[E], oth[E];
    const auto rows = [&](auto &k, auto np, uint32_t lev, bool first, auto between) {
      constexpr int NP = decltype(np)::value;
      using TH = typename std::conditional<NP == 2, CtaPairs, CtaThreads>::type;
      uint32_t x[NP][E];
#pragma unroll
      for (int r = 0; r < NP; ++r)
#pragma unroll
        for (int e = 0; e < E; ++e)
          x[r][e] = lev + r < level ? biased_digit(w[e], a.base_log, lev + r) + dig_bias : p;
      ntt_forward<LOGN, E, NP, NP, P31>(x, tw, xb, tau, npr, TH());
#pragma unroll
      for (int r = 0; r < NP; ++r)
#pragma unroll
        for (int e = 0; e < E; ++e) x[r][e] = cond_sub(x[r][e], P31 ? p : npr.p8);
      mac<P31, NP>(oth, x, k, 1, first, p, p_inv);
      between();
      mac<P31, NP>(own, x, k, 0, first, p, p_inv);
    };
    // the partner's half is on its way while the own half is multiplied
    const auto send = [&] {
#ifdef ROSETTA_DEBUG
      if (a.lose_step == step + 1 && rank == 0) return;  // (rosetta_selftest_lost_words)
#endif
      const uint32_t to = part_to + odd * 2 * T * 16u, bar = part_bar_to + 16u * odd;
      dsmem_st_async_v4(to, oth[0], oth[1], oth[2], oth[3], bar);
      dsmem_st_async_v4(to + T * 16u, oth[4], oth[5], oth[6], oth[7], bar);
    };
    const auto nothing = [] {};
    using One = std::integral_constant<int, 1>;
    using Two = std::integral_constant<int, 2>;
    if constexpr (LEV == 1) {
      rows(key, One(), 0, true, send);
    } else if constexpr (LEV == 2) {
      rows(key, Two(), 0, true, send);
    } else if constexpr (LEV == 3) {
      RowKeys<1> last;
      last.load(key_own + step_off(i) + 2 * 2 * N, key_oth + step_off(i) + 2 * 2 * N, 2 * N, key_ok(i));
      rows(key, Two(), 0, true, nothing);
      rows(last, One(), 2, false, send);
    } else {
      for (uint32_t lev = 0; lev < level; lev += 2) {
        if (lev > 0)
          key.load(key_own + step_off(i) + lev * 2 * N, key_oth + step_off(i) + lev * 2 * N, 2 * N, key_ok(i),
                   level - lev);
        if (lev + 2 < level)
          rows(key, Two(), lev, lev == 0, nothing);
        else
          rows(key, Two(), lev, lev == 0, send);
      }
    }
    if (next < a.n) load_first(next);
    wait(part_bar, phase);
    const uint4 pa = part[odd * 2 * T + tau], pb = part[odd * 2 * T + T + tau];
    const uint32_t got[E] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
    uint32_t y[1][E];
#pragma unroll
    for (int e = 0; e < E; ++e)  // (28-bit primes: both below 4p)
      y[0][e] = P31 ? cond_sub(own[e], p) + cond_sub(got[e], p) : cond_sub(own[e] + got[e], 4 * p);
    // the exchange buffer changes from pairs to single words, whose warp-local
    // parts lie elsewhere: every forward read first
    if constexpr (LEV != 1) __syncthreads();
    ntt_inverse<LOGN, E, 1, 1, P31>(y, tw, xb, tau, npr, CtaThreads());  // CRT-scaled through the keys

    // ---- residues of the other primes, explicit CRT of component comp ----
#pragma unroll
    for (uint32_t k = 1; k < PRIMES; ++k) {
      const uint32_t to = (q + PRIMES - k) % PRIMES * 2 + comp;  // whose peer k - 1 this prime is
      const uint32_t dst = dsmem_map(res_s + ((odd * (PRIMES - 1) + k - 1) * 2 * T + tau) * 16u, to);
      const uint32_t bar = dsmem_map(res_bar, to);
      dsmem_st_async_v4(dst, y[0][0], y[0][1], y[0][2], y[0][3], bar);
      dsmem_st_async_v4(dst + T * 16u, y[0][4], y[0][5], y[0][6], y[0][7], bar);
    }
    wait(res_bar, phase);
    uint4 yo[PRIMES - 1][2];  // of primes q + 1, q + 2, ..
#pragma unroll
    for (int k = 0; k < PRIMES - 1; ++k) {
      yo[k][0] = res[(odd * (PRIMES - 1) + k) * 2 * T + tau];
      yo[k][1] = res[(odd * (PRIMES - 1) + k) * 2 * T + T + tau];
    }
    constexpr int QS = P31 ? 3 : 2;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      uint64_t s = acc[tau + e * T] + static_cast<uint64_t>(y[0][e]) * a.cc.pr[q].Mp_mod64;
      uint32_t ysum = y[0][e] >> QS;
#pragma unroll
      for (int k = 0; k < PRIMES - 1; ++k) {
        const uint32_t yv = word(yo[k][e / 4], e % 4);
        s += static_cast<uint64_t>(yv) * a.cc.pr[(q + 1 + k) % PRIMES].Mp_mod64;
        ysum += yv >> QS;
      }
      const uint32_t u = P31 ? crt_quotient31(ysum) : crt_quotient(ysum);
      acc[tau + e * T] = s - static_cast<uint64_t>(u) * a.cc.M_mod64;
    }
    i = next;
    ++step;
    __syncthreads();
  }
  const bool gave_up = *stop != 0u;  // in step - 1, the last that was run

  // the CTAs of a component all hold it: CTA (q, comp) writes its share
  const uint32_t j0 = N / PRIMES * q, j1 = q == PRIMES - 1 ? N : N / PRIMES * (q + 1);
  if (gave_up) {
    // the accumulator is not one of the ciphertext's
  } else if (a.glwe_out) {
    // ---- the rotated accumulator itself ----
    uint64_t *gout = a.glwe_out + (static_cast<size_t>(ct) * 2 + comp) * N;
    for (uint32_t j = j0 + tau; j < j1; j += T) gout[j] = acc[j];
  } else {
    // ---- sample extraction of the constant coefficient ----
    uint64_t *out = a.lwe_big_out + static_cast<size_t>(ct) * (N + 1);
    if (comp == 0)
      for (uint32_t j = j0 + tau; j < j1; j += T) out[j == 0 ? 0 : N - j] = j == 0 ? acc[j] : 0ull - acc[j];
    else if (q == 0 && tau == 0)
      out[N] = acc[0];
  }
  cluster.sync();  // no CTA leaves while a peer may still store into it
  if (gave_up && tau == 0) {
    // Every store has been issued by now and takes microseconds to arrive.  The next
    // step's mbarriers count the early words: they were armed before the loop was left,
    // or after the last step of all are armed here (their phase before, the last step's but
    // one, was complete when that step was run).
    const auto arrived = [&](uint32_t st, bool arm) {
      const uint32_t pb = bar0 + 16u * (st & 1u), ph = (st >> 1) & 1u;
      if (arm) {
        expect_tx(pb, N * 4u);
        expect_tx(pb + 8u, (PRIMES - 1) * N * 4u);
      }
      mbar_wait_cluster(pb, ph, wait_cycles / 64);
      mbar_wait_cluster(pb + 8u, ph, wait_cycles / 64);
    };
    arrived(step - 1, false);
    arrived(step, i >= a.n);
  }
}

template <int LOGN, int LEV, int PRIMES>
struct BrsKernel {
  static constexpr auto kernel = blind_rotate_small_kernel<LOGN, LEV, PRIMES>;

  // configuration of a launch of `batch` clusters (attr: room for one)
  static cudaError_t config(uint32_t n, uint32_t batch, cudaLaunchAttribute *attr, cudaLaunchConfig_t *cfg) {
    cudaError_t e = allow_dynamic_smem(kernel);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    *cfg = {};
    cfg->gridDim = dim3(2 * PRIMES * batch, 1, 1);
    cfg->blockDim = dim3(BrsShape<LOGN, LEV>::T, 1, 1);
    cfg->dynamicSmemBytes = brs_smem(size_t(1) << LOGN, LEV == 1, n, PRIMES);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2 * PRIMES;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
  }
};

// f(BrsKernel) of the kernel for a parameter set that br_small_supported accepts
template <typename F>
static cudaError_t with_brs_kernel(uint32_t logN, uint32_t level, uint32_t primes, F f) {
  if (!br_small_supported(logN, level, primes)) return cudaErrorInvalidValue;
  if (primes == kPrimes31) {
    switch (level) {
      case 1: return f(BrsKernel<12, 1, 3>());
      case 2: return f(BrsKernel<12, 2, 3>());
      default: return f(BrsKernel<12, 3, 3>());
    }
  }
  switch (logN) {
    case 8: return level == 1 ? f(BrsKernel<8, 1, 4>()) : level == 2 ? f(BrsKernel<8, 2, 4>()) : f(BrsKernel<8, 0, 4>());
    case 9: return level == 1 ? f(BrsKernel<9, 1, 4>()) : f(BrsKernel<9, 0, 4>());
    case 10: return level == 1 ? f(BrsKernel<10, 1, 4>()) : f(BrsKernel<10, 0, 4>());
    default: return level == 1 ? f(BrsKernel<11, 1, 4>()) : f(BrsKernel<11, 2, 4>());
  }
}

size_t br_small_smem_bytes(uint32_t logN, uint32_t level, uint32_t n, uint32_t primes) {
  return brs_smem(size_t(1) << logN, level == 1, n, primes);
}

// ---------------------------------------------------------------------------- the smallest ring
//
// N = 256 beyond a few dozen ciphertexts: the whole cluster's work in one CTA per
// ciphertext, a warp per prime and component, so that what the cluster sends through
// distributed shared memory goes through the CTA's own, and an SM holds two
// ciphertexts (16 warps) instead of clusters of one-warp CTAs that wait for each
// other.  The accumulator is there once; each warp does the CRT of a quarter of its
// component.  Three CTA barriers per step.  Bounded by the latency of a step (2.5 us)
// up to two ciphertexts per SM, by the integer multiplies and the barriers beyond.
// Measured with the key switch, n = 64, level 2, against the four-CTA cluster kernel:
// 152 ciphertexts 172 us (312), 304: 273 (527), 2000: 1.61 ms (1.97), 20000: 14.8 (18.4).
// One level is one row per component, transformed by itself (a pair with an empty row was
// 8 % behind the cluster kernel from 600 ciphertexts on): 152: 117 us (158 in pairs, 230 the
// cluster kernel), 608: 352 (494, 449), 2000: 1.15 ms (1.63, 1.49).
// Three CTAs per SM (85 registers): 1.64 / 14.98 ms; four (64, spilling): 1.68 / 15.15.  The
// same at N = 512 (two warps per group, six levels, n = 64): 600 us against 515 at 100
// ciphertexts, 7.98 ms against 7.14 at 2000: not built there.
struct BrtShape {
  static constexpr int LOGN = 8, N = 1 << LOGN, T = N / 8, GROUPS = 2 * kPrimes, THREADS = GROUPS * T;
  static constexpr int XB_WORDS = 2 * (N + N / 8);  // per group
};

// Shared memory: twiddles uint2 [4][N], acc uint64 [2][N], exchange buffers
// [8][2 (N + N/8)], partial products uint32 [8][N], residues uint32 [4][2][N],
// switched mask and body uint16 [n+1].
size_t br_tiny_smem_bytes(uint32_t n) {
  constexpr size_t N = BrtShape::N;
  return (kPrimes * N * sizeof(uint2) + 2 * N * sizeof(uint64_t) + 8 * 2 * (N + N / 8) * sizeof(uint32_t) +
          8 * N * sizeof(uint32_t) + 8 * N * sizeof(uint32_t) + (n + 1) * sizeof(uint16_t) + 15) & ~size_t(15);
}

template <int LEV>
__global__ void __launch_bounds__(BrtShape::THREADS, 2)
    blind_rotate_tiny_kernel(const __grid_constant__ BrArgs a) {
  using B = BrtShape;
  constexpr uint32_t LOGN = B::LOGN, N = B::N, T = B::T, TWO_N = 2 * N;
  constexpr int E = 8;
  const uint32_t group = __shfl_sync(0xffffffffu, threadIdx.x / T, 0);  // (warp-uniform for the compiler)
  const uint32_t tau = threadIdx.x % T, q = group / 2, comp = group % 2;
  const uint32_t ct = blockIdx.x;
  if (!dbg_ok(ct < a.batch, a.err_flag)) return;
  constexpr int NP = LEV == 1 ? 1 : 2;  // rows transformed together
  using Rows = typename std::conditional<NP == 2, GroupThreads, GroupSingles>::type;
  const GroupSingles singles{group + 1u, T};
  Rows row_threads;
  row_threads.id = group + 1u;
  row_threads.threads = T;

  extern __shared__ __align__(16) unsigned char smem[];
  uint2 *tw_s = reinterpret_cast<uint2 *>(smem);
  uint64_t *acc_all = reinterpret_cast<uint64_t *>(tw_s + kPrimes * N);
  uint64_t *acc = acc_all + comp * N;
  uint32_t *xb = reinterpret_cast<uint32_t *>(acc_all + 2 * N) + group * B::XB_WORDS;
  uint4 *part = reinterpret_cast<uint4 *>(reinterpret_cast<uint32_t *>(acc_all + 2 * N) + B::GROUPS * B::XB_WORDS);
  uint32_t *res = reinterpret_cast<uint32_t *>(part + B::GROUPS * 2 * T);
  uint16_t *atil = reinterpret_cast<uint16_t *>(res + 8 * N);

  const uint32_t p = a.cc.pr[q].p, p_inv = a.cc.pr[q].p_inv;
  const NttPrime npr(a.cc.pr[q]);
  const uint32_t level = LEV > 0 ? static_cast<uint32_t>(LEV) : a.level;

  for (uint32_t m = threadIdx.x; m < kPrimes * N; m += B::THREADS)
    tw_s[m / N * N + split_tw_slot<LOGN>(m % N)] = a.tw[m];
  const SplitTw<LOGN, 3> tw{tw_s + q * N, a.tw_lo[q]};
  const uint64_t *lwe = a.lwe_in + static_cast<size_t>((a.lwe_first + ct) % a.lwe_count) * (a.n + 1);
  constexpr uint32_t SH = 63 - LOGN;  // 64 - log2(2N)
  for (uint32_t i = threadIdx.x; i <= a.n; i += B::THREADS)
    atil[i] = static_cast<uint16_t>(((lwe[i] + (1ull << (SH - 1))) >> SH) & (TWO_N - 1));
  __syncthreads();
  {
    const uint32_t btil = atil[a.n];
    uint32_t li = 0;
    if (!a.glwe_in && a.lut_index) {
      li = a.lut_index[ct];
      if (li >= a.num_luts) {  // never read outside the LUT array
        if (threadIdx.x == 0 && a.err_flag) atomicExch(a.err_flag, 1u);
        li = 0;
      }
    }
    for (uint32_t m = threadIdx.x; m < 2 * N; m += B::THREADS) {
      const uint32_t c = m / N, j = m % N, e = (j + btil) & (TWO_N - 1), t = e & (N - 1);
      uint64_t v;
      if (a.glwe_in) {
        // encrypted test polynomial: ACC = X^{-b~} (A, B) for this ciphertext
        v = a.glwe_in[(static_cast<size_t>(ct) * 2 + c) * N + t];
      } else {
        // trivial GLWE (0, X^{-b~} v): (X^{2N - b~} v)[j] = +-v[t], t = (j + b~) mod 2N folded into [0, N)
        const uint64_t *lut = a.lut + (static_cast<size_t>(li) << a.msg_bits);
        const uint32_t box = N >> a.msg_bits, h = box >> 1;
        v = c == 0 ? 0ull : ((t < N - h) ? lut[(t + h) / box] : (0ull - lut[0]));
      }
      acc_all[m] = e >= N ? 0ull - v : v;
    }
  }
  __syncthreads();

  const uint64_t dig_add = dig_offset(a.base_log, level);
  const uint32_t dig_bias = p - (1u << (a.base_log - 1));
  const size_t kblk = static_cast<size_t>(2 * level) * 2 * N;  // words of one step's key block per prime
  const uint32_t *key_own = a.bsk + q * kblk + (static_cast<size_t>(comp) * level * 2 + comp) * N + E * tau;
  const uint32_t *key_oth = a.bsk + q * kblk + (static_cast<size_t>(comp) * level * 2 + (comp ^ 1u)) * N + E * tau;
  const auto step_off = [&](uint32_t i) { return static_cast<size_t>(i) * kPrimes * kblk; };
  const auto key_ok = [&](uint32_t i) {
    return dbg_ok(a.bsk_words == 0 || (static_cast<size_t>(i) * kPrimes + q + 1) * kblk <= a.bsk_words, a.err_flag);
  };
  RowKeys<NP> key;  // of the first rows of the coming step
  const auto load_first = [&](uint32_t i) {
    key.load(key_own + step_off(i), key_oth + step_off(i), 2 * N, key_ok(i), level);
  };
  const auto next_step = [&](uint32_t i) {
    while (i < a.n && atil[i] == 0) ++i;
    return i;
  };
  uint32_t i = next_step(0);
  if (i < a.n) load_first(i);
#pragma unroll 1
  while (i < a.n) {
    const uint32_t at = atil[i];
    // ---- rotated difference of component comp, digit offsets added ----
    uint64_t w[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t j = tau + e * T, t = (j + TWO_N - at) & (TWO_N - 1);
      const uint64_t v = acc[t & (N - 1)];
      w[e] = (t >= N ? 0ull - v : v) - acc[j] + dig_add;
    }
    const uint32_t next = next_step(i + 1);

    // ---- forward transforms, products with both components of the key ----
    uint32_t own[E], oth[E];
#pragma unroll
    for (uint32_t lev = 0; lev < level; lev += NP) {
      if (lev > 0)
        key.load(key_own + step_off(i) + lev * 2 * N, key_oth + step_off(i) + lev * 2 * N, 2 * N, key_ok(i),
                 level - lev);
      uint32_t x[NP][E];
#pragma unroll
      for (int r = 0; r < NP; ++r)
#pragma unroll
        for (int e = 0; e < E; ++e)
          x[r][e] = lev + r < level ? biased_digit(w[e], a.base_log, lev + r) + dig_bias : p;
      ntt_forward<LOGN, E, NP, NP>(x, tw, xb, tau, npr, row_threads);
#pragma unroll
      for (int r = 0; r < NP; ++r)
#pragma unroll
        for (int e = 0; e < E; ++e) x[r][e] = cond_sub(x[r][e], npr.p8);
      mac<false, NP>(oth, x, key, 1, lev == 0, p, p_inv);
      mac<false, NP>(own, x, key, 0, lev == 0, p, p_inv);
    }
    if (next < a.n) load_first(next);
    part[(group ^ 1u) * 2 * T + tau] = make_uint4(oth[0], oth[1], oth[2], oth[3]);
    part[(group ^ 1u) * 2 * T + T + tau] = make_uint4(oth[4], oth[5], oth[6], oth[7]);
    __syncthreads();  // partial products there (and the exchange buffer free to change layout)
    const uint4 pa = part[group * 2 * T + tau], pb = part[group * 2 * T + T + tau];
    const uint32_t got[E] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
    uint32_t y[1][E];
#pragma unroll
    for (int e = 0; e < E; ++e) y[0][e] = cond_sub(own[e] + got[e], 4 * p);  // both below 4p
    ntt_inverse<LOGN, E, 1, 1>(y, tw, xb, tau, npr, singles);  // CRT-scaled through the keys

    // ---- explicit CRT: group (q, comp) takes slots 2q and 2q + 1 of its component ----
#pragma unroll
    for (int e = 0; e < E; ++e) res[(q * 2 + comp) * N + e * T + tau] = y[0][e];
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t j = (2 * q + h) * T + tau;
      uint64_t s = acc[j];
      uint32_t ysum = 0;
#pragma unroll
      for (int k = 0; k < kPrimes; ++k) {
        const uint32_t yv = res[(k * 2 + comp) * N + j];
        s += static_cast<uint64_t>(yv) * a.cc.pr[k].Mp_mod64;
        ysum += yv >> 2;
      }
      acc[j] = s - static_cast<uint64_t>(crt_quotient(ysum)) * a.cc.M_mod64;
    }
    i = next;
    __syncthreads();
  }

  if (a.glwe_out) {
    // ---- the rotated accumulator itself ----
    uint64_t *gout = a.glwe_out + static_cast<size_t>(ct) * 2 * N;
    for (uint32_t m = threadIdx.x; m < 2 * N; m += B::THREADS) gout[m] = acc_all[m];
  } else {
    // ---- sample extraction of the constant coefficient ----
    uint64_t *out = a.lwe_big_out + static_cast<size_t>(ct) * (N + 1);
    for (uint32_t j = threadIdx.x; j < N; j += B::THREADS) out[j == 0 ? 0 : N - j] = j == 0 ? acc_all[j] : 0ull - acc_all[j];
    if (threadIdx.x == 0) out[N] = acc_all[N];
  }
}

template <int LEV>
static cudaError_t launch_brt_t(const BrArgs &a, cudaStream_t s) {
  auto kern = blind_rotate_tiny_kernel<LEV>;
  const size_t smem = br_tiny_smem_bytes(a.n);
  cudaError_t e = allow_dynamic_smem(kern);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  kern<<<a.batch, BrtShape::THREADS, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_blind_rotate_tiny(const BrArgs &a, cudaStream_t s) {
  return a.level == 1 ? launch_brt_t<1>(a, s) : a.level == 2 ? launch_brt_t<2>(a, s) : launch_brt_t<0>(a, s);
}

bool br_small_supported(uint32_t logN, uint32_t level, uint32_t primes) {
  if (primes == kPrimes31) return logN == 12 && level >= 1 && level <= 3;
  return logN >= 8 && (logN <= 10 || (logN == 11 && level >= 1 && level <= 2));
}

cudaError_t launch_blind_rotate_small(const BrArgs &a, uint32_t logN, cudaStream_t s) {
  return with_brs_kernel(logN, a.level, a.primes, [&](auto k) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    const cudaError_t e = k.config(a.n, a.batch, attr, &cfg);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, k.kernel, a) : e;
  });
}

uint32_t br_small_resident(uint32_t logN, uint32_t level, uint32_t n, uint32_t primes) {
  int clusters = 0;
  const cudaError_t st = with_brs_kernel(logN, level, primes, [&](auto k) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg;
    const cudaError_t e = k.config(n, 1, attr, &cfg);
    return e == cudaSuccess ? cudaOccupancyMaxActiveClusters(&clusters, k.kernel, &cfg) : e;
  });
  if (st != cudaSuccess) cudaGetLastError();
  return st == cudaSuccess && clusters > 0 ? static_cast<uint32_t>(clusters) : 0;
}

}  // namespace rosetta
