// LWE key switch on the tensor cores in 8-bit floating point (tcgen05
// kind::f8f6f4, accumulators in tensor memory), for key-switch bases up to 2^5.
//
//   out[b][j] = [j = n] b'_b - sum_r d[b][r] KSK[r][j]      (mod 2^64)
// over r = (lev, i).  The digits (|d| <= 2^(beta-1) <= 16) and the key words cut
// into 13 signed limbs of 5 bits (-16 .. 15, the top one 0 .. 15) are integers
// that e4m3 holds exactly; every product is at most 256 and, as checked on the
// host, every sum stays below 2^24, so the fp32 accumulators hold the exact
// integers C_t[b][j] = sum_r d[b][r] L_t[r][j], and
//   sum_r d KSK = sum_t C_t 2^(5 t)   (mod 2^64)
// is recombined in the epilogue.  Same words as keyswitch_kernel.
//
// Measured: n = 742, N = 2048, base 2^3 x 5, 4096 ciphertexts: 668 us with the
// bf16 kernel, 262 here (the tensor floor is 208); n = 840, N = 4096, base 2^4 x 5,
// 61 ciphertexts: 355 us with the CUDA-core kernel, 47 here (225 MB of limbs: 33).
// So it takes every batch.  The main kernel starts while the digits are cut
// (programmatic launch) and fetches its first key tiles meanwhile: 271 and 51 us without.
//
// Against the bf16 kernel (keyswitch_tc.cu: 8 limbs of 8 bits, or 16 of 4 bits
// for long sums, at half the rate and two bytes each) a key word takes 13 bytes
// instead of 16 or 32 and 0.81 or 0.41 of the tensor time.
//
// Operands lie in global memory cut into the tiles one pipeline stage takes, in
// the no-swizzle K-major layout of the tensor cores (core matrices of 8 rows x
// 16 bytes; K-adjacent ones 128 B apart, 8-row groups 1024 B apart; 128 K
// elements a stage), so each comes in with one bulk copy.  Column t 16 + jj of
// a key tile is limb t of its output word jj: the epilogue reads one limb of 16
// words at a time.  K runs level-major, r = (lev-1) kN + i.
//
// Per CTA: MT x 128 ciphertexts x 16 output words (208 limb columns), one
// thread issuing the copies, one the MMAs (M = 128, N = 208, K = 32), four
// warps the epilogue.  With two row tiles (MT = 2) a key tile is read once for
// 256 ciphertexts: the loop is bound by the operands' way from L2 (about 10
// TB/s), not by the tensor cores.  Where the tiles alone do not fill the GPU the
// K range is split over several CTAs, whose sums meet in 64-bit atomic adds
// (exact and order-independent mod 2^64) on a zeroed output.  Rows past the
// batch are neither copied nor written: their accumulators are garbage of their
// own lanes.
//
// Every wait on an mbarrier gives up after about two seconds and sets the error
// flag; the CTA then skips its epilogue, waits (again bounded) for the copies
// it issued, and frees the tensor memory only when nothing it issued can still
// be in flight.
#include <stdint.h>

#include "dsmem.cuh"
#include "internal.h"
#include "tcgen.cuh"

namespace rosetta {

namespace {

constexpr uint32_t F8_M = 128, F8_K = 128, F8_LIMBS = 13, F8_WORDS = 16, F8_N = F8_LIMBS * F8_WORDS;
constexpr uint32_t F8_A_TILE = F8_M * F8_K, F8_B_TILE = F8_N * F8_K;  // bytes
constexpr uint32_t F8_LBITS = 5;
constexpr uint32_t F8_THREADS = 192;  // four epilogue warps, the copy warp, the MMA warp

// Byte offset of (row, k) inside a tile.
__host__ __device__ constexpr uint32_t f8_off(uint32_t row, uint32_t k) {
  return ((row >> 3) * (F8_K / 16) + (k >> 4)) * 128 + (row & 7u) * 16 + (k & 15u);
}

// four integers |v| <= 16 as e4m3 bytes, v0 lowest
__device__ __forceinline__ uint32_t e4m3x4(int v0, int v1, int v2, int v3) {
  uint16_t lo, hi;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(static_cast<float>(v1)), "f"(static_cast<float>(v0)));
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(static_cast<float>(v3)), "f"(static_cast<float>(v2)));
  return static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
}

// Instruction descriptor, kind::f8f6f4: D f32, A and B e4m3, both K-major.
constexpr uint32_t kIdescF8 = (1u << 4) | ((F8_N >> 3) << 17) | ((F8_M >> 4) << 24);

__device__ __forceinline__ void mma_f8(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(adesc), "l"(bdesc), "r"(kIdescF8), "r"(accumulate)
      : "memory");
}

// 16 consecutive fp32 columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The digits (and the zeroed output) of the kernel before this one are complete.
__device__ __forceinline__ void digits_ready() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <int MT>
struct F8Shape {
  static constexpr uint32_t STAGE = MT * F8_A_TILE + F8_B_TILE;
  static constexpr uint32_t STAGES = MT == 2 ? 3 : 5;
  static constexpr uint32_t TMEM_COLS = MT == 2 ? 512 : 256;  // a power of two; MT x 208 used
};

}  // namespace

// Digit tiles: A[b][r] = digit lev of a'_i (closed form, see biased_digit),
// all levels of 128 mask words x 32 ciphertexts per CTA: a word is read once.  A
// warp writes whole core matrices (8 rows x 16 bytes, 128 contiguous bytes).
// Also zeroes `zero_words` words of the output.  The grid has one dimension, kN / 128
// CTAs (at most 64) per 32 ciphertexts: its limit of 2^31 - 1 lies beyond any batch
// that fits the memory, that of a second dimension (65535) does not.
__global__ void __launch_bounds__(256) ks8_digits_kernel(const uint64_t *__restrict__ big, uint8_t *__restrict__ a_tiles,
                                                         uint32_t batch, uint32_t kN, uint32_t base_log, uint32_t level,
                                                         uint32_t k_steps, uint64_t offset, uint64_t *__restrict__ zero,
                                                         size_t zero_words) {
  // ks8_kernel may start: it sets itself up and fetches key tiles until these digits are complete
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // (the output, when K is split: the sums are added into it)
  const size_t gid = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (size_t w = gid; w < zero_words; w += static_cast<size_t>(gridDim.x) * blockDim.x) zero[w] = 0;
  const uint32_t k_blocks = kN / F8_K, group = blockIdx.x / k_blocks;
  const uint32_t i0 = (blockIdx.x - group * k_blocks) * F8_K, g0 = group * 4;  // first mask word, group of 8 ciphertexts
  const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t r = lane >> 2, q = lane & 3u;  // row of the group, four of the core matrix's 16 words
  const int half = 1 << (base_log - 1);
  const uint32_t mask = (1u << base_log) - 1u;
  for (uint32_t item = warp; item < 4 * (F8_K / 16); item += 8) {
    const uint32_t rg = g0 + item / (F8_K / 16), kg = item % (F8_K / 16);
    if (rg * 8 >= batch) continue;  // (the same for the whole warp)
    const uint32_t b = rg * 8 + r;
    uint64_t w[4] = {0, 0, 0, 0};
    if (b < batch) {
      const uint64_t *src = big + static_cast<size_t>(b) * (kN + 1) + i0 + kg * 16 + q * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = src[e] + offset;
    }
    for (uint32_t lev = 0; lev < level; ++lev) {
      const uint32_t sh = 64 - (lev + 1) * base_log;
      int d[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) d[e] = static_cast<int>(static_cast<uint32_t>(w[e] >> sh) & mask) - half;
      const uint32_t ks = (lev * kN + i0) / F8_K;
      uint8_t *tile = a_tiles + (static_cast<size_t>(rg >> 4) * k_steps + ks) * F8_A_TILE;
      *reinterpret_cast<uint32_t *>(tile + f8_off((rg & 15u) * 8 + r, kg * 16 + q * 4)) = e4m3x4(d[0], d[1], d[2], d[3]);
    }
  }
}

// Limb tiles of the key, once per key: column t 16 + jj of tile nt is limb t of
// word nt 16 + jj (zero past word n).  Grid: k_steps x n_tiles.
__global__ void __launch_bounds__(256) ks8_limbs_kernel(const uint64_t *__restrict__ ksk, uint8_t *__restrict__ b_tiles,
                                                        uint32_t kN, uint32_t level, uint32_t n, uint32_t k_steps) {
  const uint32_t ks = blockIdx.x, nt = blockIdx.y;
  const uint32_t lev = ks * F8_K / kN, i0 = ks * F8_K % kN;
  uint64_t offset = 0;  // 16 at every limb but the top one
#pragma unroll
  for (uint32_t t = 0; t + 1 < F8_LIMBS; ++t) offset |= 16ull << (F8_LBITS * t);
  uint8_t *tile = b_tiles + (static_cast<size_t>(nt) * k_steps + ks) * F8_B_TILE;
  for (uint32_t item = threadIdx.x; item < F8_WORDS * (F8_K / 4); item += blockDim.x) {
    const uint32_t jj = item % F8_WORDS, kq = item / F8_WORDS, j = nt * F8_WORDS + jj;
    uint64_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      w[e] = j <= n ? ksk[(static_cast<size_t>(i0 + kq * 4 + e) * level + lev) * (n + 1) + j] + offset : offset;
#pragma unroll
    for (uint32_t t = 0; t < F8_LIMBS; ++t) {
      const int bias = t + 1 < F8_LIMBS ? 16 : 0;
      int d[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) d[e] = static_cast<int>((w[e] >> (F8_LBITS * t)) & 31u) - bias;
      *reinterpret_cast<uint32_t *>(tile + f8_off(t * F8_WORDS + jj, kq * 4)) = e4m3x4(d[0], d[1], d[2], d[3]);
    }
  }
}

template <int MT>
__global__ void __launch_bounds__(F8_THREADS, 1) ks8_kernel(const KsTcArgs a) {
  using S = F8Shape<MT>;
  constexpr uint32_t STAGES = S::STAGES;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 1];  // full[s], empty[s], done
  __shared__ uint32_t tmem_slot;
  // s_fail: a wait gave up, the accumulators are partial; s_unsafe: copies or
  // MMAs this CTA issued may still be in flight; stages issued and consumed
  __shared__ uint32_t s_fail, s_unsafe, s_issued, s_consumed;
  const uint32_t mt = blockIdx.x, nt = blockIdx.y;
  const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t base = smem_addr(smem), bar0 = smem_addr(bars);
  auto full = [&](uint32_t s) { return bar0 + 8u * s; };
  auto empty = [&](uint32_t s) { return bar0 + 8u * (STAGES + s); };
  const uint32_t done = bar0 + 8u * (2 * STAGES);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_slot)),
                 "r"(S::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    s_fail = s_unsafe = s_issued = s_consumed = 0u;
    for (uint32_t s = 0; s < 2 * STAGES + 1; ++s) mbar_init(bar0 + 8u * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  // this CTA's K range and rows
  const uint32_t per = (a.k_steps + gridDim.z - 1) / gridDim.z;
  const uint32_t k0 = blockIdx.z * per, steps = min(a.k_steps, k0 + per) - k0;
  const uint32_t row0 = mt * MT * F8_M;
  uint32_t a_bytes[MT];  // of a stage's row tiles: the groups of eight rows that exist
#pragma unroll
  for (int m = 0; m < MT; ++m) {
    const uint32_t first = row0 + m * F8_M;
    const uint32_t rows = first < a.batch ? min(F8_M, a.batch - first) : 0u;
    a_bytes[m] = (rows + 7) / 8 * (8 * F8_K);
  }
  const uint8_t *a8 = reinterpret_cast<const uint8_t *>(a.a_tiles);
  const uint8_t *b8 = reinterpret_cast<const uint8_t *>(a.b_tiles);

  if (warp == 4 && lane == 0) {
    // ---- copies ----
    uint32_t stage_bytes = F8_B_TILE, k = 0;
#pragma unroll
    for (int m = 0; m < MT; ++m) stage_bytes += a_bytes[m];
    const auto load_key = [&](uint32_t k) {
      const uint32_t slot = k % STAGES;
      expect_tx(full(slot), stage_bytes);
      bulk_load(base + slot * S::STAGE + MT * F8_A_TILE, b8 + (static_cast<size_t>(nt) * a.k_steps + k0 + k) * F8_B_TILE,
                F8_B_TILE, full(slot));
    };
    // the first stages' key tiles do not depend on the digits kernel
    const uint32_t early = min(steps, STAGES);
    for (uint32_t e = 0; e < early; ++e) load_key(e);
    digits_ready();
    for (; k < steps; ++k) {
      const uint32_t slot = k % STAGES;
      if (k >= STAGES) {
        if (!mbar_wait(empty(slot), (k / STAGES - 1) & 1u)) break;  // the MMAs reading the slot are done
        load_key(k);
      }
#pragma unroll
      for (int m = 0; m < MT; ++m)
        if (a_bytes[m])
          bulk_load(base + slot * S::STAGE + m * F8_A_TILE,
                    a8 + (static_cast<size_t>(mt * MT + m) * a.k_steps + k0 + k) * F8_A_TILE, a_bytes[m], full(slot));
    }
    s_issued = k;
    if (k < steps) {
      atomicExch(a.err_flag, 2u);
      s_fail = 1u;
    }
  } else if (warp == 5 && lane == 0) {
    // ---- MMAs ----
    uint32_t k = 0;
    for (; k < steps; ++k) {
      const uint32_t slot = k % STAGES;
      if (!mbar_wait(full(slot), (k / STAGES) & 1u)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sa = base + slot * S::STAGE, sb = sa + MT * F8_A_TILE;
#pragma unroll
      for (uint32_t kk = 0; kk < F8_K / 32; ++kk)  // K = 32 per MMA: two core matrices, 256 B
#pragma unroll
        for (int m = 0; m < MT; ++m)
          if (MT == 1 || a_bytes[m])
            mma_f8(tmem + m * F8_N, smem_desc(sa + m * F8_A_TILE + kk * 256u), smem_desc(sb + kk * 256u), (k | kk) != 0);
      mma_commit(empty(slot));
    }
    s_consumed = k;
    if (k < steps) {
      atomicExch(a.err_flag, 2u);
      s_fail = 1u;
    }
    mma_commit(done);
  }
  __syncwarp();
  const bool fin = __all_sync(0xffffffffu, mbar_wait(done, 0));  // warp-uniform for tcgen05.ld
  if (!fin && lane == 0) {
    atomicExch(a.err_flag, 2u);
    s_unsafe = 1u;  // the MMAs may still be writing tensor memory
  }
  __syncthreads();
  const bool partial = s_fail != 0u;
  if (partial && threadIdx.x == 0) {
    // let the copies already issued land before the shared memory is released
    bool drained = true;
    for (uint32_t k = s_consumed; k < s_issued; ++k)
      drained = mbar_wait(full(k % STAGES), (k / STAGES) & 1u) && drained;
    if (!drained) s_unsafe = 1u;
  }
  __syncthreads();
  const bool unsafe = s_unsafe != 0u;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (!unsafe && !partial && warp < 4) {
    digits_ready();  // (long since; orders the output's zeros before the additions below)
    // epilogue: lane = ciphertext row of this warp's quarter of tensor memory
    const uint32_t n1 = a.n + 1, j0 = nt * F8_WORDS;
#pragma unroll 1
    for (int m = 0; m < MT; ++m) {
      const uint32_t b = row0 + m * F8_M + warp * 32 + lane;
      if (!__any_sync(0xffffffffu, b < a.batch)) continue;
      uint64_t s[F8_WORDS];
#pragma unroll
      for (uint32_t t = 0; t < F8_LIMBS; ++t) {
        uint32_t v[16];
        tmem_ld16(tmem + ((warp * 32u) << 16) + m * F8_N + t * F8_WORDS, v);
#pragma unroll
        for (uint32_t jj = 0; jj < F8_WORDS; ++jj) {
          const int64_t c = __float2int_rn(__uint_as_float(v[jj]));
          s[jj] = (t == 0 ? 0ull : s[jj]) + (static_cast<uint64_t>(c) << (F8_LBITS * t));
        }
      }
      if (b < a.batch) {
        const bool whole = gridDim.z == 1;
        const uint64_t body =
            blockIdx.z == 0 && j0 + F8_WORDS > a.n ? a.big[static_cast<size_t>(b) * (a.kN + 1) + a.kN] : 0ull;
        uint64_t *out = a.out + static_cast<size_t>(b) * n1 + j0;
#pragma unroll
        for (uint32_t jj = 0; jj < F8_WORDS; ++jj) {
          if (j0 + jj >= n1) continue;
          const uint64_t v = (j0 + jj == a.n ? body : 0ull) - s[jj];
          if (whole)
            out[jj] = v;
          else
            atomicAdd(reinterpret_cast<unsigned long long *>(out + jj), static_cast<unsigned long long>(v));
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // After a wait that gave up with work still in flight nothing is safe: the
  // tensor memory is left allocated rather than handed to another CTA while
  // an MMA may still write it, the outputs are not written, and the error
  // flag reports TIMEOUT.  The CUDA context must then be destroyed.
  if (warp == 0 && !unsafe)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::TMEM_COLS) : "memory");
}

// ---------------------------------------------------------------------------- host side

bool ks8_exact(uint32_t kN, uint32_t level, uint32_t base_log) {
  if (base_log > 5 || kN % F8_K != 0) return false;
  return static_cast<double>(1u << (base_log - 1)) * 16.0 * kN * level < 16777216.0;
}

size_t ks8_b_bytes(uint32_t kN, uint32_t level, uint32_t n) {
  return static_cast<size_t>((n + F8_WORDS) / F8_WORDS) * (static_cast<size_t>(kN) * level / F8_K) * F8_B_TILE;
}

size_t ks8_a_bytes(uint32_t batch, uint32_t kN, uint32_t level) {
  return static_cast<size_t>((batch + F8_M - 1) / F8_M) * (static_cast<size_t>(kN) * level / F8_K) * F8_A_TILE;
}

cudaError_t launch_ks8_limbs(const uint64_t *ksk, uint8_t *b_tiles, uint32_t kN, uint32_t level, uint32_t n,
                             cudaStream_t s) {
  const uint32_t k_steps = kN * level / F8_K;
  ks8_limbs_kernel<<<dim3(k_steps, (n + F8_WORDS) / F8_WORDS), 256, 0, s>>>(ksk, b_tiles, kN, level, n, k_steps);
  return cudaGetLastError();
}

template <int MT>
static cudaError_t launch_ks8_t(const KsTcArgs &a, dim3 grid, cudaStream_t s) {
  const int smem = static_cast<int>(F8Shape<MT>::STAGES * F8Shape<MT>::STAGE);
  cudaError_t e = cudaFuncSetAttribute(ks8_kernel<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(F8_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ks8_kernel<MT>, a);
}

cudaError_t launch_keyswitch_fp8(const KsTcArgs &a, uint32_t base_log, uint32_t level, uint32_t sms, cudaStream_t s) {
  uint64_t offset = level * base_log >= 64 ? 0 : 1ull << (63 - level * base_log);
  for (uint32_t m = 1; m <= level; ++m) offset += 1ull << (64 - m * base_log + base_log - 1);
  const uint32_t mt = a.batch > F8_M ? 2 : 1;
  const uint32_t m_blocks = (a.batch + mt * F8_M - 1) / (mt * F8_M), n_tiles = (a.n + F8_WORDS) / F8_WORDS;
  // K splits: the fewest rounds of the GPU per unit of work; a split costs each
  // CTA its fill and epilogue, about 8 stages
  const uint32_t tiles = m_blocks * n_tiles;
  uint32_t splits = 1;
  double best = 1e30;
  for (uint32_t z = 1; z <= 16 && z <= a.k_steps; ++z) {
    const uint32_t per = (a.k_steps + z - 1) / z;
    if ((a.k_steps + per - 1) / per != z) continue;  // no empty splits
    const double cost = static_cast<double>((static_cast<uint64_t>(tiles) * z + sms - 1) / sms) * (per + 8);
    if (cost < best) {
      best = cost;
      splits = z;
    }
  }
  const uint64_t digit_ctas = static_cast<uint64_t>((a.batch + 31ull) / 32) * (a.kN / F8_K);
  if (digit_ctas > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
  ks8_digits_kernel<<<static_cast<uint32_t>(digit_ctas), 256, 0, s>>>(
      a.big, reinterpret_cast<uint8_t *>(const_cast<uint16_t *>(a.a_tiles)), a.batch, a.kN, base_log, level, a.k_steps,
      offset, a.out, splits > 1 ? static_cast<size_t>(a.batch) * (a.n + 1) : 0);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const dim3 grid(m_blocks, n_tiles, splits);
  return mt == 2 ? launch_ks8_t<2>(a, grid, s) : launch_ks8_t<1>(a, grid, s);
}

}  // namespace rosetta
