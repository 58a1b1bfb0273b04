// Single-precision complex transforms that estimate an external product's
// size: the worker-per-ciphertext kernels (blind_rotate_solo.cu, trace_solo.cu) run
// them in place of a fourth prime's number-theoretic transforms.
//
// A real polynomial a(X) of N coefficients, multiplied modulo X^N + 1, is
// carried as the complex polynomial sum_j (a_j + i a_{j+C}) X^j modulo
// X^C - i, C = N / 2 (X^N + 1 = (X^C - i)(X^C + i); the other factor holds
// the conjugates).  The decimation tree is that of the integer transforms:
// X^len - w^2 splits into X^{len/2} -+ w, natural-order input, bit-reversed
// output, the inverse the other way round without its 1/C.  The two children
// of a node use the twiddles w2 and i w2, so a pass of two stages needs two
// twiddles per thread, w1 and w2, held together in one 16-byte table entry.
//
// 4 complex values of 2 polynomials per thread, T = C / 4 threads.
//
// Rounding, u = 2^-24, |twiddle error| <= u / sqrt 2.  Forward butterfly
// (X' = X + w Y by two fused multiply-adds per component, Y' = 2 X - X' by one):
// 3.9 u of the vector's 2-norm per stage.  Inverse butterfly (X + Y, then
// (X - Y) conj(w) by a product and a fused multiply-add): each summand of an
// output picks up a factor within 1 +- 3.8 u per stage.  Keys are rounded once
// (1 u); a sum of 2 l products adds (4 l + 2) u.  By Cauchy-Schwarz a
// coefficient of the product is off by less than
//   (3.9 log2 C + 1 + (4 l + 2) + 3.8 log2 C) u sum_r |d_r| |g_r|,
// below kCfftErr = 100 u times (k+1) l N 2^(beta-1) 2^63 for C <= 1024 and l <= 3 (the
// trace's sums of four products are those of l = 2); the product of three stages'
// second-order terms is far below the slack.
#pragma once
#include <stdint.h>

#include "ntt.cuh"

namespace rosetta {

// entries of the pass twiddle table: 4^0 + 4^1 + ... over the log2(C)/2 passes
__host__ __device__ constexpr uint32_t cfft_tw_offset(int pass) { return ((1u << (2 * pass)) - 1u) / 3u; }

__device__ __forceinline__ void cfft_fwd_bfly(uint32_t &xr, uint32_t &xi, uint32_t &yr, uint32_t &yi, float wr,
                                              float wi) {
  const float Xr = __uint_as_float(xr), Xi = __uint_as_float(xi), Yr = __uint_as_float(yr), Yi = __uint_as_float(yi);
  const float ar = fmaf(-wi, Yi, fmaf(wr, Yr, Xr));
  const float ai = fmaf(wi, Yr, fmaf(wr, Yi, Xi));
  xr = __float_as_uint(ar);
  xi = __float_as_uint(ai);
  yr = __float_as_uint(fmaf(2.0f, Xr, -ar));
  yi = __float_as_uint(fmaf(2.0f, Xi, -ai));
}

__device__ __forceinline__ void cfft_inv_bfly(uint32_t &xr, uint32_t &xi, uint32_t &yr, uint32_t &yi, float wr,
                                              float wi) {
  const float Xr = __uint_as_float(xr), Xi = __uint_as_float(xi), Yr = __uint_as_float(yr), Yi = __uint_as_float(yi);
  const float dr = Xr - Yr, di = Xi - Yi;
  xr = __float_as_uint(Xr + Yr);
  xi = __float_as_uint(Xi + Yi);
  yr = __float_as_uint(fmaf(di, wi, dr * wr));
  yi = __float_as_uint(fmaf(-dr, wi, di * wr));
}

// Exchange-buffer slot (16 bytes: both parts of both polynomials) of element
// i: bits 0, 1 and 2 are flipped by bits 3, 4 and 4, which keeps every pass free
// of bank conflicts (the eight threads of a quarter-warp differ in bits 0-2; 0, 1
// and 4; 2-4).
__host__ __device__ constexpr uint32_t cfft_swz(uint32_t i) { return i ^ ((i >> 3) & 3u) ^ ((i >> 2) & 4u); }

// Slot e of a thread in the pass at stage S0 is cfft_base ^ cfft_swz(e SIG).
template <int LOGC, int S0>
__device__ __forceinline__ uint32_t cfft_base(uint32_t tau) {
  constexpr uint32_t C = 1u << LOGC, SIG = C >> (S0 + 2);
  return cfft_swz((tau / SIG) * 4 * SIG + tau % SIG);
}

template <int LOGC, int S0>
__device__ __forceinline__ void cfft_store(uint4 *xb, const uint32_t (&x)[4][4], uint32_t tau) {
  constexpr uint32_t SIG = (1u << LOGC) >> (S0 + 2);
  const uint32_t b = cfft_base<LOGC, S0>(tau);
#pragma unroll
  for (int e = 0; e < 4; ++e) xb[b ^ cfft_swz(e * SIG)] = make_uint4(x[0][e], x[1][e], x[2][e], x[3][e]);
}

template <int LOGC, int S0>
__device__ __forceinline__ void cfft_load(const uint4 *xb, uint32_t (&x)[4][4], uint32_t tau) {
  constexpr uint32_t SIG = (1u << LOGC) >> (S0 + 2);
  const uint32_t b = cfft_base<LOGC, S0>(tau);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint4 v = xb[b ^ cfft_swz(e * SIG)];
    x[0][e] = v.x;
    x[1][e] = v.y;
    x[2][e] = v.z;
    x[3][e] = v.w;
  }
}

// From the layout of the pass at stage SA to that of the pass at SB.
template <int LOGC, int SA, int SB, class TH>
__device__ __forceinline__ void cfft_exchange(uint32_t (&x)[4][4], uint32_t *xb_words, uint32_t tau, const TH &th) {
  uint4 *xb = reinterpret_cast<uint4 *>(xb_words);
  constexpr int G = pass_group_warps<LOGC, 4, (SA < SB ? SA : SB)>();
  constexpr int WARPS = (1 << LOGC) / 128;
  group_sync<G, WARPS>(tau, th);
  cfft_store<LOGC, SA>(xb, x, tau);
  group_sync<G, WARPS>(tau, th);
  cfft_load<LOGC, SB>(xb, x, tau);
}

// x[2 k][e], x[2 k + 1][e]: real and imaginary part (float bits) of slot e of
// polynomial k.  xb: 4 C words.
template <int LOGC, int PASS = 0, class TH>
__device__ __forceinline__ void cfft_forward(uint32_t (&x)[4][4], const float4 *tw, uint32_t *xb, uint32_t tau,
                                             const TH &th) {
  static_assert(LOGC % 2 == 0, "whole passes of two stages");
  constexpr int S0 = 2 * PASS;
  constexpr uint32_t SIG = (1u << LOGC) >> (S0 + 2);
  const float4 w = tw[cfft_tw_offset(PASS) + tau / SIG];
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    cfft_fwd_bfly(x[k][0], x[k + 1][0], x[k][2], x[k + 1][2], w.x, w.y);
    cfft_fwd_bfly(x[k][1], x[k + 1][1], x[k][3], x[k + 1][3], w.x, w.y);
    cfft_fwd_bfly(x[k][0], x[k + 1][0], x[k][1], x[k + 1][1], w.z, w.w);
    cfft_fwd_bfly(x[k][2], x[k + 1][2], x[k][3], x[k + 1][3], -w.w, w.z);  // i w2
  }
  if constexpr (S0 + 2 < LOGC) {
    cfft_exchange<LOGC, S0, S0 + 2>(x, xb, tau, th);
    cfft_forward<LOGC, PASS + 1>(x, tw, xb, tau, th);
  }
}

template <int LOGC, int PASS = LOGC / 2 - 1, class TH>
__device__ __forceinline__ void cfft_inverse(uint32_t (&x)[4][4], const float4 *tw, uint32_t *xb, uint32_t tau,
                                             const TH &th) {
  constexpr int S0 = 2 * PASS;
  constexpr uint32_t SIG = (1u << LOGC) >> (S0 + 2);
  const float4 w = tw[cfft_tw_offset(PASS) + tau / SIG];
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    cfft_inv_bfly(x[k][0], x[k + 1][0], x[k][1], x[k + 1][1], w.z, w.w);
    cfft_inv_bfly(x[k][2], x[k + 1][2], x[k][3], x[k + 1][3], -w.w, w.z);
    cfft_inv_bfly(x[k][0], x[k + 1][0], x[k][2], x[k + 1][2], w.x, w.y);
    cfft_inv_bfly(x[k][1], x[k + 1][1], x[k][3], x[k + 1][3], w.x, w.y);
  }
  if constexpr (PASS > 0) {
    cfft_exchange<LOGC, S0, S0 - 2>(x, xb, tau, th);
    cfft_inverse<LOGC, PASS - 1>(x, tw, xb, tau, th);
  }
}

}  // namespace rosetta
