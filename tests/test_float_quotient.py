"""CPU model of the float quotient (csrc/cfft.cuh, modarith.cuh: qf_quotient):
the single-precision transforms in the kernel's order of operations, their
error against the stated worst case, and the CRT over three 28-bit primes
whose multiple of the primes' product comes from the estimate."""

import math

import numpy as np
import pytest

PRIMES = (268369921, 268271617, 268238849)      # kPrimeList, the first three
M3 = math.prod(PRIMES)
SHIFT = 16                                       # kQfShift
F = np.float32
LOGN = 11
C = 1 << (LOGN - 1)


def fma(a, b, c):
    """float32 fused multiply-add: the product is exact in float64, the sum
    rounds to 53 bits before it rounds to 24 (an extra 2^-53)."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def twiddles():
    e = [0, C // 2] + [0] * (C - 2)
    for m in range(1, C // 2):
        e[2 * m], e[2 * m + 1] = e[m] // 2, e[m] // 2 + C
    a = np.array(e) * (math.pi / (1 << LOGN))
    return np.cos(a), np.sin(a)


WR, WI = twiddles()


def stage_twiddles(s):
    """float32 twiddles of stage s: odd groups of odd stages use i times their
    left neighbour's, as the kernel does."""
    g = np.arange(1 << s)
    if s % 2 == 0:
        return WR[(1 << s) + g].astype(F), WI[(1 << s) + g].astype(F)
    left = (1 << s) + (g & ~1)
    wr, wi = WR[left].astype(F), WI[left].astype(F)
    return np.where(g & 1, -wi, wr), np.where(g & 1, wr, wi)


def forward(re, im):
    for s in range(LOGN - 1):
        wr, wi = (w[:, None] for w in stage_twiddles(s))
        re, im = re.reshape(1 << s, 2, -1), im.reshape(1 << s, 2, -1)
        Xr, Yr, Xi, Yi = re[:, 0], re[:, 1], im[:, 0], im[:, 1]
        ar = fma(-wi, Yi, fma(wr, Yr, Xr))
        ai = fma(wi, Yr, fma(wr, Yi, Xi))
        two = F(2) * np.ones_like(ar)
        re = np.stack([ar, fma(two, Xr, -ar)], 1)
        im = np.stack([ai, fma(two, Xi, -ai)], 1)
    return re.reshape(-1), im.reshape(-1)


def inverse(re, im):
    for s in range(LOGN - 2, -1, -1):
        wr, wi = (w[:, None] for w in stage_twiddles(s))
        re, im = re.reshape(1 << s, 2, -1), im.reshape(1 << s, 2, -1)
        Xr, Yr, Xi, Yi = re[:, 0], re[:, 1], im[:, 0], im[:, 1]
        dr, di = Xr - Yr, Xi - Yi
        re = np.stack([Xr + Yr, fma(di, wi, dr * wr)], 1)
        im = np.stack([Xi + Yi, fma(-dr, wi, di * wr)], 1)
    return re.reshape(-1), im.reshape(-1)


def key_transform(g):
    """Double precision (numpy complex), scaled, rounded once."""
    z = np.array([complex(float(a), float(b)) for a, b in zip(g[:C], g[C:])])
    w = WR + 1j * WI
    for s in range(LOGN - 1):
        z = z.reshape(1 << s, 2, -1)
        t = z[:, 1] * w[(1 << s):(2 << s), None]
        z = np.stack([z[:, 0] + t, z[:, 0] - t], 1)
    z = z.reshape(-1) * (2.0 ** SHIFT / C / float(M3))
    return z.real.astype(F), z.imag.astype(F)


def estimate(digits, keys):
    """2^SHIFT X / M3 for X = sum_r digits[r] * keys[r], per coefficient."""
    sr = si = np.zeros(C, F)
    for d, g in zip(digits, keys):
        zr, zi = forward(d[:C].astype(F), d[C:].astype(F))
        gr, gi = key_transform(g)
        sr, si = fma(-zi, gi, fma(zr, gr, sr)), fma(zi, gr, fma(zr, gi, si))
    return np.concatenate(inverse(sr, si))


def exact(digits, keys):
    N = 2 * C
    out = np.zeros(N, dtype=object)
    for d, g in zip(digits, keys):
        gl = [int(v) for v in g]
        # negacyclic convolution with Python integers through one big-integer product
        bits = 128
        off = 1 << 90
        A = sum(int(v) << (bits * i) for i, v in enumerate(d))
        B = sum(v << (bits * i) for i, v in enumerate(gl))
        P = A * B
        neg = P < 0
        P = abs(P)
        co, carry = [], 0
        for i in range(2 * N):
            v = (P >> (bits * i)) & ((1 << bits) - 1)
            v += carry
            carry = 0
            if v >= 1 << (bits - 1):
                v -= 1 << bits
                carry = 1
            co.append(-v if neg else v)
        assert off
        out += np.array([co[i] - co[i + N] for i in range(N)], dtype=object)
    return out


def quotient(ys, est):
    """qf_quotient on 32-bit words, from y < 8p."""
    ysum = 0
    for y in ys:
        assert 0 <= y < 8 * PRIMES[0] < 1 << 31
        ysum += y >> 17
    assert ysum < 1 << 16
    fi = int(np.rint(np.float64(est)))
    assert -(1 << 31) <= fi < 1 << 31
    t = ((ysum << (SHIFT - 11)) + (1 << 31) + (1 << (SHIFT - 1)) - fi) % (1 << 32)
    return t >> SHIFT


def cases():
    g = np.random.default_rng(5)
    N = 2 * C
    top = (1 << 63) - 1
    for beta in (23, 24, 8):
        half = 1 << (beta - 1)
        yield beta, [g.integers(-half, half, N) for _ in range(2)], [g.integers(-top - 1, top, N) for _ in range(2)]
        # largest magnitude: every term of coefficient N - 1 (or 0) of one sign
        yield beta, [np.full(N, -half)] * 2, [np.full(N, top)] * 2
        yield beta, [np.full(N, -half)] * 2, [np.full(N, -top - 1)] * 2
        s = np.where(np.arange(N) % 2, 1, -1)
        yield beta, [-half * (s > 0).astype(np.int64) + (half - 1) * (s < 0)] * 2, [np.where(s > 0, top, -top)] * 2


@pytest.mark.parametrize("case", list(cases()), ids=lambda c: f"beta{c[0]}")
def test_estimate_and_quotient_give_the_exact_product(case):
    beta, digits, keys = case
    X = exact(digits, keys)
    est = estimate(digits, keys)
    # the stated worst case: 100 u (k+1) l N 2^(beta-1) 2^63, u = 2^-24
    bound = 2 * 2 * C * (1 << (beta - 1)) * (1 << 63)
    assert bound <= 1 << 98
    err = max(abs(float(e) * float(M3) / 2 ** SHIFT - float(x)) for e, x in zip(est, X))
    assert err <= 100 * 2.0 ** -24 * float(bound)
    g = np.random.default_rng(beta)
    for j in (0, 1, C - 1, C, 2 * C - 1, *g.integers(0, 2 * C, 40)):
        x = int(X[j])
        ys = []
        for q, p in enumerate(PRIMES):
            y = x * pow(M3 // p, -1, p) % p
            ys.append(y + p * int(g.integers(0, 8 if y + 7 * p < 8 * p else 7)))   # any representative below 8p
        u = quotient(ys, est[j])
        w = sum(y * (M3 // p) for y, p in zip(ys, PRIMES)) - u * M3 + (1 << (31 - SHIFT)) * M3
        assert w == x


def test_margin_of_the_rule():
    """Shortfall of 2^28 against p for y < 8p, the dropped low bits, and the
    estimate's worst case for the largest admitted bound stay below one half."""
    short = sum(8 * (2 ** 28 - p) / 2 ** 28 + 2.0 ** -11 for p in PRIMES)
    est = 100 * 2.0 ** -24 * 2.0 ** 98 / M3 + 2.0 ** -(SHIFT + 1)
    assert short + est < 0.25
    assert 2.0 ** 98 / M3 * 2 ** SHIFT * 1.01 < 2 ** 31     # the conversion to int32
