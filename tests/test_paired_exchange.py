"""CPU models of the paired exchange layout (ntt.cuh: xb_pad2), the float
transforms' slot swizzle (cfft.cuh: cfft_swz), the split twiddle table
(split_tw_slot) and the closed-form gadget digits (modarith.cuh)."""

import numpy as np
import pytest


def passes(L):
    n = (L + 2) // 3
    return [(3 * i, 3 if i < n - 1 else L - 3 * (n - 1)) for i in range(n)]


def pad2(i):
    return i + 2 * (i >> 4)


def positions(L, S0, H, tau):
    """Element positions of the 8 slots of thread tau (non-last: one block)."""
    N, SIG, SPAN = 1 << L, (1 << L) >> (S0 + H), (1 << L) >> S0
    if SIG == 1:
        return [8 * tau + e for e in range(8)]
    return [(tau // SIG) * SPAN + tau % SIG + e * SIG for e in range(8)]


def wavefronts(units, group, width):
    """Accesses of one warp, `group` lanes at a time, `units` in elements of
    width/4 words: the largest number of distinct units on one bank group."""
    banks = 128 // width
    worst = 0
    for k in range(0, 32, group):
        seen = {}
        for u in units[k:k + group]:
            seen.setdefault(u % banks, set()).add(u)
        worst = max(worst, max(len(v) for v in seen.values()))
    return worst


@pytest.mark.parametrize("L", [11, 12, 13])
def test_pairs_are_bijective_in_bounds_additive_and_conflict_free(L):
    N, T = 1 << L, (1 << L) // 8
    for S0, H in passes(L):
        SIG = N >> (S0 + H)
        seen = set()
        for tau in range(T):
            pos = positions(L, S0, H, tau)
            base = pad2(pos[0])
            for e, i in enumerate(pos):
                off = pad2(e if SIG == 1 else e * SIG)
                assert base + off == pad2(i) < N + N // 8
                seen.add(i)
            if SIG == 1:
                assert base % 2 == 0                       # 16-byte accesses of two elements
        assert len(seen) == N
        for w in range(0, T, 32):
            lanes = [positions(L, S0, H, t) for t in range(w, w + 32)]
            if SIG == 1:
                for k in range(4):                         # quarter-warps, two elements each
                    assert wavefronts([pad2(p[2 * k]) // 2 for p in lanes], 8, 16) == 1
            else:
                for e in range(8):                         # half-warps, one element each
                    assert wavefronts([pad2(p[e]) for p in lanes], 16, 8) == 1


def test_float_slots_are_bijective_linear_and_conflict_free():
    C, swz = 1024, lambda i: i ^ ((i >> 3) & 3) ^ ((i >> 2) & 4)
    assert sorted(map(swz, range(C))) == list(range(C))
    for S0 in range(0, 10, 2):
        SIG = C >> (S0 + 2)
        for w in range(0, 256, 32):
            for e in range(4):
                units = []
                for tau in range(w, w + 32):
                    b = (tau // SIG) * 4 * SIG + tau % SIG
                    assert swz(b) ^ swz(e * SIG) == swz(b + e * SIG)
                    units.append(swz(b + e * SIG))
                assert wavefronts(units, 8, 16) == 1


@pytest.mark.parametrize("L", [11, 12, 13])
def test_split_twiddle_table(L):
    N = 1 << L
    slot = lambda i: i if i < N // 2 else N // 2 + ((i >> 1) & 1) * (N // 4) + (((i - N // 2) >> 2) << 1) + (i & 1)
    assert sorted(map(slot, range(N))) == list(range(N))
    for start in range(N // 2, N, 4):                      # the four entries a thread loads
        for k in range(2):
            a = N // 2 + k * (N // 4) + (start - N // 2) // 2
            assert [slot(start + 2 * k), slot(start + 2 * k + 1)] == [a, a + 1] and a % 2 == 0
    for S in range(6):                                     # warp-uniform groups of the first six stages
        SIG = N >> (3 + 3 * (S // 3))
        assert SIG >= 32 and (2 << S) <= 64


@pytest.mark.parametrize("beta,level", [(23, 1), (15, 2), (14, 3), (16, 4), (28, 2), (1, 1), (1, 64), (10, 2), (8, 6), (7, 9)])
def test_closed_form_digits_equal_the_carry_rule(beta, level):
    g = np.random.default_rng(beta * 100 + level)
    M = (1 << 64) - 1
    B, half, bits = 1 << beta, 1 << (beta - 1), beta * level
    edges = [0, 1, M, 1 << 63, (1 << 63) - 1, (1 << 63) + 1]
    for m in range(1, level + 1):
        for d in (-1, 0, 1):
            for s in (half << (64 - m * beta), (half << (64 - m * beta)) - (1 << max(0, 63 - bits)), (B - 1) << (64 - m * beta)):
                edges.append((s + d) & M)
    off = (0 if bits >= 64 else 1 << (63 - bits)) + sum(1 << (64 - m * beta + beta - 1) for m in range(1, level + 1))
    for v in edges + [int(x) for x in g.integers(0, 1 << 64, 3000, dtype=np.uint64)]:
        cv = v if bits >= 64 else ((v + (1 << (63 - bits))) & M) >> (64 - bits)
        want = [0] * level
        for lev in range(level - 1, -1, -1):
            d = cv & (B - 1)
            cv >>= beta
            if d >= half:
                d, cv = d - B, cv + 1
            want[lev] = d
        w = (v + off) & M
        assert [((w >> (64 - (lev + 1) * beta)) & (B - 1)) - half for lev in range(level)] == want
