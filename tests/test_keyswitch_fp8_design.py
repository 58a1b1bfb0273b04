"""CPU model of the 8-bit key switch's number formats (keyswitch_fp8.cu): signed
5-bit limbs that e4m3 holds exactly, their recombination mod 2^64, and the
bound on the fp32 sums."""

import numpy as np
import pytest

import workload as W

M64 = (1 << 64) - 1


def e4m3_values():
    """Every finite e4m3 value (4 exponent bits, bias 7, 3 mantissa bits)."""
    out = set()
    for s in (1, -1):
        for e in range(16):
            for m in range(8):
                if e == 15 and m == 7:
                    continue                                   # NaN
                out.add(s * (m / 8 * 2.0 ** -6 if e == 0 else (1 + m / 8) * 2.0 ** (e - 7)))
    return out


def limbs(w):
    off = sum(16 << (5 * t) for t in range(12))
    v = (w + off) & M64
    return [((v >> (5 * t)) & 31) - (16 if t < 12 else 0) for t in range(13)]


def test_digits_and_limbs_are_e4m3_integers():
    vals = e4m3_values()
    assert all(float(i) in vals for i in range(-16, 17))
    assert 17.0 not in vals


def test_limbs_recombine_mod_2_64():
    g = np.random.default_rng(3)
    words = [0, 1, M64, 1 << 63, (1 << 63) - 1, 15, 16, 17, (-16) & M64]
    for w in words + [int(x) for x in g.integers(0, 1 << 64, 2000, dtype=np.uint64)]:
        ls = limbs(w)
        assert all(-16 <= x <= 15 for x in ls[:12]) and 0 <= ls[12] <= 15
        assert sum(x << (5 * t) for t, x in enumerate(ls)) & M64 == w


@pytest.mark.parametrize("name", sorted(W.CONFIGS))
def test_sums_of_the_named_sets_are_exact_in_fp32(name):
    p = W.CONFIGS[name]
    assert 2 ** (p.ks_base_log - 1) * 16 * p.kN * p.ks_level < 2 ** 24
