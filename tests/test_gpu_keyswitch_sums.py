"""The 8-bit tensor-core key switch where its fp32 accumulators are almost full
and their low bits count.

Sums just below 2^24 whose terms are not all multiples of a power of two: large
products (digit and limb at -B/2 and -16) with small odd ones among them, before
them, behind them, and products that cancel them again.  The accumulators have to
be exact integers all the way; one that keeps fewer bits than 24, or drops the
low bits of a small product beside a large one, gives other words.  K is not split
(the tiles alone fill the GPU), so each accumulator takes a whole sum.
Checked on a choice of rows and columns against the definition with integers mod 2^64."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

LIMBS = 13


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _large_share(order, rows, g):
    """For each of the sum's rows: is it a large product?  (0: small and odd)"""
    if order == "mixed":
        return g.random(rows) < 0.97
    if order == "alternating":      # both within every K = 32 instruction
        return np.arange(rows) % 32 != 5
    large = np.ones(rows, bool)
    k = rows // 24
    if order == "small last":
        large[-k:] = False
    else:
        large[:k] = False
    return large


# sums up to 0.85 x 2^24 (base 2^5), 0.91 x 2^24 (base 2^4) and 0.73 x 2^24 (base 2^3)
@pytest.mark.parametrize("N,base_log,level", [(8192, 5, 7), (8192, 4, 15), (8192, 3, 21)])
@pytest.mark.parametrize("order", ["mixed", "alternating", "small last", "small first", "cancelling"])
def test_low_bits_of_nearly_full_sums(N, base_log, level, order):
    import torch
    import paper_2609_16915_gb300 as R
    n, batch = 1215, 512                       # 76 column tiles x 2 row tiles
    p = W.Params(f"s{N}_{base_log}x{level}", n=n, k=1, N=N, pbs_base_log=10, pbs_level=1, ks_base_log=base_log,
                 ks_level=level, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",),
                 msg=("uniform",), batch=1, seed=1)
    assert 2 ** (base_log - 1) * 16 * N * level < 2 ** 24
    g = np.random.default_rng(N + base_log + len(order))
    rows = N * level                           # in the kernel's order: level-major
    half = 1 << (base_log - 1)
    if order == "cancelling":                  # up to the middle and down again, odd products in between
        large = _large_share("mixed", rows, g)
        sign = np.where(np.arange(rows) < rows // 2, -1, 1)
    else:
        large = _large_share(order, rows, g)
        sign = np.full(rows, -1)
    # digits: -B/2 at the large rows, small and odd at the others (8 patterns of small ones)
    odd = 2 * g.integers(0, max(1, half // 2), size=(8, rows)) + 1
    odd = np.where(g.random((8, rows)) < 0.5, -np.minimum(odd, half - 1), np.minimum(odd, half - 1))
    d = np.where(large[None, :], -half, odd)   # [8][rows]
    # words with exactly these digits: sum of d 2^(64 - (lev+1) beta)
    a = np.zeros((8, N), np.uint64)
    for lev in range(level):
        a += d[:, lev * N:(lev + 1) * N].astype(np.int64).view(np.uint64) << np.uint64(64 - (lev + 1) * base_log)
    big = np.empty((batch, N + 1), np.uint64)
    pattern = g.integers(0, 8, size=batch)
    big[:, :N] = a[pattern]
    big[:, N] = g.integers(0, 2**64, size=batch, dtype=np.uint64)
    # key words from their limbs: -16 (or 15) at the large rows, -15 .. 15 odd at the others; 16 patterns of
    # columns, top limbs 0 .. 15
    extreme = np.where(sign < 0, -16, 15)
    cols = np.zeros((16, rows), np.uint64)
    for t in range(LIMBS):
        small = 2 * g.integers(-8, 8, size=(16, rows)) + 1
        limb = np.where(large[None, :], extreme[None, :], small)
        if t == LIMBS - 1:
            limb = np.abs(limb) % 16
        cols += limb.astype(np.int64).view(np.uint64) << np.uint64(5 * t)
    # ksk [i][lev][j], j of pattern (5 j) mod 16
    which = (5 * np.arange(n + 1)) % 16
    dev = torch.from_numpy(np.ascontiguousarray(cols.reshape(16, level, N).transpose(2, 1, 0)).view(np.int64)).cuda()
    ksk = dev[:, :, torch.from_numpy(which).cuda()].contiguous()
    del dev
    ctx = R.Context(p)
    ctx.upload_ksk(ksk)
    got = G.gpu_keyswitch(ctx, p, big)
    ctx.close()
    del ksk
    torch.cuda.empty_cache()
    prod = np.zeros((8, 16), np.uint64)
    for k in range(0, rows, 4096):             # d KSK mod 2^64 of every pair of patterns
        prod += (d[:, None, k:k + 4096].astype(np.int64).view(np.uint64) * cols[None, :, k:k + 4096]).sum(
            axis=2, dtype=np.uint64)
    want = np.uint64(0) - prod[pattern][:, which]
    want[:, n] += big[:, N]
    assert np.array_equal(got, want)
