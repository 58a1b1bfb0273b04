"""The 8-bit tensor-core key switch (bases up to 2^5): tile edges in both
directions, K splits, and the largest sums its accumulators can see, every
output word against the oracle."""

import numpy as np
import pytest

import oracle as O
import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _params(N, n, base_log, level):
    return W.Params(f"k{N}_{n}_{base_log}x{level}", n=n, k=1, N=N, pbs_base_log=10, pbs_level=1, ks_base_log=base_log,
                    ks_level=level, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",),
                    msg=("uniform",), batch=1, seed=N + n + base_log)


def _check(p, ksk, big):
    import paper_2609_16915_gb300 as R
    ctx = R.Context(p)
    ctx.upload_ksk(G.to_dev(ksk))
    got = G.gpu_keyswitch(ctx, p, big)
    ctx.close()
    assert np.array_equal(got, O.keyswitch_batch(p, ksk, big))


@pytest.mark.parametrize("N,n,base_log,level,batch", [
    (256, 1, 5, 1, 1), (256, 15, 4, 4, 9), (256, 16, 1, 1, 128), (512, 14, 3, 5, 129), (512, 31, 4, 8, 256),
    (1024, 47, 2, 3, 257), (2048, 64, 5, 12, 7), (2048, 742, 3, 5, 1), (4096, 840, 4, 5, 61), (8192, 33, 4, 6, 255)])
def test_tile_edges_bitexact(N, n, base_log, level, batch):
    p = _params(N, n, base_log, level)
    g = np.random.default_rng(N + n + batch)
    ksk = g.integers(0, 2**64, size=p.ksk_shape(), dtype=np.uint64)
    big = g.integers(0, 2**64, size=(batch, p.kN + 1), dtype=np.uint64)
    _check(p, ksk, big)


@pytest.mark.parametrize("base_log,level,batch", [(8, 2, 260), (6, 3, 256), (8, 2, 30)])
def test_wider_bases_keep_their_kernels(base_log, level, batch):
    """Bases of 2^6 and more: bf16 limbs from 256 ciphertexts on, CUDA cores below."""
    p = _params(512, 20, base_log, level)
    g = np.random.default_rng(base_log + batch)
    _check(p, g.integers(0, 2**64, size=p.ksk_shape(), dtype=np.uint64),
           g.integers(0, 2**64, size=(batch, p.kN + 1), dtype=np.uint64))


@pytest.mark.parametrize("N,base_log,level", [(2048, 3, 5), (8192, 5, 7), (8192, 4, 6)])
@pytest.mark.parametrize("limbs", ["low", "high"])
def test_largest_sums(N, base_log, level, limbs):
    """Every digit at -B/2, every limb of every key word at -16 or at 15: the
    sums reach 16 x 16 x 57344 = 0.88 x 2^24 in the widest case."""
    p = _params(N, 40, base_log, level)
    bits, B = base_log * level, 1 << base_log
    C = sum((B >> 1) << (m * base_log) for m in range(level))
    a = (((-C) % (1 << bits)) << (64 - bits)) % (1 << 64)
    off = sum(16 << (5 * t) for t in range(12))
    word = (-off) % (1 << 64) if limbs == "low" else ((1 << 64) - 1 - off) % (1 << 64)
    _check(p, np.full(p.ksk_shape(), np.uint64(word), np.uint64), np.full((140, p.kN + 1), np.uint64(a), np.uint64))
