"""The trace by one worker per ciphertext (N = 2048, three primes and a float
quotient) at the gadgets it takes and where batches are split, against the oracle and
the cluster kernel, which small batches take."""

import numpy as np
import pytest

import oracle as O
import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
N, LOGN = 2048, 11


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _ctx():
    p = W.Params("trs", n=4, k=1, N=N, pbs_base_log=23, pbs_level=1, ks_base_log=4, ks_level=4, msg_bits=3,
                 lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1, seed=7)
    bsk, ksk = W.uniform_keys(p)
    return G.make_ctx(p, bsk, ksk)


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


# in multiples of the SM count: two workers, three, whole waves and each kind of rest
@pytest.mark.parametrize("base_log,level", [(16, 4), (24, 2), (12, 4), (1, 2), (32 - 4, 2)])
def test_every_split_gives_the_same_words(base_log, level):
    """(2^28 x 2 lies past the float quotient's bound: clusters only.)"""
    import torch
    S = _sms()
    ctx = _ctx()
    g = np.random.default_rng(base_log)
    keys = g.integers(0, 2**64, size=(LOGN, level, 2, N), dtype=np.uint64)
    ctx.upload_trace_keys(G.to_dev(keys), base_log, level)
    most = 6 * S + 1
    glwe = g.integers(0, 2**64, size=(most, 2, N), dtype=np.uint64)
    d_in, small = G.to_dev(glwe), G.empty_dev(most, 2, N)
    for a in range(0, most, 100):
        ctx.trace_batch(d_in[a:a + 100], small[a:a + 100])
    for batch in (S * 5 // 3 + 1, 2 * S, 2 * S + S // 4 + 1, 3 * S, 3 * S + 1, 5 * S - 1, 6 * S - 1, most):
        out = G.empty_dev(batch, 2, N)
        ctx.trace_batch(d_in[:batch], out)
        ctx.sync_status()
        assert torch.equal(out, small[:batch]), batch
    pick = [0, S, 3 * S - 1]
    assert np.array_equal(G.to_host(small[pick]), O.trace_batch(keys, glwe[pick], base_log, level))
    ctx.close()


@pytest.mark.parametrize("base_log,level", [(16, 4), (24, 2)])
@pytest.mark.parametrize("key_word", [1 << 63, (1 << 63) - 1])
def test_largest_magnitude(base_log, level, key_word):
    """Keys of one word of the largest magnitude and either sign; every digit of the
    first automorphism's image is -B/2 (ciphertext 0) or B/2 - 1, then random."""
    batch = 2 * _sms()
    ctx = _ctx()
    g = np.random.default_rng(level)
    keys = np.full((LOGN, level, 2, N), key_word, dtype=np.uint64)
    ctx.upload_trace_keys(G.to_dev(keys), base_log, level)
    B = 1 << base_log
    low = sum(-(B // 2) << (64 - base_log * m) for m in range(1, level + 1)) % 2**64
    high = sum((B // 2 - 1) << (64 - base_log * m) for m in range(1, level + 1)) % 2**64
    glwe = g.integers(0, 2**64, size=(batch, 2, N), dtype=np.uint64)
    for b, w in ((0, low), (1, high)):
        glwe[b, 0, 0::2] = w               # sigma of the first step, X -> X^(N+1), negates the odd coefficients
        glwe[b, 0, 1::2] = (-w) % 2**64
    out = G.empty_dev(batch, 2, N)
    ctx.trace_batch(G.to_dev(glwe), out)
    ctx.sync_status()
    pick = [0, 1, batch - 1]
    assert np.array_equal(G.to_host(out)[pick], O.trace_batch(keys, glwe[pick], base_log, level))
    ctx.close()


def test_keys_of_another_gadget_replace_the_first():
    S = _sms()
    ctx = _ctx()
    g = np.random.default_rng(5)
    glwe = g.integers(0, 2**64, size=(2 * S, 2, N), dtype=np.uint64)
    d_in, out = G.to_dev(glwe), G.empty_dev(2 * S, 2, N)
    pick = [0, 2 * S - 1]
    for base_log, level in ((16, 4), (24, 2), (10, 6), (13, 4)):
        keys = g.integers(0, 2**64, size=(LOGN, level, 2, N), dtype=np.uint64)
        ctx.upload_trace_keys(G.to_dev(keys), base_log, level)
        ctx.trace_batch(d_in, out)
        ctx.sync_status()
        assert np.array_equal(G.to_host(out)[pick], O.trace_batch(keys, glwe[pick], base_log, level))
    ctx.close()
