"""Blind rotation at N = 256 with one CTA per ciphertext (batches above 7/16 of the
SMs), at the levels and digit widths it takes, against the oracle."""

import numpy as np
import pytest

import oracle as O
import workload as W
from tests import extreme_util as X
from tests import gpu_util as G
from tests.test_gpu_small_batch import _params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _batch():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * 7 // 16 + 1


@pytest.mark.parametrize("base_log,level,n", [(10, 2, 9), (28, 2, 4), (28, 1, 5), (7, 9, 3), (4, 16, 2), (1, 33, 1)])
def test_every_level_bitexact(base_log, level, n):
    """Dense masks, skipped steps at both ends and an all-zero mask; the whole
    bootstrapping, several LUTs and GLWE test polynomials."""
    p, batch = _params(256, base_log, level, n), _batch()
    bsk, ksk = W.uniform_keys(p)
    lwe = W.uniform_ciphertexts(p, batch, sub=2)
    lwe[1, 0] = lwe[1, n - 1] = 0
    lwe[2, :n] = 0
    lut = W.lut_torus(p)
    ctx = G.make_ctx(p, bsk, ksk)
    d_lwe = G.to_dev(lwe)
    want = O.blind_rotate_extract_batch(p, bsk, lwe, lut)
    assert np.array_equal(G.gpu_br_extract(ctx, p, lwe, lut), want)
    assert np.array_equal(G.gpu_pbs(ctx, p, lwe, lut), O.keyswitch_batch(p, ksk, want))

    import torch
    g = np.random.default_rng(n)
    luts = np.stack([lut, g.integers(0, 2**64, size=lut.shape, dtype=np.uint64)])
    index = (np.arange(batch) % 2).astype(np.int32)
    out = G.empty_dev(batch, n + 1)
    ctx.pbs_batch_multi_lut(d_lwe, G.to_dev(luts), torch.from_numpy(index).cuda(), out)
    ctx.sync_status()
    both = [O.keyswitch_batch(p, ksk, O.blind_rotate_extract_batch(p, bsk, lwe, l)) for l in luts]
    assert np.array_equal(G.to_host(out), np.where(index[:, None] == 0, both[0], both[1]))

    glwe = g.integers(0, 2**64, size=(batch, 2, 256), dtype=np.uint64)
    gout = G.empty_dev(batch, 2, 256)
    ctx.blind_rotate_glwe_batch(d_lwe, G.to_dev(glwe), gout)
    ctx.sync_status()
    assert np.array_equal(G.to_host(gout), O.blind_rotate_glwe_batch(p, bsk, lwe, glwe))
    ctx.close()


@pytest.mark.parametrize("sign", [+1, -1])
def test_external_product_at_its_largest_magnitude(sign):
    p, batch = _params(256, 28, 2, 2), _batch()
    bsk, lwe, glwe, C = X.case(p, sign, seed=256)
    ctx = G.make_ctx(p, bsk, W.uniform_keys(p)[1])
    out = G.empty_dev(batch, 2, 256)
    ctx.blind_rotate_glwe_batch(G.to_dev(np.repeat(lwe, batch, axis=0)), G.to_dev(np.repeat(glwe, batch, axis=0)), out)
    ctx.sync_status()
    want, _ = X.expected(p, bsk, C)
    got = G.to_host(out)
    assert all(np.array_equal(got[b], got[0]) for b in range(batch))
    assert [[int(w) for w in row] for row in got[0]] == want
    ctx.close()
