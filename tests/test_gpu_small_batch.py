"""The small-batch blind rotation (two CTAs per prime, component-wise) at every
ring size and level it is compiled for, against the oracle, and its batch limit
against the cluster kernels."""

import numpy as np
import pytest

import oracle as O
import workload as W
from tests import extreme_util as X
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _params(N, base_log, level, n):
    return W.Params(f"b{N}_{base_log}x{level}_{n}", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=level,
                    ks_base_log=4, ks_level=4, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20,
                    lut=("square_mod",), msg=("uniform",), batch=1, seed=N + 7 * base_log + level + n)


@pytest.mark.parametrize("N,base_log,level,n,batch", [
    (256, 10, 2, 7, 3), (256, 28, 1, 5, 1), (256, 7, 9, 4, 2), (512, 8, 6, 5, 2), (512, 21, 3, 4, 3), (1024, 16, 1, 4, 2),
    (1024, 12, 5, 3, 1), (2048, 23, 1, 4, 3), (2048, 28, 1, 3, 1), (2048, 15, 2, 3, 2), (2048, 28, 2, 2, 1),
    (4096, 16, 1, 3, 1), (4096, 15, 2, 3, 2), (4096, 15, 3, 2, 1)])
def test_every_level_bitexact(N, base_log, level, n, batch):
    """Dense masks (and one ciphertext with skipped steps at both ends and in
    between), the whole bootstrapping and GLWE test polynomials."""
    p = _params(N, base_log, level, n)
    bsk, ksk = W.uniform_keys(p)
    lwe = W.uniform_ciphertexts(p, batch, sub=2)
    if batch > 1:
        lwe[1, 0] = lwe[1, n - 1] = 0
    lut = W.lut_torus(p)
    ctx = G.make_ctx(p, bsk, ksk)
    want = O.blind_rotate_extract_batch(p, bsk, lwe, lut)
    assert np.array_equal(G.gpu_br_extract(ctx, p, lwe, lut), want)
    assert np.array_equal(G.gpu_pbs(ctx, p, lwe, lut), O.keyswitch_batch(p, ksk, want))
    g = np.random.default_rng(n)
    glwe = g.integers(0, 2**64, size=(batch, 2, N), dtype=np.uint64)
    out = G.empty_dev(batch, 2, N)
    ctx.blind_rotate_glwe_batch(G.to_dev(lwe), G.to_dev(glwe), out)
    ctx.sync_status()
    assert np.array_equal(G.to_host(out), O.blind_rotate_glwe_batch(p, bsk, lwe, glwe))
    ctx.close()


@pytest.mark.parametrize("N,base_log,level", [(256, 10, 2), (512, 8, 6), (1024, 15, 2), (2048, 23, 1), (2048, 15, 2),
                                              (4096, 15, 2)])
def test_long_chains_equal_the_cluster_kernels(N, base_log, level):
    """A hundred dense steps, the same ciphertexts one and a few at a time (this
    kernel) and as one large batch (the others)."""
    import torch
    p = _params(N, base_log, level, 100)
    batch = 200 if N <= 2048 else 40
    bsk, ksk = W.uniform_keys(p)
    ctx = G.make_ctx(p, bsk, ksk)
    d_in = G.to_dev(W.uniform_ciphertexts(p, batch, sub=4))
    lut = G.to_dev(W.lut_torus(p))
    whole, part = G.empty_dev(batch, p.n + 1), G.empty_dev(batch, p.n + 1)
    ctx.pbs_batch(d_in, lut, whole)
    a = 0
    while a < batch:
        b = min(batch, a + 1 + a % 14)
        ctx.pbs_batch(d_in[a:b], lut, part[a:b])
        a = b
    ctx.sync_status()
    assert torch.equal(whole, part)
    ctx.close()


@pytest.mark.parametrize("N,base_log,level", [(256, 28, 2), (1024, 28, 2), (2048, 28, 1), (4096, 15, 3)])
@pytest.mark.parametrize("sign", [+1, -1])
def test_external_product_at_its_largest_magnitude(N, base_log, level, sign):
    p = _params(N, base_log, level, 2)
    bsk, lwe, glwe, C = X.case(p, sign, seed=N + level)
    ctx = G.make_ctx(p, bsk, W.uniform_keys(p)[1])
    out = G.empty_dev(1, 2, N)
    ctx.blind_rotate_glwe_batch(G.to_dev(lwe), G.to_dev(glwe), out)
    ctx.sync_status()
    want, _ = X.expected(p, bsk, C)
    assert [[int(w) for w in row] for row in G.to_host(out)[0]] == want
    ctx.close()
