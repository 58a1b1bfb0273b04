"""The cluster kernels of the blind rotation, past the batches that the small-batch
kernel takes, against the oracle: every compiled ring size, digit width, level and
exchange buffer, LUTs, many LUTs, GLWE test polynomials, a LUT index out of range, and the
largest magnitudes.

A few different ciphertexts fill the batch over and over, and every copy's words are
compared.  At a large LWE dimension all but a few mask words are zero: their CMux steps add
nothing, so the oracle runs on the other words and their key blocks alone."""

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
    return W.Params(f"c{N}_{base_log}x{level}_{n}", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=level,
                    ks_base_log=4, ks_level=2, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20,
                    lut=("square_mod",), msg=("uniform",), batch=1, seed=N + 7 * base_log + level + n)


def _batch(N):
    """Past the small-batch kernel's largest batch, and at N = 2048 below a whole wave of
    the worker kernel."""
    import torch
    S = torch.cuda.get_device_properties(0).multi_processor_count
    return {512: S * 3 // 4 + 4, 1024: S // 5 + 5, 2048: S // 10 + 3, 4096: S * 3 // 20 + 2, 8192: 3}[N]


def _setup(N, base_log, level, n, few=None):
    """Context, its parameters, and the oracle's: the mask words that are not zero (all, or
    `few` with the first and the last), their key blocks and the ciphertexts."""
    import torch
    import paper_2609_16915_gb300 as R
    p = _params(N, base_log, level, n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(p.seed)
    bsk = torch.randint(-(1 << 63), (1 << 63) - 1, p.bsk_shape(), dtype=torch.int64, device="cuda", generator=gen)
    g = np.random.default_rng(p.seed)
    steps = np.arange(n) if few is None else np.unique(np.r_[0, n - 1, g.choice(n, few, replace=False)])
    small = g.integers(0, 2**64, size=(3, len(steps) + 1), dtype=np.uint64)
    lwe = np.zeros((3, n + 1), np.uint64)
    lwe[:, np.r_[steps, n]] = small
    po = _params(N, base_log, level, len(steps))
    key = G.to_host(bsk[torch.from_numpy(steps).cuda()])
    ctx = R.Context(p)
    ctx.upload_bsk(bsk)
    del bsk
    torch.cuda.empty_cache()
    return ctx, p, lwe, po, key, small


CASES = [
    # four primes
    (512, 10, 2, 4, None), (512, 28, 1, 4, None), (512, 7, 5, 3, None), (512, 21, 3, 3, None),
    (1024, 16, 1, 4, None), (1024, 24, 2, 3, None), (1024, 9, 6, 2, None),
    (2048, 16, 1, 4, None), (2048, 23, 1, 4, None), (2048, 28, 1, 3, None), (2048, 13, 2, 3, None), (2048, 24, 2, 3, None),
    (2048, 11, 3, 3, None), (2048, 21, 3, 2, None), (2048, 16, 4, 2, None), (2048, 16, 1, 6500, 4), (2048, 15, 2, 6500, 3),
    (4096, 28, 1, 3, None), (4096, 16, 2, 3, None), (4096, 24, 2, 2, None), (4096, 16, 3, 2, None), (4096, 9, 5, 2, None),
    # three primes, exchange in pairs and (from these dimensions on) in single words
    (4096, 16, 1, 4, None), (4096, 15, 2, 3, None), (4096, 15, 3, 3, None), (4096, 11, 3, 3, None),
    (4096, 16, 1, 7680, 4), (4096, 15, 2, 4608, 4), (4096, 15, 3, 1536, 3),
    (4096, 16, 1, 7679, 2), (4096, 15, 2, 4607, 2), (4096, 15, 3, 1535, 2),
    (8192, 15, 1, 3, None), (8192, 14, 2, 2, None), (8192, 14, 3, 2, None),
    (8192, 15, 1, 15900, 3), (8192, 14, 2, 9728, 2), (8192, 14, 3, 3584, 2), (8192, 14, 3, 3583, 2),
]


@pytest.mark.parametrize("N,base_log,level,n,few", CASES)
def test_every_cluster_kernel_bitexact(N, base_log, level, n, few):
    ctx, p, lwe, po, key, small = _setup(N, base_log, level, n, few)
    batch = _batch(N)
    which = np.arange(batch) % 3
    lut = W.lut_torus(p)
    assert np.array_equal(G.gpu_br_extract(ctx, p, lwe[which], lut),
                          O.blind_rotate_extract_batch(po, key, small, lut)[which])
    glwe = np.random.default_rng(n).integers(0, 2**64, size=(3, 2, N), dtype=np.uint64)
    out = G.empty_dev(batch, 2, N)
    ctx.blind_rotate_glwe_batch(G.to_dev(lwe[which]), G.to_dev(glwe[which]), out)
    ctx.sync_status()
    assert np.array_equal(G.to_host(out), O.blind_rotate_glwe_batch(po, key, small, glwe)[which])
    ctx.close()


@pytest.mark.parametrize("N,base_log,level,n", [(512, 10, 2, 3), (1024, 16, 1, 3), (2048, 23, 1, 3), (2048, 15, 2, 3),
                                                (4096, 16, 1, 3), (4096, 15, 2, 3), (4096, 15, 3, 2), (8192, 14, 3, 2)])
def test_many_luts_and_an_index_out_of_range(N, base_log, level, n):
    """Each ciphertext its own table; one index out of range takes table 0 and is reported
    once."""
    import torch
    import paper_2609_16915_gb300 as R
    ctx, p, lwe, po, key, _ = _setup(N, base_log, level, n)
    g = np.random.default_rng(N)
    ksk = g.integers(0, 2**64, size=p.ksk_shape(), dtype=np.uint64)
    ctx.upload_ksk(G.to_dev(ksk))
    batch = _batch(N)
    which, index = np.arange(batch) % 3, (np.arange(batch) // 3) % 4
    luts = np.stack([W.lut_torus(p, codes=[(m * (j + 1) + j) % 8 for m in range(8)]) for j in range(4)])
    want = {(c, j): O.pbs_batch(p, key, ksk, lwe[c:c + 1], luts[j])[0]
            for c, j in sorted(set(zip(which.tolist(), index.tolist())))}
    out = G.empty_dev(batch, p.n + 1)
    d_lwe, d_luts = G.to_dev(lwe[which]), G.to_dev(luts)
    ctx.pbs_batch_multi_lut(d_lwe, d_luts, torch.from_numpy(index.astype(np.int32)).cuda(), out)
    ctx.sync_status()
    assert np.array_equal(G.to_host(out), np.stack([want[c, j] for c, j in zip(which, index)]))
    bad = index.copy()
    bad[batch - 2] = 4
    ctx.pbs_batch_multi_lut(d_lwe, d_luts, torch.from_numpy(bad.astype(np.int32)).cuda(), out)
    with pytest.raises(R.RosettaError) as e:
        ctx.sync_status()
    assert e.value.status == -1
    ctx.sync_status()
    got, bad[batch - 2] = G.to_host(out), 0
    want.update({(which[batch - 2], 0): O.pbs_batch(p, key, ksk, lwe[which[batch - 2]][None], luts[0])[0]})
    assert np.array_equal(got, np.stack([want[c, j] for c, j in zip(which, bad)]))
    ctx.close()


@pytest.mark.parametrize("N,base_log,level", [(512, 28, 2), (1024, 28, 2), (2048, 28, 1), (2048, 28, 2), (4096, 15, 3),
                                              (4096, 28, 2), (8192, 14, 3)])
@pytest.mark.parametrize("sign", [+1, -1])
def test_external_product_at_its_largest_magnitude(N, base_log, level, sign):
    p, batch = _params(N, base_log, level, 2), _batch(N)
    bsk, lwe, glwe, C = X.case(p, sign, seed=N + level)
    ctx = G.make_ctx(p, bsk, W.uniform_keys(p)[1])
    out = G.empty_dev(batch, 2, N)
    ctx.blind_rotate_glwe_batch(G.to_dev(np.repeat(lwe, batch, axis=0)), G.to_dev(np.repeat(glwe, batch, axis=0)), out)
    ctx.sync_status()
    want = np.array(X.expected(p, bsk, C)[0], dtype=np.uint64)
    assert np.array_equal(G.to_host(out), np.broadcast_to(want, (batch, 2, N)))
    ctx.close()
