"""One gadget level at the small rings, where a component has a single row: the
small-batch kernel and, at N = 256, the kernel of one CTA per ciphertext, on both sides of
their dispatch lines, against the oracle."""

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


def _params(N, base_log, n):
    return W.Params(f"one{N}_{base_log}_{n}", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=1, ks_base_log=4,
                    ks_level=4, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",),
                    msg=("uniform",), batch=1, seed=N + base_log + n)


@pytest.mark.parametrize("N,base_log,n,batches", [(256, 28, 6, (1, 66, 67, 305)), (256, 9, 5, (2, 200)),
                                                  (512, 28, 4, (1, 110, 111, 116)), (512, 16, 5, (3, 120)),
                                                  (1024, 28, 3, (1, 30, 40)), (1024, 16, 4, (2, 60))])
def test_one_row_per_component_bitexact(N, base_log, n, batches):
    """Dense masks and one with skipped steps, seven different ciphertexts over and over;
    LUTs, GLWE test polynomials."""
    p = _params(N, base_log, n)
    bsk, ksk = W.uniform_keys(p)
    lwe = W.uniform_ciphertexts(p, 7, sub=2)
    lwe[3, 0] = lwe[3, n - 1] = 0
    glwe = np.random.default_rng(n).integers(0, 2**64, size=(7, 2, N), dtype=np.uint64)
    lut = W.lut_torus(p)
    want = O.blind_rotate_extract_batch(p, bsk, lwe, lut)
    want_glwe = O.blind_rotate_glwe_batch(p, bsk, lwe, glwe)
    ctx = G.make_ctx(p, bsk, ksk)
    for batch in batches:
        which = np.arange(batch) % 7
        assert np.array_equal(G.gpu_br_extract(ctx, p, lwe[which], lut), want[which])
        out = G.empty_dev(batch, 2, N)
        ctx.blind_rotate_glwe_batch(G.to_dev(lwe[which]), G.to_dev(glwe[which]), out)
        ctx.sync_status()
        assert np.array_equal(G.to_host(out), want_glwe[which])
    ctx.close()


@pytest.mark.parametrize("N,batch", [(256, 70), (512, 5), (1024, 5)])
@pytest.mark.parametrize("sign", [+1, -1])
def test_external_product_at_its_largest_magnitude(N, batch, sign):
    p = _params(N, 28, 2)
    bsk, lwe, glwe, C = X.case(p, sign, seed=N)
    ctx = G.make_ctx(p, bsk, W.uniform_keys(p)[1])
    out = G.empty_dev(batch, 2, N)
    ctx.blind_rotate_glwe_batch(G.to_dev(np.repeat(lwe, batch, axis=0)), G.to_dev(np.repeat(glwe, batch, axis=0)), out)
    ctx.sync_status()
    want, _ = X.expected(p, bsk, C)
    for got in G.to_host(out):
        assert [[int(w) for w in row] for row in got] == want
    ctx.close()
