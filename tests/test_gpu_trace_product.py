"""The trace and the plaintext product at every ring size: both digit widths of
the trace, the largest gadgets, and plaintexts and words at the ends of their
ranges, every output word against the oracle."""

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


def _ctx(N):
    import paper_2609_16915_gb300 as R
    p = W.Params(f"r{N}", n=4, k=1, N=N, pbs_base_log=10, pbs_level=1, ks_base_log=4, ks_level=4, msg_bits=3,
                 lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1, seed=N)
    return R.Context(p)


@pytest.mark.parametrize("N,base_log,level", [(256, 16, 4), (256, 17, 2), (512, 28, 2), (512, 8, 8), (1024, 16, 2),
                                              (1024, 20, 2), (2048, 17, 2), (2048, 4, 16), (4096, 16, 4), (4096, 21, 2)])
def test_trace(N, base_log, level):
    g = np.random.default_rng(N + base_log)
    keys = g.integers(0, 2**64, size=(N.bit_length() - 1, level, 2, N), dtype=np.uint64)
    glwe = g.integers(0, 2**64, size=(2, 2, N), dtype=np.uint64)
    glwe[1, :, ::3] = np.uint64(1 << 63)
    glwe[1, :, 1::3] = np.uint64((1 << 64) - 1)
    ctx = _ctx(N)
    ctx.upload_trace_keys(G.to_dev(keys), base_log, level)
    out = G.empty_dev(2, 2, N)
    ctx.trace_batch(G.to_dev(glwe), out)
    ctx.sync_status()
    assert np.array_equal(G.to_host(out), O.trace_batch(keys, glwe, base_log, level))
    ctx.close()


@pytest.mark.parametrize("N", [256, 512, 1024, 2048, 4096])
def test_plaintext_product_at_the_ends_of_the_range(N):
    """Constant words and plaintext coefficients of one sign at the largest
    magnitude (2 N 2^31 2^63 before reduction), the digits' carry edges, and
    uniform ones."""
    g = np.random.default_rng(N)
    lo = np.iinfo(np.int64).min
    edges = np.array([0, 1, (1 << 31) - 1, 1 << 31, (1 << 31) + 1, (1 << 32) - 1, 1 << 32, 1 << 63, (1 << 63) - 1,
                      ((1 << 63) - 1) ^ (1 << 31), (1 << 64) - 1, 0x7FFFFFFF80000000, 0x8000000080000000,
                      0x800000007FFFFFFF], dtype=np.uint64)
    glwe = g.integers(0, 2**64, size=(4, 2, N), dtype=np.uint64)
    glwe[0] = np.uint64(0x8000000080000000 - (1 << 63))     # low digit -2^31
    glwe[1] = np.uint64(1 << 63)                             # high digit -2^31
    glwe[2] = g.choice(edges, size=(2, N))
    q = g.integers(0, 2**64, size=N, dtype=np.uint64)
    ctx = _ctx(N)
    for P in (np.full(N, lo), np.full(N, -(lo + 1)), g.integers(lo, -(lo + 1), N, endpoint=True)):
        out = G.empty_dev(4, 2, N)
        ctx.plaintext_mul_batch(G.to_dev(glwe), P.astype(np.int64), out, q)
        assert np.array_equal(G.to_host(out), O.plaintext_mul_batch(glwe, P, q))
    ctx.close()


@pytest.mark.parametrize("N,batch", [(256, 1), (512, 40), (2048, 1), (2048, 400), (4096, 90)])
def test_each_product_takes_its_own_plaintext(N, batch):
    """Calls one after the other on the same buffers: a product kernel starts before
    its plaintext is transformed and must not meet the rows of the call before."""
    g = np.random.default_rng(N + batch)
    glwe = g.integers(0, 2**64, size=(batch, 2, N), dtype=np.uint64)
    pick = sorted({0, batch // 2, batch - 1})
    ctx = _ctx(N)
    d_in, out = G.to_dev(glwe), G.empty_dev(batch, 2, N)
    for _ in range(4):
        P = g.integers(-(1 << 40), 1 << 40, N)
        q = g.integers(0, 2**64, size=N, dtype=np.uint64)
        ctx.plaintext_mul_batch(d_in, P, out, q)
        assert np.array_equal(G.to_host(out[pick]), O.plaintext_mul_batch(glwe[pick], P, q))
    ctx.close()
