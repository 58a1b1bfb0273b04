"""Calls captured in CUDA graphs, replayed after other calls have made the context's
scratch grow."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _captured(call):
    """A graph of one call (made once before, so that its kernels are loaded)."""
    import torch
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    return graph


@pytest.mark.parametrize("base_log,level,batch", [(4, 5, 1), (4, 5, 61), (3, 5, 255), (6, 3, 200)])
def test_small_key_switch_outlives_a_larger_one(base_log, level, batch):
    """Key switches of up to 255 ciphertexts hold no scratch that a larger batch
    replaces (base 2^6: the CUDA-core kernel, which has none)."""
    import torch
    import paper_2609_16915_gb300 as R
    p = W.Params("graph", n=100, k=1, N=1024, pbs_base_log=10, pbs_level=1, ks_base_log=base_log, ks_level=level,
                 msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1,
                 seed=batch)
    g = np.random.default_rng(batch)
    ctx = R.Context(p)
    ctx.upload_ksk(G.to_dev(g.integers(0, 2**64, size=p.ksk_shape(), dtype=np.uint64)))
    big = G.to_dev(g.integers(0, 2**64, size=(9000, p.kN + 1), dtype=np.uint64))
    out, want, many = (G.empty_dev(b, p.n + 1) for b in (batch, batch, 9000))
    graph = _captured(lambda: ctx.keyswitch_batch(big[:batch], out))
    want.copy_(out)
    for rows in (300, 9000, 5000):
        ctx.keyswitch_batch(big[:rows], many[:rows])
        out.zero_()
        graph.replay()
        ctx.sync_status()
        assert torch.equal(out, want)
        assert torch.equal(many[:batch], want)
    ctx.close()


def _lookup_context(n_seg):
    p = W.Params("graph_lk", n=5, k=1, N=256, pbs_base_log=10, pbs_level=2, ks_base_log=4, ks_level=4, msg_bits=3,
                 lwe_sigma_log2=24, glwe_sigma_log2=24, lut=("square_mod",), msg=("uniform",), batch=1, seed=3)
    g = np.random.default_rng(n_seg)
    bsk, ksk = W.uniform_keys(p)
    ctx = G.make_ctx(p, bsk, ksk)
    ctx.upload_trace_keys(G.to_dev(g.integers(0, 2**64, size=(8, 4, 2, 256), dtype=np.uint64)), 16, 4)
    _upload_table(ctx, n_seg)
    return p, ctx


def _upload_table(ctx, n_seg):
    g = np.random.default_rng(100 + n_seg)
    ctx.upload_lookup_table(g.integers(-2**40, 2**40, size=256), g.integers(0, 2**64, size=256, dtype=np.uint64),
                            g.integers(-2**40, 2**40, size=(n_seg, 256)),
                            g.integers(0, 2**64, size=(n_seg, 256), dtype=np.uint64))


def _lookup_inputs(p, batch):
    g = np.random.default_rng(batch)
    return (G.to_dev(g.integers(0, 2**64, size=(batch, 2, 256), dtype=np.uint64)),
            G.to_dev(W.uniform_ciphertexts(p, batch, sub=4)))


@pytest.mark.parametrize("warm,captured,later", [(2000, 1365, (819, 512, 100, 1)), (1000, 1000, (819, 512, 999)),
                                                 (4096, 300, (4000, 1365, 4096))])
def test_lookup_works_in_what_a_larger_one_left(warm, captured, later):
    """A lookup is captured after one of a larger batch, whose groups of segments were
    smaller, and replayed after smaller batches with larger groups."""
    import torch
    p, ctx = _lookup_context(8)
    x, lwe = _lookup_inputs(p, 4096)
    out, other = G.empty_dev(captured, 2, 256), G.empty_dev(4096, 2, 256)
    ctx.segmented_lookup_batch(x[:warm], lwe[:warm], other[:warm])
    torch.cuda.synchronize()
    want = other[:captured].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.segmented_lookup_batch(x[:captured], lwe[:captured], out)
    for rows in later:
        ctx.segmented_lookup_batch(x[:rows], lwe[:rows], other[:rows])
        out.zero_()
        graph.replay()
        ctx.sync_status()
        assert torch.equal(out, want)
        assert torch.equal(other[:min(rows, captured)], want[:min(rows, captured)])
    ctx.close()


def test_lookup_of_a_longer_table_is_captured_in_the_scratch_there_is():
    """The first lookup of a table with more segments, captured: in the scratch that the
    shorter table's lookups left (one segment at a time); then as usual."""
    import torch
    p, ctx = _lookup_context(2)
    x, lwe = _lookup_inputs(p, 300)
    out, want = G.empty_dev(300, 2, 256), G.empty_dev(300, 2, 256)
    ctx.segmented_lookup_batch(x, lwe, want)
    _upload_table(ctx, 16)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.segmented_lookup_batch(x, lwe, out)
    graph.replay()
    torch.cuda.synchronize()
    ctx.segmented_lookup_batch(x, lwe, want)
    ctx.sync_status()
    assert torch.equal(out, want)
    ctx.close()
