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
