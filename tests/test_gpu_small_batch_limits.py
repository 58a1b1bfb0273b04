"""LWE dimensions around the most the small-batch kernel's shared memory holds: the
context takes that kernel or the cluster kernel, and either gives the words that a
larger batch gets from the cluster kernel."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


# shared memory without the 2 (n + 1) bytes of the switched mask reaches 227 KB at n
# about 62448 (N = 2048, one level) and 25072 (N = 4096, one level)
@pytest.mark.parametrize("N,first,last", [(2048, 62430, 62466), (4096, 25054, 25090)])
def test_every_dimension_at_the_edge_of_shared_memory(N, first, last):
    import torch
    import paper_2609_16915_gb300 as R
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    words = torch.randint(-(1 << 63), (1 << 63) - 1, (last, 2, 2, N), dtype=torch.int64, device="cuda", generator=g)
    rng = np.random.default_rng(N)
    batch = 24                                      # beyond the small-batch kernel
    for n in sorted({first, last} | set(range(first, last, 4))):
        p = W.Params(f"edge{n}", n=n, k=1, N=N, pbs_base_log=16, pbs_level=1, ks_base_log=4, ks_level=1, msg_bits=3,
                     lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1, seed=n)
        lwe = np.zeros((batch, n + 1), np.uint64)   # few steps, the first and the last among them
        for i in (0, 1, n // 2, n - 1, n):
            lwe[:, i] = rng.integers(0, 2**64, size=batch, dtype=np.uint64)
        ctx = R.Context(p)
        ctx.upload_bsk(words[:n])
        d_in, lut = G.to_dev(lwe), G.to_dev(W.lut_torus(p))
        whole, part = G.empty_dev(batch, N + 1), G.empty_dev(2, N + 1)
        ctx.blind_rotate_extract_batch(d_in, lut, whole)
        ctx.blind_rotate_extract_batch(d_in[:1], lut, part[:1])
        ctx.blind_rotate_extract_batch(d_in[1:2], lut, part[1:])
        ctx.sync_status()
        assert torch.equal(whole[:2], part), n
        ctx.close()
    del words
    torch.cuda.empty_cache()
