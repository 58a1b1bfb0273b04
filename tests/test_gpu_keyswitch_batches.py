"""The 8-bit key switch past 2,097,120 ciphertexts (65535 groups of 32), the most
a second grid dimension would take."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


@pytest.mark.parametrize("batch", [2097120, 2097121, 2200003])
def test_more_ciphertexts_than_a_second_grid_dimension_takes(batch):
    """2039 different ciphertexts over and over: each block of 2039 outputs equals
    the first, which is a batch of ordinary size."""
    import torch
    import paper_2609_16915_gb300 as R
    p = W.Params("many", n=3, k=1, N=256, pbs_base_log=10, pbs_level=1, ks_base_log=5, ks_level=2, msg_bits=3,
                 lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1, seed=2)
    g = np.random.default_rng(7)
    ctx = R.Context(p)
    ctx.upload_ksk(G.to_dev(g.integers(0, 2**64, size=p.ksk_shape(), dtype=np.uint64)))
    few = G.to_dev(g.integers(0, 2**64, size=(2039, p.kN + 1), dtype=np.uint64))
    want = G.empty_dev(2039, p.n + 1)
    ctx.keyswitch_batch(few, want)
    big = few.repeat(batch // 2039 + 1, 1)[:batch]
    out = torch.zeros((batch, p.n + 1), dtype=torch.int64, device="cuda")
    ctx.keyswitch_batch(big, out)
    ctx.sync_status()
    whole = batch // 2039 * 2039
    assert torch.equal(out[:whole].view(-1, 2039, p.n + 1), want.expand(whole // 2039, -1, -1))
    assert torch.equal(out[whole:], want[:batch - whole])
    ctx.close()
    del big, out
    torch.cuda.empty_cache()
