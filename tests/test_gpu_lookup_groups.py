"""The segmented lookup with its segments in one launch, in several groups and
one at a time: the same words."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


@pytest.mark.parametrize("n_seg,batch", [(8, 1100), (4, 4097), (2, 2048)])
def test_groups_of_segments_give_the_same_words(n_seg, batch):
    """1100 ciphertexts: groups of 3, 3 and 2 segments; 4097: one at a time;
    against slices small enough for all segments at once."""
    import torch
    p = W.Params("groups", n=6, k=1, N=256, pbs_base_log=10, pbs_level=2, ks_base_log=4, ks_level=4, msg_bits=3,
                 lwe_sigma_log2=24, glwe_sigma_log2=24, lut=("square_mod",), msg=("uniform",), batch=1, seed=9)
    g = np.random.default_rng(n_seg)
    bsk, ksk = W.uniform_keys(p)
    ctx = G.make_ctx(p, bsk, ksk)
    ctx.upload_trace_keys(G.to_dev(g.integers(0, 2**64, size=(8, 4, 2, 256), dtype=np.uint64)), 16, 4)
    ctx.upload_lookup_table(g.integers(-2**40, 2**40, size=256), g.integers(0, 2**64, size=256, dtype=np.uint64),
                            g.integers(-2**40, 2**40, size=(n_seg, 256)),
                            g.integers(0, 2**64, size=(n_seg, 256), dtype=np.uint64))
    x = G.to_dev(g.integers(0, 2**64, size=(batch, 2, 256), dtype=np.uint64))
    lwe = G.to_dev(W.uniform_ciphertexts(p, batch, sub=n_seg))
    whole, part = G.empty_dev(batch, 2, 256), G.empty_dev(batch, 2, 256)
    ctx.segmented_lookup_batch(x, lwe, whole)
    for a in range(0, batch, 97):
        b = min(batch, a + 97)
        ctx.segmented_lookup_batch(x[a:b], lwe[a:b], part[a:b])
    ctx.sync_status()
    assert torch.equal(whole, part)
    ctx.close()
