"""The worker-per-ciphertext blind rotation (N = 2048, one level, float
quotient) that full batches take, against the oracle and against the cluster
kernel that small batches take."""

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


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _params(base_log, n):
    return W.Params(f"s{base_log}_{n}", n=n, k=1, N=2048, pbs_base_log=base_log, pbs_level=1, ks_base_log=3,
                    ks_level=5, msg_bits=4, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",),
                    msg=("uniform",), batch=1, seed=base_log + 100 * n)


@pytest.mark.parametrize("base_log,n", [(23, 2), (24, 1), (1, 1), (16, 1)])
def test_every_output_word_against_the_oracle(base_log, n):
    """One worker per SM with a few SMs idle: every word of blind rotation +
    extraction, and of the whole bootstrapping."""
    p = _params(base_log, n)
    batch = _sms() - 3
    bsk, ksk = W.uniform_keys(p)
    lwe = W.uniform_ciphertexts(p, batch, sub=1)
    lwe[5, :n] = 0                                  # no CMux step at all
    lut = W.lut_torus(p)
    ctx = G.make_ctx(p, bsk, ksk)
    want = O.blind_rotate_extract_batch(p, bsk, lwe, lut)
    assert np.array_equal(G.gpu_br_extract(ctx, p, lwe, lut), want)
    assert np.array_equal(G.gpu_pbs(ctx, p, lwe, lut), O.keyswitch_batch(p, ksk, want))
    ctx.close()


@pytest.mark.parametrize("waves,extra", [(0, -1), (1, 1), (1, 2), (2, -1), (2, 1), (3, 0), (3, 1), (5, 2)])
def test_batch_split_equals_the_cluster_kernel(waves, extra):
    """Batches around the lines of the dispatch rule (whole waves of three
    workers, one or two workers, a cluster-kernel rest), many LUTs, full
    masks: the words of the same ciphertexts in slices small enough for the
    cluster kernel."""
    import torch
    p = _params(23, 12)
    S = _sms()
    batch = S - S // 4 + 1 if waves == 0 else waves * S + extra
    bsk, ksk = W.uniform_keys(p)
    ctx = G.make_ctx(p, bsk, ksk)
    lwe = W.uniform_ciphertexts(p, batch, sub=waves)
    codes = W.lut_codes(p)
    luts = G.to_dev(np.stack([W.lut_torus(p, np.roll(codes, r)) for r in range(3)]))
    idx = torch.from_numpy((np.arange(batch) % 3).astype(np.int32)).cuda()
    d_in, out = G.to_dev(lwe), G.empty_dev(batch, p.n + 1)
    ctx.pbs_batch_multi_lut(d_in, luts, idx, out)
    ctx.sync_status()
    part = G.empty_dev(batch, p.n + 1)
    for a in range(0, batch, 64):
        b = min(batch, a + 64)
        ctx.pbs_batch_multi_lut(d_in[a:b], luts, idx[a:b], part[a:b])
    ctx.sync_status()
    assert torch.equal(out, part)
    ctx.close()


@pytest.mark.parametrize("base_log", [23, 24])
@pytest.mark.parametrize("sign", [+1, -1])
def test_external_product_at_its_largest_magnitude(base_log, sign):
    """Every digit at -B/2 against key words of one sign close to 2^63 (the
    largest quotient the float estimate has to place), GLWE test polynomials,
    on a batch for the workers, against the closed form."""
    p = _params(base_log, 2)
    bsk, lwe, glwe, C = X.case(p, sign, seed=base_log)
    batch = _sms()
    ctx = G.make_ctx(p, bsk, W.uniform_keys(p)[1])
    out = G.empty_dev(batch, 2, p.N)
    ctx.blind_rotate_glwe_batch(G.to_dev(np.repeat(lwe, batch, 0)), G.to_dev(np.repeat(glwe, batch, 0)), out)
    ctx.sync_status()
    got = G.to_host(out)
    want, peak = X.expected(p, bsk, C)
    assert peak > 1 << (base_log + 73)
    assert np.array_equal(got, np.repeat(got[:1], batch, 0))
    assert [[int(w) for w in row] for row in got[0]] == want
    ctx.close()


def test_many_lut_index_out_of_range_is_reported_and_not_followed():
    import paper_2609_16915_gb300 as R
    import torch
    p = _params(23, 2)
    batch = _sms()
    bsk, ksk = W.uniform_keys(p)
    ctx = G.make_ctx(p, bsk, ksk)
    lwe = W.uniform_ciphertexts(p, batch, sub=3)
    lut = W.lut_torus(p)
    idx = torch.zeros(batch, dtype=torch.int32, device="cuda")
    idx[7] = 9
    out = G.empty_dev(batch, p.n + 1)
    ctx.pbs_batch_multi_lut(G.to_dev(lwe), G.to_dev(lut[None]), idx, out)
    with pytest.raises(R.RosettaError) as e:
        ctx.sync_status()
    assert e.value.status == -1
    assert np.array_equal(G.to_host(out), G.gpu_pbs(ctx, p, lwe, lut))
    ctx.close()
