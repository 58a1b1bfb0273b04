"""Device memory too short for what is only there to be faster: the second formats of
the keys at N = 2048, and the lookup's scratch for several segments at a time.  The
calls succeed all the same, with the same words."""

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


class _Left:
    """All device memory but about `mib` MiB taken, for the length of a with block."""

    def __init__(self, mib):
        self.mib, self.held = mib, []

    def __enter__(self):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        for step in (1024, 64, 2):
            while True:
                over = (torch.cuda.mem_get_info()[0] // MIB - self.mib) // step * step
                if over <= 0:
                    break
                try:
                    self.held.append(torch.empty(over * MIB, dtype=torch.uint8, device="cuda"))
                except torch.OutOfMemoryError:
                    break
        return self

    def __exit__(self, *exc):
        import torch
        self.held.clear()
        torch.cuda.empty_cache()


def _lookup_set(p, seed, n_seg):
    g = np.random.default_rng(seed)
    N = p.N
    return {"trace": G.to_dev(g.integers(0, 2**64, size=(N.bit_length() - 1, 4, 2, N), dtype=np.uint64)),
            "table": (g.integers(-2**40, 2**40, size=N), g.integers(0, 2**64, size=N, dtype=np.uint64),
                      g.integers(-2**40, 2**40, size=(n_seg, N)),
                      g.integers(0, 2**64, size=(n_seg, N), dtype=np.uint64))}


def _params(N, n, base_log, level):
    return W.Params("short", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=level, ks_base_log=4, ks_level=4, msg_bits=3,
                    lwe_sigma_log2=24, glwe_sigma_log2=24, lut=("square_mod",), msg=("uniform",), batch=1, seed=n)


def test_lookup_one_segment_at_a_time():
    """512 lookups of eight segments at N = 4096: 2 x 256 MiB for all segments, 2 x 32 for
    one.  Short on memory twice in a row, then with more, then after another upload."""
    import torch
    p, batch = _params(4096, 3, 15, 2), 512
    s = _lookup_set(p, 1, 8)
    bsk, ksk = W.uniform_keys(p)
    g = np.random.default_rng(2)
    x = G.to_dev(g.integers(0, 2**64, size=(batch, 2, p.N), dtype=np.uint64))
    lwe = G.to_dev(W.uniform_ciphertexts(p, batch, sub=4))
    want, out = G.empty_dev(batch, 2, p.N), G.empty_dev(batch, 2, p.N)

    def context():
        ctx = G.make_ctx(p, bsk, ksk)
        ctx.upload_trace_keys(s["trace"], 16, 4)
        ctx.upload_lookup_table(*s["table"])
        return ctx

    def run(ctx, rows=batch):
        out.zero_()
        ctx.segmented_lookup_batch(x[:rows], lwe[:rows], out[:rows])
        ctx.sync_status()
        assert torch.equal(out[:rows], want[:rows])

    ample = context()
    ample.segmented_lookup_batch(x, lwe, want)
    ample.sync_status()
    ample.close()
    ctx = context()
    with _Left(400):
        run(ctx)
        free = torch.cuda.mem_get_info()[0]
        run(ctx)
        run(ctx, 511)
        assert abs(torch.cuda.mem_get_info()[0] - free) < 16 * MIB    # nothing allocated and freed again
    run(ctx)
    ctx.upload_lookup_table(*s["table"])
    run(ctx)
    ctx.close()


@pytest.mark.parametrize("key", ["bootstrapping", "trace"])
def test_keys_without_their_second_format(key):
    """N = 2048: the bootstrapping key (and with it the trace's), or the trace key alone,
    in one format only; whole waves of ciphertexts, which the other format's kernels would
    have taken, and a rest."""
    import torch
    import paper_2609_16915_gb300 as R
    p = _params(2048, 400, 23, 1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    batch = 3 * sms + 30
    g = np.random.default_rng(3)
    bsk = G.to_dev(g.integers(0, 2**64, size=p.bsk_shape(), dtype=np.uint64))     # 50 MiB a format
    trace = G.to_dev(g.integers(0, 2**64, size=(11, 4, 2, p.N), dtype=np.uint64))   # 2.75 MiB a format
    lwe = G.to_dev(G.sparse_lwe(p, batch, 5, seed=4))
    glwe = G.to_dev(g.integers(0, 2**64, size=(batch, 2, p.N), dtype=np.uint64))
    lut = G.to_dev(W.lut_torus(p))
    outs = [(G.empty_dev(batch, p.kN + 1), G.empty_dev(batch, 2, p.N)) for _ in range(2)]

    def run(ctx, o):
        ctx.blind_rotate_extract_batch(lwe, lut, o[0])
        ctx.trace_batch(glwe, o[1])
        ctx.sync_status()

    def same():
        assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])

    ample = R.Context(p)
    ample.upload_bsk(bsk)
    ample.upload_trace_keys(trace, 16, 4)
    run(ample, outs[0])
    short = R.Context(p)
    if key == "trace":
        short.upload_bsk(bsk)
    with _Left(72 if key == "bootstrapping" else 6):
        before = torch.cuda.mem_get_info()[0]
        if key == "bootstrapping":
            short.upload_bsk(bsk)
            assert 50 * MIB <= before - torch.cuda.mem_get_info()[0] < 60 * MIB
            short.upload_trace_keys(trace, 16, 4)
        else:
            short.upload_trace_keys(trace, 16, 4)
            assert 2 * MIB <= before - torch.cuda.mem_get_info()[0] <= 4 * MIB
        run(short, outs[1])
    same()
    short.upload_bsk(bsk)                                    # with memory again
    short.upload_trace_keys(trace, 16, 4)
    run(short, outs[1])
    same()
    short.close()
    ample.close()
