"""Two host threads, each with a context and a stream of its own, whose batches take
the same kernels with different amounts of shared memory (one and three workers per SM;
other LWE dimensions): every call succeeds and gives its words."""

import threading

import numpy as np
import pytest

import workload as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2609_16915_gb300 import build
    build.build()


def _params(N, n, base_log, level):
    return W.Params(f"thr{N}_{n}", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=level, ks_base_log=4, ks_level=4,
                    msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",), msg=("uniform",), batch=1,
                    seed=n)


def _together(jobs, repeats):
    """Each job in a thread of its own, called as fast as a host thread can: the
    library is entered without the interpreter's lock."""
    start, failed = threading.Barrier(len(jobs)), []

    def work(job):
        start.wait()
        for _ in range(repeats):
            status = job()
            if status != 0:
                failed.append(status)
                return

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


def _sizes():
    import torch
    S = torch.cuda.get_device_properties(0).multi_processor_count
    return S, 3 * S


@pytest.mark.parametrize("kind", ["workers", "dimensions", "trace"])
def test_threads_with_their_own_contexts(kind):
    import torch
    import paper_2609_16915_gb300 as R
    L = R.load()
    one, three = _sizes()
    g = np.random.default_rng(5)
    jobs, checks, ctxs = [], [], []
    sets = {"workers": [(_params(2048, 2, 23, 1), one), (_params(2048, 2, 23, 1), three)],
            "dimensions": [(_params(256, 2, 10, 2), 90), (_params(256, 20000, 10, 2), 80)],
            "trace": [(_params(2048, 2, 23, 1), 2 * one), (_params(2048, 2, 23, 1), three)]}[kind]
    for p, batch in sets:
        ctx, stream = R.Context(p), torch.cuda.Stream()
        ctxs.append(ctx)
        ctx.upload_bsk(G.to_dev(g.integers(0, 2**64, size=p.bsk_shape(), dtype=np.uint64)))
        if kind == "trace":
            ctx.upload_trace_keys(G.to_dev(g.integers(0, 2**64, size=(11, 2, 2, p.N), dtype=np.uint64)), 16, 2)
            x = G.to_dev(g.integers(0, 2**64, size=(batch, 2, p.N), dtype=np.uint64))
            want, out = G.empty_dev(batch, 2, p.N), G.empty_dev(batch, 2, p.N)
            ctx.trace_batch(x, want)
            jobs.append(lambda h=ctx._h, a=x.data_ptr(), b=batch, o=out.data_ptr(), s=stream.cuda_stream:
                        L.rosetta_trace_batch(h, a, b, o, s))
        else:
            x, lut = G.to_dev(G.sparse_lwe(p, batch, 1, seed=p.n)), G.to_dev(W.lut_torus(p))
            want, out = G.empty_dev(batch, p.kN + 1), G.empty_dev(batch, p.kN + 1)
            ctx.blind_rotate_extract_batch(x, lut, want)
            jobs.append(lambda h=ctx._h, a=x.data_ptr(), b=batch, l=lut.data_ptr(), o=out.data_ptr(),
                        s=stream.cuda_stream: L.rosetta_blind_rotate_extract_batch(h, a, b, l, o, s))
        ctx.sync_status()
        checks.append((out, want, x, stream))
    _together(jobs, 4000)
    torch.cuda.synchronize()
    for c, (out, want, _, _) in zip(ctxs, checks):
        c.sync_status()
        assert torch.equal(out, want)
        c.close()
