"""Run in a child process by tests/test_gpu_lost_words.py: with the library built
with -DROSETTA_DEBUG (a process holds one librosetta), make the small-batch blind
rotation miss words at every ring size and level it has a kernel for, then use the
same context again.  Prints one JSON line: case -> [status, status after it, words right]."""

import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import oracle as O  # noqa: E402
import paper_2609_16915_gb300 as R  # noqa: E402
import workload as W  # noqa: E402


def status(ctx):
    try:
        ctx.sync_status()
        return 0
    except R.RosettaError as e:
        return e.status


def main():
    R.load(R.DEBUG_LIB_PATH)
    from tests import gpu_util as G
    res = {}
    for N, base_log, level in [(256, 10, 2), (512, 8, 5), (1024, 16, 1), (2048, 23, 1), (2048, 15, 2), (4096, 16, 1),
                               (4096, 15, 2), (4096, 15, 3)]:
        for n in (1, 2, 3, 4, 7):                      # the lost step: the first to the fourth, the last one too
            p = W.Params(f"lost{N}_{level}_{n}", n=n, k=1, N=N, pbs_base_log=base_log, pbs_level=level, ks_base_log=4,
                         ks_level=4, msg_bits=3, lwe_sigma_log2=40, glwe_sigma_log2=20, lut=("square_mod",),
                         msg=("uniform",), batch=1, seed=N + n)
            bsk, ksk = W.uniform_keys(p)
            ctx = G.make_ctx(p, bsk, ksk)
            ctx.selftest_lost_words(2000)
            first, second = status(ctx), status(ctx)
            lwe, lut = W.uniform_ciphertexts(p, 2, sub=1), W.lut_torus(p)
            right = np.array_equal(G.gpu_br_extract(ctx, p, lwe, lut), O.blind_rotate_extract_batch(p, bsk, lwe, lut))
            res[f"{N} {level} {n}"] = [first, second, bool(right)]
            ctx.close()
    print(json.dumps(res), flush=True)


if __name__ == "__main__":
    main()
