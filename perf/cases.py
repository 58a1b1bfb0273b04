"""The work a user of this library has it do, as timed cases: bootstrapping
calls from one ciphertext to a whole decode token's activations at every named
parameter set, the key switch alone, and the pieces and the whole of the
encrypted segmented lookup.  Sizes are those of the named workloads
(``workload.CONFIGS``), of the batch sweep and of the benchmark's lookup.

A case is a dict: ``kind`` (the entry point), ``set`` (the parameter set),
``batch``, and where they apply ``n`` (another LWE dimension than the set's),
``luts`` (tables of a many-LUT call), ``host`` (ciphertexts in pinned host
memory) and ``segments`` (of the lookup's table).
"""

from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

import paper_2609_16915_gb300 as R
import workload as W
from paper_2609_16915_gb300 import segmented as SG

TRACE_BASE_LOG, TRACE_LEVEL = 16, 4     # gadget of the trace keys (the benchmark's lookup)
DX, DR = 32, 30                         # fixed-point scales of the lookup's x and values


def listed():
    return [
        # one softmax logit on its own: the latency of a single bootstrapping
        {"name": "pbs_one", "kind": "pbs", "set": "exp_sweep", "batch": 1},
        # the smallest parameter set, a short vector of 3-bit messages
        {"name": "pbs_tiny", "kind": "pbs", "set": "tiny", "batch": 16},
        # the logits of one attention head over a short, odd context
        {"name": "pbs_ragged", "kind": "pbs", "set": "exp_sweep", "batch": 77},
        # the standard set at its full batch: 4-bit GELU (the headline workload)
        {"name": "pbs_standard", "kind": "pbs", "set": "standard", "batch": 4096},
        # one GPT-2-small token: 3072 MLP activations, 6-bit GELU, N = 4096
        {"name": "pbs_gpt2_mlp", "kind": "pbs", "set": "gpt2_mlp", "batch": 3072},
        # a slice of one LLaMA-3-8B token's activations, 7-bit SiLU, N = 8192
        {"name": "pbs_llama_silu", "kind": "pbs", "set": "llama_silu", "batch": 1024},
        # four nonlinear layers in one launch at the paper's dimensions,
        # ciphertexts coming from and going back to pinned host memory
        {"name": "pbs_luts_host", "kind": "multi_lut", "set": "paper_dims", "batch": 1000, "luts": 4, "host": True},
        # the key switch alone, full batch
        {"name": "keyswitch", "kind": "keyswitch", "set": "standard", "batch": 4096},
        # the key switch alone, a few extracted ciphertexts
        {"name": "keyswitch_few", "kind": "keyswitch", "set": "gpt2_mlp", "batch": 61},
        # RLWE traces as the lookup runs them
        {"name": "trace", "kind": "trace", "set": "standard", "batch": 1024},
        # the lookup's linear mapping p(X) [[x]] + q(X) with a plaintext on the host
        {"name": "plaintext_mul", "kind": "plaintext_mul", "set": "standard", "batch": 512},
        # the encrypted segmented lookup, four segments
        {"name": "lookup", "kind": "lookup", "set": "standard", "batch": 256, "segments": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# sets with a ring of N <= 4096, where the trace and the plaintext product exist
_SMALL_RINGS = ("tiny", "lookup_small", "standard", "paper_dims", "gpt2_mlp")
# LWE dimensions around the sets' own, by ring size
_DIMS = {256: (48, 96), 512: (48, 128), 2048: (600, 1024), 4096: (700, 960), 8192: (800, 960)}
# largest drawn batches: no drawn case costs more than the largest listed one
_MOST = {"tiny": 65536, "lookup_small": 16384, "standard": 6000, "exp_sweep": 6000, "paper_dims": 4096,
         "gpt2_mlp": 2800, "llama_silu": 900}


def draw(rng):
    kind = rng.choice(["pbs", "pbs", "pbs", "pbs", "noalloc", "multi_lut", "extract", "glwe", "keyswitch", "keyswitch",
                       "trace", "plaintext_mul", "lookup"])
    if kind in ("trace", "plaintext_mul"):
        name = rng.choice(_SMALL_RINGS)
        return {"kind": kind, "set": name, "batch": _log_int(rng, 1, 2048)}
    if kind == "lookup":
        name = rng.choice(("lookup_small", "standard", "paper_dims"))
        return {"kind": kind, "set": name, "batch": _log_int(rng, 1, 400), "segments": rng.choice((2, 4, 8))}
    name = rng.choice(sorted(_MOST))
    p = W.CONFIGS[name]
    c = {"kind": kind, "set": name}
    if rng.random() < 0.5:
        c["n"] = rng.randint(*_DIMS[p.N])
    n = c.get("n", p.n)
    most = int(_MOST[name] * min(1.0, p.n / n))
    if kind == "keyswitch":
        most = 4096
    elif kind == "noalloc":
        most = min(most, (2 << 20) // (p.N + 1))
    elif kind == "glwe":
        most = min(most, 2048)
    c["batch"] = _log_int(rng, 1, most)
    if kind == "multi_lut":
        c["luts"] = rng.randint(2, 16)
    if kind in ("pbs", "multi_lut", "extract", "keyswitch"):
        c["host"] = rng.random() < 0.25
    return c


def _params(case):
    p = W.CONFIGS[case["set"]]
    return dataclasses.replace(p, n=case["n"]) if "n" in case else p


def _words(g, *shape):
    """Uniform 64-bit words on the GPU (as int64)."""
    return torch.randint(-(1 << 63), (1 << 63) - 1, shape, dtype=torch.int64, device="cuda", generator=g)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _table(case, p, rng):
    """A 1/x table on [0.1, 2] with seeded inner boundaries, encoded for ring p.N."""
    segs = case.get("segments", 4)
    inner = np.sort(rng.uniform(0.15, 1.9, size=segs - 1))
    tau = [0.1] + [float(v) + 1e-3 * i for i, v in enumerate(inner)] + [2.0]
    return SG.encode(SG.build(SG.FUNCTIONS["reciprocal"], tau, min(64, p.N // 2)), p.N, DX, DR)


def _inputs(case, seed):
    """Everything a call takes besides the context, the keys among it."""
    p, kind, b = _params(case), case["kind"], case["batch"]
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 17)
    rng = np.random.default_rng([seed, 5])
    s = {"p": p, "kind": kind}
    # ciphertexts and keys are indistinguishable from uniform words, and the
    # path's cost does not depend on them
    if kind not in ("keyswitch", "trace", "plaintext_mul"):
        s["bsk"] = _words(g, *p.bsk_shape())
    if kind not in ("extract", "glwe", "trace", "plaintext_mul"):
        s["ksk"] = _words(g, *p.ksk_shape())
    if kind in ("trace", "lookup"):
        s["trace_keys"] = _words(g, p.N.bit_length() - 1, TRACE_LEVEL, 2, p.N)
    if kind in ("plaintext_mul", "lookup"):
        s["table"] = _table(case, p, rng)
    if kind in ("pbs", "noalloc", "multi_lut", "extract", "glwe", "lookup"):
        s["lwe"] = _words(g, b, p.n + 1)
    if kind == "keyswitch":
        s["lwe"] = _words(g, b, p.kN + 1)
    if kind in ("glwe", "trace", "plaintext_mul", "lookup"):
        s["glwe"] = _words(g, b, 2, p.N)
    if kind in ("pbs", "noalloc", "extract"):
        s["lut"] = _dev(W.lut_torus(p, np.roll(W.lut_codes(p), seed % 7)))
    if kind == "multi_lut":
        codes = W.lut_codes(p)
        s["luts"] = _dev(np.stack([W.lut_torus(p, np.roll(codes, r + seed % 5)) for r in range(case["luts"])]))
        s["index"] = torch.from_numpy(rng.integers(0, case["luts"], size=b).astype(np.int32)).cuda()
    if kind == "extract":
        shape = (b, p.kN + 1)
    elif kind in ("glwe", "trace", "plaintext_mul", "lookup"):
        shape = (b, 2, p.N)
    else:
        shape = (b, p.n + 1)
    s["out"] = torch.zeros(shape, dtype=torch.int64, device="cuda")
    if case.get("host"):
        s["lwe"] = s["lwe"].cpu().pin_memory()
        s["out"] = torch.zeros(shape, dtype=torch.int64).pin_memory()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    ctx = R.Context(s["p"])
    if "bsk" in s:
        ctx.upload_bsk(s.pop("bsk"))
    if "ksk" in s:
        ctx.upload_ksk(s.pop("ksk"))
    if "trace_keys" in s:
        ctx.upload_trace_keys(s.pop("trace_keys"), TRACE_BASE_LOG, TRACE_LEVEL)
    if s["kind"] == "lookup":
        e = s.pop("table")
        ctx.upload_lookup_table(e.p_hat, e.q_hat, e.a_hat, e.b_hat)
    ctx.sync_status()
    s["ctx"] = ctx
    return s


def run(s):
    ctx, kind, out = s["ctx"], s["kind"], s["out"]
    if kind == "pbs":
        return ctx.pbs_batch(s["lwe"], s["lut"], out)
    if kind == "noalloc":
        return ctx.rosetta_pbs_batch_noalloc(s["lwe"], s["lut"], out)
    if kind == "multi_lut":
        return ctx.pbs_batch_multi_lut(s["lwe"], s["luts"], s["index"], out)
    if kind == "extract":
        return ctx.blind_rotate_extract_batch(s["lwe"], s["lut"], out)
    if kind == "glwe":
        return ctx.blind_rotate_glwe_batch(s["lwe"], s["glwe"], out)
    if kind == "keyswitch":
        return ctx.keyswitch_batch(s["lwe"], out)
    if kind == "trace":
        return ctx.trace_batch(s["glwe"], out)
    if kind == "plaintext_mul":
        return ctx.plaintext_mul_batch(s["glwe"], s["table"].p_hat, out, s["table"].q_hat)
    return ctx.segmented_lookup_batch(s["glwe"], s["lwe"], out)


# ---------------------------------------------------------------- what a pass cannot do without


def _transforms(N, bits, forward, inverse, products):
    """32-bit operations of one exact negacyclic sum of products over as few
    31-bit primes as `bits` needs: butterflies 8 each, products 6, CRT 10 a
    prime and output coefficient."""
    primes = math.ceil(bits / 31)
    return primes * ((forward + inverse) * (N // 2) * int(math.log2(N)) * 8 + products * N * 6 + inverse * N * 10)


def _rotation_ops(p):
    bits = 63 + p.pbs_base_log + math.log2(2 * p.pbs_level * p.N)
    step = _transforms(p.N, bits, 2 * p.pbs_level, 2, 4 * p.pbs_level) + 2 * p.N * (6 * p.pbs_level + 4)
    return step * p.n


def _keyswitch_ops(p):
    return p.kN * p.ks_level * ((p.n + 1) * 3 + 6)


def _trace_ops(p):
    bits = 63 + TRACE_BASE_LOG + math.log2(TRACE_LEVEL * p.N)
    return int(math.log2(p.N)) * (_transforms(p.N, bits, TRACE_LEVEL, 2, 2 * TRACE_LEVEL) + p.N * (6 * TRACE_LEVEL + 4))


def _product_ops(p):
    return _transforms(p.N, 128 + math.log2(p.N), 2, 2, 2)


def work(case):
    p, kind, b = _params(case), case["kind"], case["batch"]
    bsk, ksk = 8 * math.prod(p.bsk_shape()), 8 * math.prod(p.ksk_shape())
    trk = 8 * int(math.log2(p.N)) * TRACE_LEVEL * 2 * p.N
    lwe, big, glwe = 8 * (p.n + 1), 8 * (p.kN + 1), 16 * p.N
    if kind in ("pbs", "noalloc", "multi_lut"):
        lut = case.get("luts", 1) * (8 << p.msg_bits)
        return {"bytes": bsk + ksk + lut + b * 2 * lwe, "flops": b * (_rotation_ops(p) + _keyswitch_ops(p))}
    if kind == "extract":
        return {"bytes": bsk + (8 << p.msg_bits) + b * (lwe + big), "flops": b * _rotation_ops(p)}
    if kind == "glwe":
        return {"bytes": bsk + b * (lwe + 2 * glwe), "flops": b * _rotation_ops(p)}
    if kind == "keyswitch":
        return {"bytes": ksk + b * (big + lwe), "flops": b * _keyswitch_ops(p)}
    if kind == "trace":
        return {"bytes": trk + b * 2 * glwe, "flops": b * _trace_ops(p)}
    if kind == "plaintext_mul":
        return {"bytes": 16 * p.N + b * 2 * glwe, "flops": b * _product_ops(p)}
    k = case["segments"]
    ops = (k + 2) * (_rotation_ops(p) + _product_ops(p)) + _keyswitch_ops(p) + (k + 1) * _trace_ops(p)
    return {"bytes": bsk + ksk + trk + 16 * (k + 1) * p.N + b * (2 * glwe + lwe), "flops": b * ops}


# ---------------------------------------------------------------- the same words by definition


def _digits(v, base_log, level):
    """Signed gadget digits (int64 [level, ...], most significant first) of uint64 words."""
    bits = base_log * level
    v = v.copy()
    if bits < 64:
        v = (v + np.uint64(1 << (63 - bits))) >> np.uint64(64 - bits)
    out = np.empty((level,) + v.shape, np.int64)
    mask, half = np.uint64((1 << base_log) - 1), np.uint64(1 << (base_log - 1))
    for lev in range(level - 1, -1, -1):
        d = v & mask
        up = d >= half
        v = (v >> np.uint64(base_log)) + up.astype(np.uint64)
        out[lev] = d.astype(np.int64) - (up.astype(np.int64) << base_log)
    return out


def _limbs(words):
    """uint64 words as four 16-bit limbs in float64, least significant first."""
    return [torch.from_numpy(((words >> np.uint64(16 * i)) & np.uint64(0xFFFF)).astype(np.float64)) for i in range(4)]


def _matmul(a, b):
    """a @ b mod 2^64 from 16-bit limbs (a list of at most four, or one matrix
    of small signed integers as one limb) of both: every float64 sum is an
    integer below 2^53."""
    out = np.zeros((a[0].shape[0], b[0].shape[1]), np.uint64)
    for i, x in enumerate(a):
        for j, y in enumerate(b[:4 - i]):
            out += (x @ y).to(torch.int64).numpy().view(np.uint64) << np.uint64(16 * (i + j))
    return out


def _negacyclic(poly):
    """[N, N] matrix T with (row @ T) = row * poly mod X^N + 1."""
    n = poly.shape[-1]
    j, t = np.arange(n)[None, :], np.arange(n)[:, None]
    m = poly[(j - t) % n]
    return np.where(j >= t, m, np.uint64(0) - m)


def _rotate(a, e):
    """X^e a for uint64 polynomials a [..., N], 0 <= e < 2N."""
    n = a.shape[-1]
    idx = (np.arange(n) - e) % (2 * n)
    v = a[..., idx % n]
    return np.where(idx >= n, np.uint64(0) - v, v)


def _key_switch(p, ksk, big):
    d = _digits(big[:, :p.kN], p.ks_base_log, p.ks_level).transpose(1, 2, 0).reshape(big.shape[0], -1)
    out = np.uint64(0) - _matmul([torch.from_numpy(d.astype(np.float64))], _limbs(ksk.reshape(-1, p.n + 1)))
    out[:, p.n] += big[:, p.kN]
    return out


def _pbs_words(p, s):
    host = {k: s[k].cpu().numpy().view(np.uint64) for k in ("lwe", "lut", "bsk", "ksk")}
    N, box = p.N, p.N >> p.msg_bits
    t, h = np.arange(N), (p.N >> p.msg_bits) // 2
    test = np.where(t < N - h, host["lut"][np.minimum((t + h) // box, (1 << p.msg_bits) - 1)],
                    np.uint64(0) - host["lut"][0])
    sh = 64 - (2 * N).bit_length() + 1
    sw = ((host["lwe"] + np.uint64(1 << (sh - 1))) >> np.uint64(sh)).astype(np.int64) % (2 * N)
    b = host["lwe"].shape[0]
    acc = np.zeros((b, 2, N), np.uint64)
    for c in range(b):
        acc[c, 1] = _rotate(test, (2 * N - int(sw[c, p.n])) % (2 * N))
    for i in range(p.n):
        diff = np.stack([_rotate(acc[c], int(sw[c, i])) - acc[c] for c in range(b)])
        d = _digits(diff, p.pbs_base_log, p.pbs_level)                     # [l, b, 2, N]
        for j in range(2):
            for lev in range(p.pbs_level):
                for comp in range(2):
                    key = host["bsk"][i, j * p.pbs_level + lev, comp]
                    acc[:, comp] += d[lev, :, j].copy().view(np.uint64) @ _negacyclic(key)
    big = np.empty((b, N + 1), np.uint64)
    big[:, 0] = acc[:, 0, 0]
    big[:, 1:N] = np.uint64(0) - acc[:, 0, :0:-1]
    big[:, N] = acc[:, 1, 0]
    return _key_switch(p, host["ksk"], big)


def exact(case, seed):
    """The words themselves, by the plain definition, where that is quick."""
    p, kind, b = _params(case), case["kind"], case["batch"]
    if kind == "pbs" and p.N <= 256 and b * p.n <= 1024:
        words = _pbs_words(p, _inputs(case, seed))
    elif kind == "keyswitch" and b * p.kN * p.ks_level * (p.n + 1) <= 1 << 35:
        s = _inputs(case, seed)
        words = _key_switch(p, s["ksk"].cpu().numpy().view(np.uint64), s["lwe"].cpu().numpy().view(np.uint64))
    elif kind == "plaintext_mul" and b * p.N * p.N <= 1 << 31:
        s = _inputs(case, seed)
        glwe = s["glwe"].cpu().numpy().view(np.uint64).reshape(2 * b, p.N)
        words = _matmul(_limbs(glwe), _limbs(_negacyclic(s["table"].p_hat.view(np.uint64)))).reshape(b, 2, p.N)
        words[:, 1] += s["table"].q_hat
    else:
        return None
    return torch.from_numpy(words.view(np.int64))
