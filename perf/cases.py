"""The work that a program built on this library has it do, as cases that can be timed.

An RL trainer drives the library through `paper_2609_35140_b200.binding`: rollout decodes token by
token against a paged KV cache and scores the sampled tokens, prompts are prefilled into the same
cache, and the policy update runs attention forward and backward over packed sequences, the FFN and
the token log-probabilities over whole batches.  Model shapes are those of the package's workloads
(`synth.get_workload`) with the FFN widths that `bench.py` uses.  Sequence lengths belong to a case
(drawn from its own `lengths` number); tensors and page placement come from the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2609_35140_b200 import binding as tik
from paper_2609_35140_b200 import synth

BF = torch.bfloat16

# query heads, KV heads, head dim, hidden, FFN intermediate, vocabulary
MODELS = {
    "tiny": (4, 1, 64, 256, 704, 2048),
    "1.5B": (12, 2, 128, 1536, 8960, 151936),
    "7B": (28, 4, 128, 3584, 18944, 152064),
    "long": (32, 8, 128, 4096, 12288, 151936),
    "32B": (64, 8, 128, 5120, 27648, 151936),
}
EPS = 1e-6


def listed():
    return [
        # one interactive rollout, or the last unfinished response of a batch: latency only
        {"name": "decode_single", "kind": "decode", "model": "7B", "seqs": 1, "lo": 4321, "hi": 4321, "page": 64,
         "group": 1, "shared": 0, "lengths": 1},
        # GRPO rollout: 8 prompts x 8 responses that share their prompt's pages, at ragged lengths
        {"name": "decode_grpo", "kind": "decode", "model": "7B", "seqs": 64, "lo": 1280, "hi": 5120, "page": 64,
         "group": 8, "shared": 1024, "lengths": 2},
        # long-context rollout: the cache is read once and does not fit L2
        {"name": "decode_long", "kind": "decode", "model": "long", "seqs": 16, "lo": 15000, "hi": 16384, "page": 64,
         "group": 1, "shared": 0, "lengths": 3},
        # one prompt into an empty cache: time to first token
        {"name": "prefill_single", "kind": "prefill", "model": "7B", "seqs": 1, "lo": 1000, "hi": 1000, "prefix": 0,
         "page": 64, "lengths": 4},
        # a batch of prompts, half of them behind a cached prefix (chunked prefill, multi-turn)
        {"name": "prefill_batch", "kind": "prefill", "model": "32B", "seqs": 32, "lo": 300, "hi": 1700, "prefix": 3000,
         "page": 64, "lengths": 5},
        # the smallest update step: two short sequences, head dim 64
        {"name": "train_tiny", "kind": "train", "model": "tiny", "seqs": 2, "lo": 96, "hi": 160, "lengths": 6},
        # a micro-batch of GRPO responses through attention forward and backward
        {"name": "train_grpo", "kind": "train", "model": "7B", "seqs": 16, "lo": 1280, "hi": 5120, "lengths": 7},
        # long-context update: one full-length and one shorter sequence
        {"name": "train_long", "kind": "train", "model": "long", "seqs": 2, "lo": 9001, "hi": 16384, "lengths": 8},
        # one decoder layer of a small model's rollout step
        {"name": "rollout_layer_small", "kind": "layer", "model": "1.5B", "seqs": 16, "lo": 640, "hi": 2560, "page": 64,
         "head": False, "lengths": 9},
        # a rollout step's last decoder layer, final norm and log-probs of the sampled tokens
        {"name": "rollout_layer_head", "kind": "layer", "model": "7B", "seqs": 64, "lo": 1280, "hi": 5120, "page": 64,
         "head": True, "lengths": 10},
        # the FFN half of a layer over an update micro-batch of odd size
        {"name": "update_ffn", "kind": "ffn", "model": "7B", "rows": 5999},
        # policy update: log-probs of a micro-batch's response tokens, sampled at temperature 0.7
        {"name": "update_logprob", "kind": "logprob", "model": "7B", "rows": 4001, "temperature": 0.7},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.6e15)


def _draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "train", "train", "layer", "ffn", "logprob"])
    c = {"kind": kind, "model": rng.choice(["1.5B", "7B", "long", "32B"])}
    if kind in ("decode", "prefill", "train") and rng.random() < 0.15:
        c["model"] = "tiny"
    if kind in ("ffn", "logprob"):
        c["rows"] = _log_uniform(rng, 1, 16384)
        if kind == "logprob":
            c["temperature"] = rng.choice([1.0, 0.7])
        return c
    c["lengths"] = rng.randrange(1 << 20)
    if kind == "train":
        c["seqs"], c["hi"] = _log_uniform(rng, 1, 64), _log_uniform(rng, 48, 16384)
    elif kind == "prefill":
        c["seqs"], c["hi"] = _log_uniform(rng, 1, 64), _log_uniform(rng, 16, 8192)
        c["prefix"] = rng.choice([0, _log_uniform(rng, 16, 8192)])
    else:
        c["seqs"], c["hi"] = _log_uniform(rng, 1, 256), _log_uniform(rng, 64, 16384)
    c["lo"] = max(1, int(c["hi"] * rng.uniform(0.1, 1.0)))
    if kind != "train":
        c["page"] = rng.choice([16, 32, 64, 64, 64, 128])
    if kind == "decode":
        c["group"] = rng.choice([1, 1, 8])
        c["shared"] = int(c["lo"] * rng.uniform(0.1, 1.0)) if c["group"] > 1 else 0
    if kind == "layer":
        c["head"] = rng.random() < 0.3
    return c


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def _lengths(case):
    """Per-sequence lengths: new tokens (prefill), whole sequences (train) or contexts (decode, layer)."""
    r = random.Random(case["lengths"])
    n, lo, hi = case["seqs"], case["lo"], case["hi"]
    got = [r.randint(lo, hi) for _ in range(n)]
    got[r.randrange(n)] = hi
    if n == 2:
        got = [hi, lo]
    return got


def _prefixes(case):
    """Cached tokens before the new ones: none for half of the sequences, ragged for the others."""
    if not case["prefix"]:
        return [0] * case["seqs"]
    r = random.Random(case["lengths"] + 1)
    return [r.randint(1, case["prefix"]) if (i % 2 or case["seqs"] == 1) else 0 for i in range(case["seqs"])]


def _contexts(case):
    got = _lengths(case)
    return [n + p for n, p in zip(got, _prefixes(case))] if case["kind"] == "prefill" else got


def _unique_context_tokens(case):
    """Cached tokens a decode step has to read: whole shared prompt pages once per group."""
    ctx, page = _contexts(case), case["page"]
    shared = case.get("shared", 0) // page * page
    group = case.get("group", 1)
    return sum(ctx) - sum(shared * (len(ctx[i:i + group]) - 1) for i in range(0, len(ctx), group) if group > 1)


class _Tensors:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.seed = seed

    def normal(self, *shape, std=1.0, mean=0.0):
        out = torch.empty(shape, dtype=BF, device="cuda")
        step = max(1, (1 << 26) // max(1, math.prod(shape[1:])))
        for r in range(0, shape[0], step):
            part = torch.randn((min(step, shape[0] - r),) + shape[1:], generator=self.g, device="cuda")
            out[r:r + step] = part.mul_(std).add_(mean)
        return out

    def ids(self, n, below):
        return torch.randint(0, below, (n,), generator=self.g, device="cuda").to(torch.int32)


def _i32(v):
    return torch.tensor(v, dtype=torch.int32, device="cuda")


def _cu(lens):
    return _i32([0] + [int(x) for x in np.cumsum(lens)])


def _cache(case, t):
    """A paged pool whose pages hold earlier tokens' keys and values, and a fragmented block table."""
    _, Hkv, d = MODELS[case["model"]][:3]
    ctx, page, group = _contexts(case), case["page"], case.get("group", 1)
    shared = case.get("shared", 0) // page
    blocks = [-(-c // page) for c in ctx]
    table = -np.ones((len(ctx), max(blocks)), dtype=np.int32)
    owner = [i // group * group for i in range(len(ctx))]
    need = sum(b - (shared if o != i else 0) for i, (b, o) in enumerate(zip(blocks, owner)))
    pages = np.random.default_rng(t.seed).permutation(need + 3)
    at = 0
    for i, (b, o) in enumerate(zip(blocks, owner)):
        own = 0 if o == i else shared
        table[i, :own] = table[o, :own]
        table[i, own:b] = pages[at:at + b - own]
        at += b - own
    kc, vc = (t.normal(need + 3, Hkv, page, d) for _ in range(2))
    return {"k_cache": kc, "v_cache": vc, "table": torch.from_numpy(table).cuda(), "ctx": _i32(ctx), "max_ctx": max(ctx)}


def prepare(case, seed):
    Hq, Hkv, d, H, inter, V = MODELS[case["model"]]
    t = _Tensors(seed)
    s = {"kind": case["kind"], "heads": (Hq, Hkv, d), "scale": float(np.float32(1.0 / math.sqrt(d)))}
    if case["kind"] == "decode":
        s.update(_cache(case, t), cu=_i32(range(case["seqs"] + 1)))
        s["q"], s["k"], s["v"] = (t.normal(case["seqs"], n, d) for n in (Hq, Hkv, Hkv))
    elif case["kind"] == "prefill":
        lens = _lengths(case)
        s.update(_cache(case, t), cu=_cu(lens), max_q=max(lens))
        s["q"], s["k"], s["v"] = (t.normal(sum(lens), n, d) for n in (Hq, Hkv, Hkv))
    elif case["kind"] == "train":
        lens = _lengths(case)
        s.update(cu=_cu(lens), max_q=max(lens))
        s["q"], s["k"], s["v"], s["d_o"] = (t.normal(sum(lens), n, d) for n in (Hq, Hkv, Hkv, Hq))
        s["lse"] = torch.empty(sum(lens), Hq, dtype=torch.float32, device="cuda")
    elif case["kind"] == "layer":
        s.update(_cache(case, t), cu=_i32(range(case["seqs"] + 1)), x=t.normal(case["seqs"], H))
        s["rope"] = synth.make_rope_table(s["max_ctx"], d, device="cuda")
        for name, n, k in (("wq", Hq * d, H), ("wk", Hkv * d, H), ("wv", Hkv * d, H), ("wo", H, Hq * d),
                           ("w_gate_up", 2 * inter, H), ("w_down", H, inter)):
            s[name] = t.normal(n, k, std=0.02)
        for name, n in (("norm1", H), ("norm2", H), ("norm_q", d), ("norm_k", d)):
            s[name] = t.normal(n, std=0.2, mean=1.0)
        s["head"] = None
        if case["head"]:
            s.update(head=t.normal(V, H, std=0.02), norm_f=t.normal(H, std=0.2, mean=1.0), ids=t.ids(case["seqs"], V))
    elif case["kind"] == "ffn":
        s.update(x=t.normal(case["rows"], H), norm2=t.normal(H, std=0.2, mean=1.0),
                 w_gate_up=t.normal(2 * inter, H, std=0.02), w_down=t.normal(H, inter, std=0.02))
    else:
        s.update(x=t.normal(case["rows"], H), head=t.normal(V, H, std=0.02), ids=t.ids(case["rows"], V),
                 inv_temperature=1.0 / case["temperature"])
    return s


def _ffn(h, s):
    return tik.tik_linear(tik.tik_swiglu(tik.tik_linear(h, s["w_gate_up"])), s["w_down"])


def _layer(s):
    Hq, Hkv, d = s["heads"]
    x, n = s["x"], s["x"].shape[0]
    h = tik.tik_rmsnorm(x, s["norm1"], EPS)
    q = tik.tik_linear(h, s["wq"]).view(n, Hq, d)
    k = tik.tik_linear(h, s["wk"]).view(n, Hkv, d)
    v = tik.tik_linear(h, s["wv"]).view(n, Hkv, d)
    tik.tik_qk_norm_rope_kv_write(q, k, v, s["norm_q"], s["norm_k"], EPS, s["rope"], s["cu"], s["ctx"], s["k_cache"],
                                  s["v_cache"], s["table"])
    o = tik.tik_attn_decode(q, s["ctx"], s["k_cache"], s["v_cache"], s["table"], s["max_ctx"], s["scale"])
    stream = tik.tik_linear(o.view(n, Hq * d), s["wo"])
    h = tik.tik_rmsnorm(x, s["norm2"], EPS, residual=stream)       # stream <- x + attention output
    y = _ffn(h, s)
    out = {"k_cache": s["k_cache"], "v_cache": s["v_cache"], "y": y, "stream": stream}
    if s["head"] is not None:
        h = tik.tik_rmsnorm(y, s["norm_f"], EPS, residual=stream)  # stream <- stream + FFN output
        out["logprob"] = tik.tik_token_logprob(h, s["head"], s["ids"])
    return out


def run(state):
    s = state
    if s["kind"] == "decode":
        tik.tik_kv_cache_write(s["k"], s["v"], s["cu"], s["ctx"], s["k_cache"], s["v_cache"], s["table"])
        o = tik.tik_attn_decode(s["q"], s["ctx"], s["k_cache"], s["v_cache"], s["table"], s["max_ctx"], s["scale"])
        return {"o": o, "k_cache": s["k_cache"], "v_cache": s["v_cache"]}
    if s["kind"] == "prefill":
        o = tik.tik_attn_prefill_kv(s["q"], s["k"], s["v"], s["cu"], s["ctx"], s["k_cache"], s["v_cache"], s["table"],
                                    s["max_q"], s["max_ctx"], s["scale"])
        return {"o": o, "k_cache": s["k_cache"], "v_cache": s["v_cache"]}
    if s["kind"] == "train":
        o = tik.tik_attn_train_fwd(s["q"], s["k"], s["v"], s["cu"], s["max_q"], s["scale"], lse=s["lse"])
        dq, dk, dv = tik.tik_attn_train_bwd(s["q"], s["k"], s["v"], o, s["d_o"], s["lse"], s["cu"], s["max_q"], s["scale"])
        return {"o": o, "lse": s["lse"], "dq": dq, "dk": dk, "dv": dv}
    if s["kind"] == "layer":
        return _layer(s)
    if s["kind"] == "ffn":
        h = tik.tik_rmsnorm(s["x"], s["norm2"], EPS)
        return {"h": h, "y": _ffn(h, s)}
    return tik.tik_token_logprob(s["x"], s["head"], s["ids"], s["inv_temperature"])


def work(case):
    Hq, Hkv, d, H, inter, V = MODELS[case["model"]]
    kind = case["kind"]
    if kind == "ffn":
        T = case["rows"]
        return {"bytes": 2.0 * (3 * T * H + 3 * inter * H), "flops": 6.0 * T * H * inter}
    if kind == "logprob":
        T = case["rows"]
        return {"bytes": 2.0 * (T * H + V * H) + 8.0 * T, "flops": 2.0 * T * H * V}
    lens, ctx = _lengths(case), _contexts(case) if kind != "train" else None
    if kind == "train":
        tok, pairs = sum(lens), sum(n * (n + 1) // 2 for n in lens)
        # q, o, d_o, dq and k, v, dk, dv once each, lse written; 2 + 5 products over the causal pairs
        return {"bytes": tok * (8.0 * Hq * d + 8.0 * Hkv * d + 4.0 * Hq), "flops": 14.0 * d * Hq * pairs}
    if kind == "prefill":
        pairs = sum(n * (c - n) + n * (n + 1) // 2 for n, c in zip(lens, ctx))
        return {"bytes": sum(lens) * (4.0 * Hq * d + 8.0 * Hkv * d) + sum(c - n for n, c in zip(lens, ctx)) * 4.0 * Hkv * d,
                "flops": 4.0 * d * Hq * pairs}
    n = case["seqs"]
    read = _unique_context_tokens(case) * 4.0 * Hkv * d
    flops = 4.0 * d * Hq * sum(ctx)
    if kind == "decode":
        return {"bytes": read + n * (4.0 * Hq * d + 8.0 * Hkv * d), "flops": flops}
    weights = H * (2 * Hq + 2 * Hkv) * d + 3 * H * inter + (V * H if case["head"] else 0)
    return {"bytes": read + 2.0 * weights + n * (6.0 * H + 4.0 * Hkv * d), "flops": flops + 2.0 * n * weights}


def tolerance(case):
    """About four times the error measured against the same path in fp64 (no roundings in between):
    attention outputs 2.0e-3 .. 2.4e-3, gradients 2.2e-3 .. 2.6e-3 (bf16 weights and results), a layer's
    outputs 4.9e-3 and the FFN's 4.3e-3 (bf16 at every operator), fp32 log-probabilities 9e-7."""
    return {"rel": {"decode": 1e-2, "prefill": 1e-2, "train": 1e-2, "layer": 2e-2, "ffn": 1.7e-2, "logprob": 4e-6}[case["kind"]]}
