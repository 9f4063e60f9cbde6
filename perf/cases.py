"""The work a serving program has this library do, as cases that can be timed: decode steps, chunked prefill, steps that
mix both, quantize-append and cache exchange, from a call of a few microseconds to tens of milliseconds.

A case is a dict of plain values; `prepare` builds on the GPU what a program holds before the call (the Q4 pool filled
through the library's own quantizer, block tables, lengths, new rows, workspace), `run` makes the calls of one pass and
returns what they write.  Lengths follow from the case alone, values and block placement from the seed.
"""
import math
import random

import torch

from paper_2603_04428_b200 import binding as B
from paper_2603_04428_b200 import synth

BLOCK = synth.BLOCK_TOKENS

DEFAULTS = {
    "op": "decode",        # decode | prefill | append | exchange
    "layers": 1, "q_heads": 32, "kv_heads": 8, "d_qk": 128, "d_v": 128, "latent": False,
    "agents": 1,           # agents with `chunk` new tokens each (a decode step: one)
    "cached_lo": 1024, "cached_hi": 1024,   # cached tokens per agent before the step, log-uniform in between
    "chunk_lo": 1, "chunk_hi": 1,           # new tokens per agent
    "decoding": 0,         # further agents of a prefill step that bring one token each
    "lens_seed": 0,
    "window": 0, "global_every": 0,         # sliding window; layer l is global iff (l + 1) % global_every == 0
    "fused": True,         # decode: update-and-fetch in one call (else append, then decode attention)
    "sb_bf16": False,      # bfloat16 scales and biases (else binary16)
    "exact": False,        # spec.exact_products
    "out_bf16": False,
    "outliers": False,     # 1 % of the channels carry 8x the values
}


def listed():
    return [
        # One layer of a two-agent batch: the smallest call, all launch and host latency.
        dict(name="decode_tiny", op="decode", layers=1, q_heads=8, kv_heads=2, agents=2, cached_lo=700, cached_hi=1000),
        # A Llama-3.1-8B-shaped decode step, all layers, five agents at 4096 tokens: the benchmark's own step.
        dict(name="decode_step", op="decode", layers=32, agents=5, cached_lo=4096, cached_hi=4096, outliers=True),
        # A Gemma-3-12B-shaped decode step over very ragged agents: five window layers to each global one, two periods.
        dict(name="decode_ragged_window", op="decode", layers=12, q_heads=16, kv_heads=8, d_qk=256, d_v=256, agents=10,
             cached_lo=1024, cached_hi=32768, lens_seed=3, window=1024, global_every=6, out_bf16=True),
        # Eight query heads to a KV head (a large GQA model), bfloat16 scales: append, then attend.
        dict(name="decode_gqa8", op="decode", layers=4, q_heads=64, kv_heads=8, agents=12, cached_lo=1000, cached_hi=12000,
             lens_seed=4, fused=False, sb_bf16=True, out_bf16=True),
        # A DeepSeek-Coder-V2-Lite-shaped step on the shared latent cache, four agents at 16384 tokens, all layers.
        dict(name="decode_latent", op="decode", layers=27, q_heads=16, kv_heads=1, d_qk=576, d_v=512, latent=True, agents=4,
             cached_lo=16384, cached_hi=16384),
        # Cross-phase context injection: eight agents put 1024 new tokens each on an 8192-token prefix.
        dict(name="prefill_inject", op="prefill", layers=4, agents=8, cached_lo=8192, cached_hi=8192, chunk_lo=1024,
             chunk_hi=1024),
        # A ragged phase at head dimension 256, window layers and a global one.
        dict(name="prefill_window_d256", op="prefill", layers=6, q_heads=16, kv_heads=8, d_qk=256, d_v=256, agents=6,
             cached_lo=1500, cached_hi=8000, lens_seed=7, chunk_lo=200, chunk_hi=700, window=1024, global_every=6,
             out_bf16=True),
        # One agent's 512-token scheduler chunk on a long context: what a single user waits for.
        dict(name="prefill_one_agent", op="prefill", layers=8, agents=1, cached_lo=15873, cached_hi=15873, chunk_lo=512,
             chunk_hi=512, out_bf16=True),
        # A chunk on the shared latent cache (absorbed form).
        dict(name="prefill_latent", op="prefill", layers=2, q_heads=16, kv_heads=1, d_qk=576, d_v=512, latent=True, agents=3,
             cached_lo=2000, cached_hi=4000, lens_seed=9, chunk_lo=250, chunk_hi=512),
        # A scheduler step: two agents' 512-token chunks interleaved with ten agents that decode one token each.
        dict(name="step_mixed", op="prefill", layers=8, agents=2, cached_lo=1024, cached_hi=6000, lens_seed=10, chunk_lo=512,
             chunk_hi=512, decoding=10, out_bf16=True),
        # Quantizing a phase of bf16 rows into the pool, all layers.
        dict(name="append_phase", op="append", layers=32, agents=8, cached_lo=1024, cached_hi=1024, chunk_lo=1024,
             chunk_hi=1024),
        # An agent leaves the pool in the persisted layout and its image comes back into other blocks.
        dict(name="exchange_agent", op="exchange", layers=32, agents=1, cached_lo=4000, cached_hi=4000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["decode", "decode", "decode", "gqa8", "latent", "prefill", "prefill", "prefill", "prefill_latent",
                         "mixed", "append", "exchange"])
    c = {"lens_seed": rng.randrange(1 << 20), "out_bf16": rng.random() < 0.5, "sb_bf16": rng.random() < 0.3}
    gqa = [(8, 2, 128, 128), (32, 8, 128, 128), (16, 16, 128, 128), (16, 8, 256, 256), (16, 16, 192, 128)]
    if family in ("decode", "gqa8", "latent"):
        hi = _log(rng, 400, 32768)
        c.update(op="decode", agents=_log(rng, 1, 16), cached_hi=hi, cached_lo=max(50, hi // rng.choice([1, 3, 30])))
        if family == "decode":
            hq, hkv, d, dv = rng.choice(gqa)
            c["outliers"] = d == 128 and rng.random() < 0.5
            if rng.random() < (0.7 if d == 256 else 0.15):
                c.update(window=rng.choice([512, 1024, 4096]), global_every=rng.choice([0, 6]))
        elif family == "gqa8":
            hkv, rep = rng.choice([2, 4, 8]), rng.choice([5, 6, 8, 8, 16])
            hq, d, dv = hkv * rep, 128, 128
            c.update(fused=False, cached_hi=min(hi, 12000), cached_lo=min(c["cached_lo"], 12000))
        else:
            hq, hkv, d, dv = rng.choice([8, 16, 16]), 1, 576, 512
            c.update(latent=True, exact=rng.random() < 0.25)
        c.update(q_heads=hq, kv_heads=hkv, d_qk=d, d_v=dv)
        most = max(1, (1500 << 20) // max(1, sum(_lens(dict(DEFAULTS, **c))[0]) * _row_bytes(dict(DEFAULTS, **c))))
        c["layers"] = min(_log(rng, 1, 32 if family != "gqa8" else 4), most)
        return c
    if family in ("prefill", "prefill_latent", "mixed"):
        hi = _log(rng, 100, 16384)
        top = _log(rng, 33, 1024)
        c.update(op="prefill", agents=_log(rng, 1, 8), cached_hi=hi, cached_lo=max(1, hi // rng.choice([1, 3, 30])),
                 chunk_hi=top, chunk_lo=max(1, top // rng.choice([1, 3])))
        if family == "prefill_latent":
            hq, hkv, d, dv = 16, 1, 576, 512
            c.update(latent=True, agents=_log(rng, 1, 3), cached_hi=min(hi, 4000), cached_lo=min(c["cached_lo"], 4000),
                     chunk_hi=min(top, 512), chunk_lo=min(c["chunk_lo"], 512))
        else:
            hq, hkv, d, dv = rng.choice(gqa[:4] if family == "mixed" else gqa + [(64, 8, 128, 128)])
            if d == 256 and rng.random() < 0.7:
                c.update(window=1024, global_every=6)
            if family == "mixed":
                c.update(agents=rng.choice([1, 2, 3]), chunk_lo=min(c["chunk_lo"], 512), chunk_hi=min(top, 512),
                         decoding=_log(rng, 1, 24))
        c.update(q_heads=hq, kv_heads=hkv, d_qk=d, d_v=dv, layers=1)
        limit = 2e11 if family == "prefill_latent" or hq == 64 else 4e12
        while work(c)["flops"] > limit:
            c["chunk_hi"] = max(1, c["chunk_hi"] // 2)
            c["chunk_lo"] = min(c["chunk_lo"], c["chunk_hi"])
        c["layers"] = max(1, min(_log(rng, 1, 8), int(limit / work(c)["flops"])))
        return c
    hq, hkv, d, dv = rng.choice(gqa + [(16, 1, 576, 512)])
    c.update(q_heads=hq, kv_heads=hkv, d_qk=d, d_v=dv, latent=d == 576)
    if family == "append":
        top = _log(rng, 32, 4096)
        c.update(op="append", agents=_log(rng, 1, 12), cached_lo=1, cached_hi=_log(rng, 2, 2048), chunk_hi=top,
                 chunk_lo=max(1, top // rng.choice([1, 2, 8])))
    else:
        n = _log(rng, 100, 16384)
        c.update(op="exchange", agents=1, cached_lo=n, cached_hi=n)
    new = sum(sum(x) for x in _lens(dict(DEFAULTS, **c)))
    c["layers"] = max(1, min(_log(rng, 1, 32), (600 << 20) // (new * _row_bytes(dict(DEFAULTS, **c)))))
    return c


# ---- sizes -------------------------------------------------------------------------------------------------------------

def _full(case):
    return dict(DEFAULTS, **case)


def _lens(c):
    """(cached tokens, new tokens) of every agent of the step."""
    r = random.Random(c["lens_seed"])
    n = c["agents"] + c["decoding"]
    cached = [min(c["cached_hi"], max(c["cached_lo"], _log(r, c["cached_lo"], c["cached_hi"]))) for _ in range(n)]
    if c["op"] == "exchange":
        return cached, [0] * n
    new = [min(c["chunk_hi"], max(c["chunk_lo"], _log(r, c["chunk_lo"], c["chunk_hi"]))) for _ in range(c["agents"])]
    new += [1] * c["decoding"]
    if c["decoding"]:
        order = list(range(n))
        r.shuffle(order)
        cached, new = [cached[i] for i in order], [new[i] for i in order]
    return cached, new


def _row_bytes(c):
    """Q4 bytes of one token of one layer, all KV heads: codes, and a 16-bit scale and bias per group of 64."""
    k = c["d_qk"] // 2 + c["d_qk"] // 16
    v = 0 if c["latent"] else c["d_v"] // 2 + c["d_v"] // 16
    return c["kv_heads"] * (k + v)


def _window(c, layer):
    if not c["window"] or (c["global_every"] and (layer + 1) % c["global_every"] == 0):
        return 0
    return c["window"]


def _scale(c):
    return 1.0 / math.sqrt(192 if c["latent"] else c["d_qk"])


def work(case):
    c = _full(case)
    cached, new = _lens(c)
    row = _row_bytes(c)
    if c["op"] == "exchange":
        return {"bytes": 4.0 * c["layers"] * cached[0] * row, "flops": 0.0}
    rows_in = 2 * c["kv_heads"] * (c["d_qk"] + (0 if c["latent"] else c["d_v"]))
    moved = c["layers"] * sum(new) * (rows_in + row)
    if c["op"] == "append":
        return {"bytes": float(moved), "flops": 0.0}
    flops = 0.0
    moved += c["layers"] * sum(new) * c["q_heads"] * (2 * c["d_qk"] + (2 if c["out_bf16"] else 4) * c["d_v"])
    for layer in range(c["layers"]):
        w = _window(c, layer)
        for p, n in zip(cached, new):
            moved += (min(p, w + n - 1) if w else p) * row
            if w:
                short = min(n, max(0, w - p))     # queries that see everything before them
                pairs = short * p + short * (short + 1) / 2 + (n - short) * w
            else:
                pairs = n * p + n * (n + 1) / 2
            flops += 2.0 * c["q_heads"] * (c["d_qk"] + c["d_v"]) * pairs
    return {"bytes": float(moved), "flops": flops}


def tolerance(case):
    c = _full(case)
    if c["op"] in ("append", "exchange"):
        return "exact"
    if c["out_bf16"]:
        return {"rel": 5e-3}          # results rounded to bfloat16
    if c["exact"] or (c["op"] == "decode" and not c["latent"]):
        return {"rel": 1e-4}          # products of the 4-bit codes, 32-bit sums
    return {"rel": 2e-3}              # the spec lets keys and values be rounded to binary16


# ---- states ------------------------------------------------------------------------------------------------------------

class State:
    pass


def _normal(g, shape, channels=None):
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    if channels is not None:
        x.view(shape[0], -1)[:, channels] *= 8.0
    return x.to(torch.bfloat16)


def _ints(values):
    return torch.tensor(values, dtype=torch.int32).cuda()


def _offsets(counts):
    offs = [0]
    for n in counts:
        offs.append(offs[-1] + n)
    return offs


def prepare(case, seed):
    c = _full(case)
    s = State()
    s.c = c
    cached, new = _lens(c)
    n, layers = len(cached), c["layers"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s.spec = B.Spec.make(layers, c["q_heads"], c["kv_heads"], c["d_qk"], c["d_v"], c["latent"], c["exact"],
                         1 if c["sb_bf16"] else 0)
    blocks = [-(-(p + m) // BLOCK) for p, m in zip(cached, new)]
    s.n_blocks = sum(blocks) + 4
    s.tables = torch.from_numpy(synth.block_tables(seed, 99, [p + m for p, m in zip(cached, new)], s.n_blocks)).cuda()
    s.batch = B.batch(s.tables)
    s.pool = torch.zeros(B.q4kv_pool_bytes(s.spec, s.n_blocks), dtype=torch.uint8, device="cuda")
    s.flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    # the cached context, through the library's quantizer, a layer at a time
    zero, offs, total = _ints([0] * n), _ints(_offsets(cached)), sum(cached)
    for layer in range(layers):
        ko = vo = None
        if c["outliers"]:
            ko = torch.from_numpy(synth.outlier_channels(seed, 100 + layer, c["kv_heads"], c["d_qk"])).cuda()
            vo = torch.from_numpy(synth.outlier_channels(seed, 200 + layer, c["kv_heads"], c["d_v"])).cuda()
        k = _normal(g, (total, c["kv_heads"], c["d_qk"]), ko)
        v = None if c["latent"] else _normal(g, (total, c["kv_heads"], c["d_v"]), vo)
        B.q4kv_quantize_append(s.spec, s.pool, s.n_blocks, layer, s.batch, zero, offs, total, k, v, s.flags)
    if c["op"] == "exchange":
        s.tokens = cached[0]
        s.image = torch.empty(B.q4kv_packed_bytes(s.spec, s.tokens), dtype=torch.uint8, device="cuda")
        s.other = torch.zeros_like(s.pool)
        s.other_row = torch.from_numpy(synth.rng(seed, 97).permutation(s.n_blocks)[:blocks[0]].astype("int32")).cuda()
        return s
    total = sum(new)
    s.pos, s.lens, s.offs = _ints(cached), _ints([p + m for p, m in zip(cached, new)]), _ints(_offsets(new))
    s.total, s.most_new, s.most_kv = total, max(new), max(p + m for p, m in zip(cached, new))
    s.k = [_normal(g, (total, c["kv_heads"], c["d_qk"])) for _ in range(layers)]
    s.v = [None if c["latent"] else _normal(g, (total, c["kv_heads"], c["d_v"])) for _ in range(layers)]
    if c["op"] == "append":
        return s
    s.q = [_normal(g, (total, c["q_heads"], c["d_qk"])) for _ in range(layers)]
    s.out_dtype = B.OUT_BF16 if c["out_bf16"] else B.OUT_F32
    s.out = torch.zeros((layers, total, c["q_heads"], c["d_v"]), device="cuda",
                        dtype=torch.bfloat16 if c["out_bf16"] else torch.float32)
    s.outs = list(s.out)
    s.scale = _scale(c)
    s.windows = [_window(c, layer) for layer in range(layers)]
    s.ws = torch.zeros(B.q4kv_workspace_bytes(s.spec, n, s.most_kv, total if c["op"] == "prefill" else 0),
                       dtype=torch.uint8, device="cuda")
    return s


def run(s):
    c = s.c
    if c["op"] == "exchange":
        B.q4kv_pack(s.spec, s.pool, s.n_blocks, s.tables[0], s.tokens, s.image, s.flags)
        B.q4kv_unpack(s.spec, s.image, s.tokens, s.other, s.n_blocks, s.other_row, s.flags)
        return s.image, s.other, s.flags
    for layer in range(c["layers"]):
        if c["op"] == "decode" and c["fused"]:
            B.q4kv_append_decode_attention(s.spec, s.pool, s.n_blocks, layer, s.batch, s.lens, s.most_kv, s.windows[layer],
                                           s.k[layer], s.v[layer], s.q[layer], s.scale, s.outs[layer], s.out_dtype, None,
                                           s.ws, s.flags)
            continue
        B.q4kv_quantize_append(s.spec, s.pool, s.n_blocks, layer, s.batch, s.pos, s.offs, s.total, s.k[layer], s.v[layer],
                               s.flags)
        if c["op"] == "decode":
            B.q4kv_decode_attention(s.spec, s.pool, s.n_blocks, layer, s.batch, s.lens, s.most_kv, s.windows[layer],
                                    s.q[layer], s.scale, s.outs[layer], s.out_dtype, None, s.ws, s.flags)
        elif c["op"] == "prefill":
            B.q4kv_prefill_attention(s.spec, s.pool, s.n_blocks, layer, s.batch, s.lens, s.offs, s.total, s.most_new,
                                     s.most_kv, s.windows[layer], s.q[layer], s.scale, s.outs[layer], s.out_dtype, None,
                                     s.ws, s.flags)
    if c["op"] == "append":
        return s.pool, s.flags
    return s.out, s.pool, s.flags
