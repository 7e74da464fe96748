"""Performance cases of the compressed KV cache: the calls a serving program makes, over the range of sizes it makes them.

Kinds of pass (`"do"` of a case):
  decode   one decoding step's attention: gear_decode_attn once per layer, every layer with a cache of its own
  rows     the same for several query rows per head (positions scored together): gear_decode_attn_multi
  prefill  a prompt's K, V blocks of every layer into new caches, and the first token's attention over them
  request  the whole life of a request: new caches, the prompt, then per token and layer one push (every buffer_cap-th
           push compresses the buffer) and one attention, then the caches are given back.  With host = True the new rows,
           the query and the result of every step are host buffers (gear_step_host, gear_cache_wait)
`pushed` tokens follow the prompt in the caches that a decode or rows pass finds, so that flushed segments and a partly
filled buffer are part of it.  Device memory of the caches comes from torch's allocator, as in any program that lives in
a torch process (gear_set_allocator); inputs are drawn on the device with the distribution of synth.make_kv.
"""
from __future__ import annotations

import math

import torch

from paper_2403_05527_b200 import binding as G

HEAD_DIM = 128
POWER_ITERS = 3


def _case(name, do, layers, batch, q_heads, kv_heads, n, bits, group, s_pct, rank, buffer_cap, pushed=0, rows=1, steps=0,
          host=False):
    c = {"do": do, "layers": layers, "batch": batch, "q_heads": q_heads, "kv_heads": kv_heads, "n": n, "bits": bits,
         "group": group, "s_pct": s_pct, "rank": rank, "buffer_cap": buffer_cap, "pushed": pushed, "rows": rows,
         "steps": steps, "host": host}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # one head, 256 tokens: the smallest call, all launch latency
        _case("decode one head", "decode", 1, 1, 1, 1, 256, 4, 64, 2.0, 4, 16, pushed=23),
        # interactive decoding of a single sequence with a 32-layer, 32-head model; ragged prompt
        _case("decode 32 layers b1", "decode", 32, 1, 32, 32, 3776, 2, 64, 2.0, 4, 64, pushed=100),
        # the benchmark's layer: batch 8, context 4096; four layers so that a step reads more than the L2 holds
        _case("decode b8 2-bit", "decode", 4, 8, 32, 32, 4096, 2, 64, 2.0, 4, 64, pushed=96),
        # throughput decoding of 40-head layers, 4-bit codes, rank 8: the largest cache
        _case("decode b16 4-bit r8", "decode", 1, 16, 40, 40, 8192, 4, 64, 1.0, 8, 64, pushed=33),
        # grouped queries over a long context
        _case("decode gqa 32k", "decode", 2, 4, 32, 8, 32768, 2, 128, 2.0, 4, 64, pushed=70),
        # per-vector key grouping with the 20-token buffer
        _case("decode per-vector b8", "decode", 3, 8, 32, 32, 4096, 4, 0, 2.0, 4, 20, pushed=31),
        # four draft positions verified at once over grouped heads: 16 query rows per kv head
        _case("rows 4 gqa", "rows", 2, 3, 32, 8, 8192, 2, 128, 2.0, 4, 64, pushed=37, rows=4),
        # prompts of the benchmark's layer
        _case("prefill b8 2-bit", "prefill", 1, 8, 32, 32, 4096, 2, 64, 2.0, 4, 64),
        # the largest prompt block: 4-bit, rank 8
        _case("prefill b16 4-bit r8", "prefill", 1, 16, 40, 40, 8192, 4, 64, 1.0, 8, 64),
        # a long prompt of grouped heads, groups of 128
        _case("prefill gqa 16k", "prefill", 2, 2, 32, 8, 16384, 2, 128, 2.0, 4, 64),
        # a short chat turn: prompt, then 200 tokens pushed and attended, three of them flushing a buffer
        _case("request b2 4-bit", "request", 2, 2, 32, 32, 448, 4, 64, 2.0, 4, 64, steps=200),
        # the same life through host buffers, per-vector keys, 20-token buffer
        _case("request host per-vector", "request", 2, 4, 32, 32, 1024, 4, 0, 2.0, 4, 20, steps=50, host=True),
    ]


# ----------------------------------------------------------------------------------------------- drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    do = rng.choice(["decode", "decode", "decode", "rows", "prefill", "prefill", "request"])
    q_heads, kv_heads = rng.choice([(32, 32), (32, 32), (40, 40), (12, 12), (5, 5), (32, 8), (32, 8), (24, 8), (28, 4), (64, 8)])
    bits = rng.choice([2, 2, 4])
    group = rng.choice([64, 64, 64, 128, 128, 32, 0])
    s_pct = rng.choice([2.0, 2.0, 1.0, 1.0, 0.0])
    rank = rng.choice([4, 4, 8, 2, 1, 16, 0])
    if group == 0:
        buffer_cap = rng.choice([20, 64, 128])
    elif group == 128:
        buffer_cap = rng.choice([64, 128])
    else:
        buffer_cap = rng.choice([64, 64, 128])
    batch = _log_int(rng, 1, 24)
    layers = _log_int(rng, 1, 12) if do == "decode" else rng.choice([1, 1, 2, 3])
    unit = 64 if group == 0 else group
    n = _log_int(rng, 32, 32768 if group else 8192)
    n = n // unit * unit if n >= unit else max(16, n // 16 * 16)
    if group == 0 and n > 128:
        n = n // 64 * 64
    rank = min(rank, buffer_cap, n)
    pushed = rows = steps = 0
    host = False
    if do in ("decode", "rows"):
        pushed = _log_int(rng, 1, 4 * buffer_cap) - 1
    if do == "rows":
        rows = _log_int(rng, 2, 12)
    if do == "request":
        steps = _log_int(rng, 8, 250)
        host = rng.random() < 0.35
    return _case(None, do, layers, batch, q_heads, kv_heads, n, bits, group, s_pct, rank, buffer_cap, pushed=pushed,
                 rows=max(rows, 1), steps=steps, host=host)


# at most about the largest listed cases of the same kind: bytes read by an attention pass, fp16 bytes of the prompts,
# and the steps of a request (tokens times layers; those through host buffers cost three times as much)
_MOST_DECODE_BYTES = 1.0e9
_MOST_PREFILL_BYTES = 1.3e9
_MOST_REQUEST_STEPS = 300


def draw(rng):
    while True:
        c = _draw_once(rng)
        prompt = c["layers"] * 2 * c["batch"] * c["kv_heads"] * c["n"] * HEAD_DIM * 2
        if c["do"] == "decode" and work(c)["bytes"] <= _MOST_DECODE_BYTES:
            return c
        if c["do"] == "rows" and work(c)["bytes"] * c["rows"] * c["q_heads"] // c["kv_heads"] <= _MOST_DECODE_BYTES:
            return c
        # general group shapes and ranks above 8 take several times as long per byte
        dear = 4 if c["group"] == 32 or c["rank"] > 8 or c["s_pct"] == 0 or (c["group"] in (0, 128) and c["s_pct"] != 2.0) else 1
        if c["do"] == "prefill" and 2e5 <= prompt <= _MOST_PREFILL_BYTES / dear:
            return c
        steps = c["layers"] * c["steps"] * (3 if c["host"] else 1) * (2 if dear > 1 else 1)
        if (c["do"] == "request" and prompt <= 0.25 * _MOST_PREFILL_BYTES / dear and steps <= _MOST_REQUEST_STEPS
                and work(c)["bytes"] <= 3e9):
            return c


# ----------------------------------------------------------------------------------------------- inputs and handles
_ALLOC = G.ALLOC_FN(lambda nbytes, _ctx: torch.cuda.caching_allocator_alloc(max(int(nbytes), 1)))
_FREE = G.FREE_FN(lambda ptr, _ctx: torch.cuda.caching_allocator_delete(ptr))


class Caches:
    """The layers' cache handles of one sequence batch; released with the object."""

    def __init__(self):
        self.handles = []

    def release(self):
        handles, self.handles = self.handles, []
        for h in handles:
            G.gear_free(h)

    def __del__(self):
        self.release()


def _normal_kv(gen, shape, channel_scale):
    """fp16 [B, H, n, 128]: N(0, 1), one entry in a hundred 20 times as large; keys with a scale per (head, channel)."""
    out = torch.empty(shape, dtype=torch.float16, device="cuda")
    for b in range(shape[0]):                        # sequence by sequence: small fp32 temporaries
        x = torch.randn(shape[1:], generator=gen, device="cuda")
        if channel_scale is not None:
            x.mul_(channel_scale)
        spikes = torch.rand(shape[1:], generator=gen, device="cuda") < 0.01
        out[b] = torch.where(spikes, x * 20.0, x)
    return out


def _prompt(gen, case):
    shape = (case["batch"], case["kv_heads"], case["n"], HEAD_DIM)
    scale = torch.exp(torch.randn((shape[1], 1, HEAD_DIM), generator=gen, device="cuda"))
    return _normal_kv(gen, shape, scale), _normal_kv(gen, shape, None), scale


def _config(case, seed):
    room = case["n"] + case["pushed"] + case["steps"] + case["buffer_cap"]
    return G.make_config(case["batch"], case["q_heads"], case["kv_heads"], case["bits"], case["group"], case["s_pct"],
                         case["buffer_cap"], case["rank"], room, rank_max=case["rank"], power_iters=POWER_ITERS,
                         seed=seed, max_queries=case["rows"])


def prepare(case, seed):
    G.gear_set_allocator(_ALLOC, _FREE)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    L, B, H, Hq, rows = case["layers"], case["batch"], case["kv_heads"], case["q_heads"], case["rows"]
    state = {"case": case, "config": _config(case, seed)}
    if case["do"] in ("decode", "rows"):
        # the caches as a running generation holds them: prompt compressed, `pushed` tokens decoded since
        caches = Caches()
        for _ in range(L):
            k, v, scale = _prompt(gen, case)
            caches.handles.append(G.gear_compress(None, state["config"], k, v, case["n"], case["rank"]))
            for _ in range(case["pushed"]):
                tok = torch.randn((2, B, H, HEAD_DIM), generator=gen, device="cuda")
                tok[0].mul_(scale[None, :, 0])
                tok = tok.half()
                G.gear_append_buffer(caches.handles[-1], tok[0], tok[1])
            del k, v
        shape = (L, B, Hq, HEAD_DIM) if case["do"] == "decode" else (L, B, Hq, rows, HEAD_DIM)
        q = torch.randn(shape, generator=gen, device="cuda").half()
        out = torch.empty(shape, dtype=torch.float32, device="cuda")
        state.update(caches=caches, q=list(q), out=out, outs=list(out))
    else:
        tokens = max(case["steps"], 1)
        prompts = [_prompt(gen, case) for _ in range(L)]
        new = torch.randn((2, tokens, L, B, H, HEAD_DIM), generator=gen, device="cuda")
        for layer, (_, _, scale) in enumerate(prompts):
            new[0, :, layer].mul_(scale[None, None, :, 0])
        new = new.half()
        q = torch.randn((tokens, L, B, Hq, HEAD_DIM), generator=gen, device="cuda").half()
        out = torch.empty((tokens, L, B, Hq, HEAD_DIM), dtype=torch.float32, device="cuda")
        if case["host"]:
            new, q = new.cpu().pin_memory(), q.cpu().pin_memory()
            out = torch.empty(out.shape, dtype=torch.float32).pin_memory()
        state.update(prompts=[p[:2] for p in prompts], k=[list(t) for t in new[0]], v=[list(t) for t in new[1]],
                     q=[list(t) for t in q], out=out, outs=[list(t) for t in out])
    return state


# ----------------------------------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    do = case["do"]
    if do == "decode":
        for cache, q, out in zip(state["caches"].handles, state["q"], state["outs"]):
            G.gear_decode_attn(cache, q, out)
        return state["out"]
    if do == "rows":
        for cache, q, out in zip(state["caches"].handles, state["q"], state["outs"]):
            G.gear_decode_attn_multi(cache, q, out, case["rows"])
        return state["out"]
    caches = Caches()
    for k, v in state["prompts"]:
        caches.handles.append(G.gear_compress(None, state["config"], k, v, case["n"], case["rank"]))
    if do == "prefill":
        for cache, q, out in zip(caches.handles, state["q"][0], state["outs"][0]):
            G.gear_decode_attn(cache, q, out)
    elif case["host"]:
        for ks, vs, qs, outs in zip(state["k"], state["v"], state["q"], state["outs"]):
            for cache, k, v, q, out in zip(caches.handles, ks, vs, qs, outs):
                G.gear_step_host(cache, k, v, q, out)
            for cache in caches.handles:
                G.gear_cache_wait(cache)
    else:
        for ks, vs, qs, outs in zip(state["k"], state["v"], state["q"], state["outs"]):
            for cache, k, v, q, out in zip(caches.handles, ks, vs, qs, outs):
                G.gear_append_buffer(cache, k, v)
                G.gear_decode_attn(cache, q, out)
    caches.release()
    return state["out"]


# ----------------------------------------------------------------------------------------------- accounting
def _outliers(s_pct, length):
    return math.ceil(round(s_pct * 10000) * length / 2000000)


def _segment_bytes(case, n):
    """Stored bytes of one compressed segment of n tokens per (sequence, kv head): codes, (scale, zero) pairs, outliers
    (fp16 value and one index byte; two in a vector longer than 256), factors A and B."""
    d, group, s, r = HEAD_DIM, case["group"], case["s_pct"], case["rank"]
    g_k, g_v = (min(group, n), min(group, d)) if group else (n, d)
    entry = 3 if g_k <= 256 else 4
    codes = 2 * n * d * case["bits"] // 8
    scales = 4 * (n // g_k * d + n * d // g_v)
    sparse = n // g_k * d * 2 * _outliers(s, g_k) * entry + n * d // g_v * 2 * _outliers(s, g_v) * 3
    return codes + scales + sparse + 2 * n * r * 2 + 2 * d * r * 2


def _cache_bytes(case, after):
    """Bytes of one layer's cache `after` tokens behind the prompt, whole batch."""
    nb = case["buffer_cap"]
    per_head = _segment_bytes(case, case["n"]) + after // nb * _segment_bytes(case, nb) + 2 * (after % nb) * HEAD_DIM * 2
    return case["batch"] * case["kv_heads"] * per_head


def _attention(case, after, rows=1):
    """bytes and flops of one attention: the cache and the query in, the result out; q K^T and p V."""
    heads = case["batch"] * case["q_heads"] * rows
    tokens = case["n"] + after
    return _cache_bytes(case, after) + heads * HEAD_DIM * (2 + 4), heads * tokens * HEAD_DIM * 4


def _compression(case, n):
    """K and V in, the segment out; two products of the residual with an n x r or 128 x r factor per loop."""
    heads = case["batch"] * case["kv_heads"]
    return (heads * (2 * n * HEAD_DIM * 2 + _segment_bytes(case, n)),
            heads * 2 * POWER_ITERS * 2 * (2 * n * HEAD_DIM * case["rank"]))


def work(case):
    L = case["layers"]
    if case["do"] in ("decode", "rows"):
        b, f = _attention(case, case["pushed"], case["rows"])
        return {"bytes": L * b, "flops": L * f}
    total_b, total_f = _compression(case, case["n"])
    if case["do"] == "prefill":
        b, f = _attention(case, 0)
        return {"bytes": L * (total_b + b), "flops": L * (total_f + f)}
    row = case["batch"] * case["kv_heads"] * 2 * HEAD_DIM * 2
    flush_b, flush_f = _compression(case, case["buffer_cap"])
    for t in range(1, case["steps"] + 1):
        b, f = _attention(case, t)
        total_b, total_f = total_b + row + b, total_f + f
        if t % case["buffer_cap"] == 0:
            total_b, total_f = total_b + flush_b, total_f + flush_f
    return {"bytes": L * total_b, "flops": L * total_f}


def tolerance(case):
    # Codes and outliers are exact; the factors A, B are stored in fp16.  Against the float64 oracle (other start of the
    # roundings, sums in another order) the attention over the stored caches differs by 2e-6 .. 2e-4, and by up to 4e-4
    # over prompts of 64 to 128 tokens.
    return {"rel": 1e-3}
