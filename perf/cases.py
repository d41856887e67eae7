"""The work that a user of this library has it do, one case each, for timing.

Everything goes through the public entry points (`paper_2510_09608_b200.binding`), as a decoder that serves a video
stream calls them: layer after layer, inputs and outputs in buffers that the program keeps, positions that go on growing
with the stream.  A pass is one second's chunk (`chunk`, `chunk_proj`), a run of generated tokens (`decode`,
`decode_proj`), or a whole second with everything in host memory (`host`).  Every pass ends with the cache at the size it
had before (append and evict balance), so passes can follow one another for as long as one likes.

Fields of a case
    op              chunk | decode | chunk_proj | decode_proj | host
    layers, q_heads, kv_heads, head_dim, rope ("1d" | "mrope")
    n_sink, vision_window, text_window      the cache policy, in tokens
    frames, grid_h, grid_w, text            a chunk: frames x grid_h x grid_w vision tokens, then `text` text tokens
    streams         independent streams served together through the batched calls (1: the single-stream calls)
    steps           generated tokens per pass (decode, decode_proj, host)
    graph           the pass is captured once as a CUDA graph and replayed, as a server does with its token loop
    hidden          width of the hidden state (the projections' side; 0 without)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_09608_b200 import binding

TABLE = 32      # passes for which positions are laid out ahead; the table then moves on by that many passes


def listed():
    tiny = dict(layers=1, q_heads=4, kv_heads=1, head_dim=64, rope="1d", n_sink=4, vision_window=64, text_window=128,
                frames=1, grid_h=4, grid_w=8, text=5, streams=1, steps=0, graph=False, hidden=0)
    qwen = dict(layers=28, q_heads=28, kv_heads=4, head_dim=128, rope="mrope", n_sink=512, vision_window=8192, text_window=512,
                frames=2, grid_h=16, grid_w=16, text=12, streams=1, steps=0, graph=False, hidden=0)
    return [
        # the smallest stream (first row of the workload table): call latency and launches are everything
        dict(tiny, name="chunk-tiny", op="chunk"),
        dict(tiny, name="decode-tiny", op="decode", steps=4),
        # one second of video on one layer of the 7B shape: what a caller sees who interleaves layers with other work
        dict(qwen, name="chunk-1layer", op="chunk", layers=1, text=19),
        # the deployed case: one second of video, all 28 layers one after another
        dict(qwen, name="chunk-28layers", op="chunk"),
        # a stream that catches up after a stall: eight seconds of video and a long prompt arrive in one chunk
        dict(qwen, name="chunk-catch-up", op="chunk", layers=4, frames=16, text=37),
        # eight streams in lock step with chunks of different lengths (8 frames/s of 64 tokens)
        dict(qwen, name="chunk-8streams", op="chunk", frames=8, grid_h=8, grid_w=8, text=32, streams=8),
        # the answer to one second: 16 tokens through 28 layers, replayed from a graph; and a token by plain calls
        dict(qwen, name="decode-28layers-graph", op="decode", steps=16, graph=True),
        dict(qwen, name="decode-28layers-calls", op="decode", steps=2),
        # sixteen streams generate together (fourth row of the workload table)
        dict(qwen, name="decode-16streams", op="decode", layers=1, streams=16, steps=16),
        # the decoder layer's attention half with its projections, hidden state in, hidden state out
        dict(qwen, name="chunk-projected", op="chunk_proj", text=19, hidden=3584),
        dict(qwen, name="decode-projected", op="decode_proj", steps=2, graph=True, hidden=3584),
        # a whole second end to end from pinned host memory, all layers per call
        dict(qwen, name="second-from-host", op="host", steps=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any head shape, window sizes and chunk lengths that are multiples of nothing."""
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["chunk", "chunk", "chunk", "decode", "decode", "decode", "chunk_proj", "decode_proj", "host"])
        q_heads, kv_heads, head_dim = rng.choice([(4, 1, 64), (28, 4, 128), (28, 4, 128), (28, 4, 128), (16, 2, 128),
                                                  (32, 8, 128), (12, 2, 64), (8, 8, 128), (16, 8, 64)])
        hidden = 0
        if op == "chunk_proj":
            head_dim, hidden = 128, 128 * _log_int(rng, 4, 32)     # 128: what the projection with the append is built for
        elif op == "decode_proj":
            q_heads, kv_heads, head_dim, hidden = 28, 4, 128, 3584  # the one decoder whose token projections a process serves
        streams = rng.choice([1, 1, 2, 3, 8, 16]) if op in ("chunk", "decode") else 1
        c = dict(op=op, layers=_log_int(rng, 1, 28), q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim,
                 rope=rng.choice(["1d", "mrope"]), n_sink=_log_int(rng, 4, 1024), vision_window=_log_int(rng, 64, 16384),
                 text_window=_log_int(rng, 64, 1024), frames=_log_int(rng, 1, 16), grid_h=_log_int(rng, 4, 16),
                 grid_w=_log_int(rng, 4, 18), text=rng.randint(0, 40), streams=streams,
                 steps=_log_int(rng, 1, 24) if op in ("decode", "decode_proj", "host") else 0,
                 graph=op in ("decode", "decode_proj") and rng.random() < 0.5,
                 hidden=hidden)
        if op == "decode" and streams > 1:
            c["layers"] = min(c["layers"], 4)
        if _cost(c) <= most and _bytes_held(c) < 25e9 and c["layers"] * c["steps"] <= 28 * 16:
            return c


# ---- geometry --------------------------------------------------------------------------------------------------

def _n_vision(c):
    return c["frames"] * c["grid_h"] * c["grid_w"]


def _chunk_lengths(c):
    """New tokens of each stream's chunk.  Streams served together bring text bursts of different lengths."""
    texts = [c["text"]] if c["streams"] == 1 else [(5 + 7 * i) % (c["text"] + 1) for i in range(c["streams"])]
    return [_n_vision(c) + t for t in texts], texts


def _retained(c):
    return c["n_sink"] + c["vision_window"] + c["text_window"]


def _capacity(c):
    return (_retained(c) + max(_chunk_lengths(c)[0]) + c["steps"] + 127) // 128 * 128


def _bytes_held(c):
    chunk = 0 if c["op"] == "decode" else sum(_chunk_lengths(c)[0]) * (2 * c["q_heads"] + 2 * c["kv_heads"])
    slab = 2 * c["streams"] * (_capacity(c) + _retained(c)) * c["kv_heads"]
    return 2 * c["layers"] * (c["head_dim"] * (chunk + slab) + c["hidden"] * (2 * c["q_heads"] + 2 * c["kv_heads"]) * c["head_dim"])


def _positions(c, tokens, base):
    """Native positions of a run of tokens (list of ("v", n, skipped) | ("t", n)) from cursor `base`, and the new cursor."""
    out = []
    for kind, n, skip in tokens:
        if c["rope"] == "1d":
            out.append(base + np.arange(n, dtype=np.int64))
            base += n
        elif kind == "t":
            out.append(np.repeat((base + np.arange(n, dtype=np.int64))[:, None], 3, axis=1))
            base += n
        else:
            f, r, w = np.meshgrid(np.arange(c["frames"]), np.arange(c["grid_h"]), np.arange(c["grid_w"]), indexing="ij")
            out.append((np.stack([f, r, w], axis=-1).reshape(-1, 3) + base)[skip:])
            base += max(c["frames"], c["grid_h"], c["grid_w"])
    return np.concatenate(out, axis=0), base


def _types(tokens):
    return np.concatenate([np.full(n, binding.VISION if k == "v" else binding.TEXT, np.uint8) for k, n, _ in tokens])


def _history(c):
    """A full cache as a running stream leaves it: sinks, then vision blocks with text between them, exactly the windows.
    A stream that only generates has its newest tokens all text: there the vision comes first."""
    v, blocks = c["vision_window"], max(1, -(-c["vision_window"] // _n_vision(c)))
    tokens, text = [("t", c["n_sink"], 0)], c["text_window"]
    first = v - (blocks - 1) * _n_vision(c)
    for b in range(blocks):
        n = first if b == 0 else _n_vision(c)
        tokens.append(("v", n, _n_vision(c) - n))
        if c["op"] not in ("decode", "decode_proj"):
            share = text // (blocks - b)
            text -= share
            if share:
                tokens.append(("t", share, 0))
    if text:
        tokens.append(("t", text, 0))
    return tokens


# ---- states ----------------------------------------------------------------------------------------------------

class _State:
    pass


class _PositionTable:
    """Positions of the next passes, one row a pass; the whole table moves on when it is used up."""

    def __init__(self, rows, advance, views, device):
        t = torch.from_numpy((rows[None] + advance * np.arange(TABLE).reshape((TABLE,) + (1,) * rows.ndim)).astype(np.int32))
        self.table = t.to(device) if device == "cuda" else t.pin_memory()
        self.step = TABLE * advance
        self.views = [views(self.table[k]) for k in range(TABLE)]
        self.at = 0

    def next(self):
        if self.at == TABLE:
            self.table.add_(self.step)
            self.at = 0
        self.at += 1
        return self.views[self.at - 1]


def _normal(gen, *shape, scale=1.0):
    x = torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    return x.mul_(scale) if scale != 1.0 else x


def _new_cache(c, gen):
    """A cache in its steady state (every window full) and the stream's position cursor."""
    cache = binding.Cache(c["layers"], c["kv_heads"], c["head_dim"], c["n_sink"], c["vision_window"], c["text_window"], _capacity(c))
    half = c["head_dim"] // 2
    if c["rope"] == "1d":
        cache.set_rope(binding.ROPE_1D, 1.0e4)
    else:
        cache.set_rope(binding.ROPE_MROPE, 1.0e6, (half // 4, 3 * half // 8, half - half // 4 - 3 * half // 8))
    tokens = _history(c)
    pos, base = _positions(c, tokens, 0)
    shape = (c["layers"], len(pos), c["kv_heads"], c["head_dim"])
    cache.append(-1, _normal(gen, *shape), _normal(gen, *shape), torch.from_numpy(_types(tokens)).cuda(),
                 torch.from_numpy(pos.astype(np.int32)).cuda())
    cache.evict()
    return cache, base


def _chunk_tokens(c, text):
    return [("v", _n_vision(c), 0)] + ([("t", text, 0)] if text else [])


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    s = _State()
    s.case = c
    made = [_new_cache(c, gen) for _ in range(c["streams"])]
    s.caches, s.base = [m[0] for m in made], made[0][1]
    s.cache = s.caches[0]
    return {"chunk": _prepare_chunk, "chunk_proj": _prepare_chunk, "decode": _prepare_decode, "decode_proj": _prepare_decode,
            "host": _prepare_host}[c["op"]](s, c, gen)


def _prepare_chunk(s, c, gen):
    lengths, texts = _chunk_lengths(c)
    L, hq, hk, d = c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"]
    total = sum(lengths)
    s.types = [torch.from_numpy(_types(_chunk_tokens(c, t))).cuda() for t in texts]
    rows, ends = zip(*[_positions(c, _chunk_tokens(c, t), s.base) for t in texts])
    cuts = np.cumsum([0] + lengths)
    # one advance for all streams: the longest chunk's (a stream may skip positions, as after a longer silence)
    s.pos = _PositionTable(np.concatenate(rows, axis=0), max(ends) - s.base,
                           lambda row: (row, [row[cuts[i]:cuts[i + 1]] for i in range(len(lengths))]), "cuda")
    s.n_q = lengths
    if c["op"] == "chunk":
        k, v = _normal(gen, L, total, hk, d), _normal(gen, L, total, hk, d)
        s.kv = [[(k[l, cuts[i]:cuts[i + 1]], v[l, cuts[i]:cuts[i + 1]]) for i in range(c["streams"])] for l in range(L)]
        s.q = list(_normal(gen, L, total, hq, d))
        s.out = torch.empty(L, total, hq, d, dtype=torch.bfloat16, device="cuda")
        s.outs = list(s.out)
    else:
        h = c["hidden"]
        s.x = list(_normal(gen, L, total, h))
        s.w_qkv = list(_normal(gen, L, (hq + 2 * hk) * d, h, scale=h ** -0.5))
        s.w_o = list(_normal(gen, L, h, hq * d, scale=(hq * d) ** -0.5))
        s.q1 = torch.empty(total, hq, d, dtype=torch.bfloat16, device="cuda")
        s.a1 = torch.empty_like(s.q1)
        s.a1_rows = s.a1.view(total, hq * d)
        s.out = torch.empty(L, total, h, dtype=torch.bfloat16, device="cuda")
        s.outs = list(s.out)
    return s


def _prepare_decode(s, c, gen):
    L, hq, hk, d, T, B = c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], c["steps"], c["streams"]
    s.type = torch.zeros(B, dtype=torch.uint8, device="cuda")                      # generated tokens are text
    rows, _ = _positions(c, [("t", T, 0)], s.base)
    rows = np.repeat(rows[:, None], B, axis=1)                                     # [T, B(, 3)]
    if c["op"] == "decode":
        k, v, q = _normal(gen, T, L, B, hk, d), _normal(gen, T, L, B, hk, d), _normal(gen, T, L, B, hq, d)
        s.out = torch.empty(T, L, B, hq, d, dtype=torch.bfloat16, device="cuda")
        s.io = [[(k[t, l], v[t, l], q[t, l], s.out[t, l]) for l in range(L)] for t in range(T)]
    else:
        h = c["hidden"]
        s.w_qkv = list(_normal(gen, L, (hq + 2 * hk) * d, h, scale=h ** -0.5))
        s.w_o = list(_normal(gen, L, h, hq * d, scale=(hq * d) ** -0.5))
        x = _normal(gen, T, L, 1, h)
        s.out = torch.empty(T, L, 1, h, dtype=torch.bfloat16, device="cuda")
        s.io = [[(x[t, l], s.out[t, l]) for l in range(L)] for t in range(T)]
        s.qkv = torch.empty(1, (hq + 2 * hk) * d, dtype=torch.bfloat16, device="cuda")
        s.q1 = s.qkv[:, :hq * d].view(1, hq, d)
        s.k1 = s.qkv[:, hq * d:(hq + hk) * d].view(1, hk, d)
        s.v1 = s.qkv[:, (hq + hk) * d:].view(1, hk, d)
        s.a1 = torch.empty(1, hq, d, dtype=torch.bfloat16, device="cuda")
        s.a1_row = s.a1.view(1, hq * d)
    # one stream: a token's position is [1] or [1, 3]; several: [B] or [B, 3]
    s.graph = None
    if not c["graph"]:
        s.pos = _PositionTable(rows, T, lambda row: list(row), "cuda")
        return s
    s.static_pos = torch.from_numpy(rows.astype(np.int32)).cuda()
    views = list(s.static_pos)
    torch.cuda.synchronize()
    s.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s.graph):
        for cache in s.caches:
            cache.set_stream(torch.cuda.current_stream())
        _generate(s, views)
        s.static_pos.add_(T)
    for cache in s.caches:
        cache.set_stream(torch.cuda.current_stream())
    return s


def _prepare_host(s, c, gen):
    lengths, texts = _chunk_lengths(c)
    n, L, hq, hk, d, T = lengths[0], c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], c["steps"]
    pinned = lambda *shape: torch.empty(*shape, dtype=torch.bfloat16, pin_memory=True)          # noqa: E731
    filled = lambda *shape: pinned(*shape).copy_(_normal(gen, *shape))                           # noqa: E731
    s.types = torch.from_numpy(_types(_chunk_tokens(c, texts[0]))).pin_memory()
    s.type = torch.zeros(1, dtype=torch.uint8).pin_memory()
    chunk, base = _positions(c, _chunk_tokens(c, texts[0]), s.base)
    token, end = _positions(c, [("t", T, 0)], base)
    s.pos = _PositionTable(np.concatenate([chunk, token], axis=0), end - s.base,
                           lambda row: (row[:n], [row[n + t:n + t + 1] for t in range(T)]), "cpu")
    s.kv, s.q, s.out = (filled(L, n, hk, d), filled(L, n, hk, d)), filled(L, n, hq, d), pinned(L, n, hq, d)
    s.tok_out = pinned(T, L, 1, hq, d)
    k, v, q = filled(T, L, 1, hk, d), filled(T, L, 1, hk, d), filled(T, L, 1, hq, d)
    s.io = [(k[t], v[t], q[t], s.tok_out[t]) for t in range(T)]
    return s


# ---- passes ----------------------------------------------------------------------------------------------------

def run(state):
    s = state
    op = s.case["op"]
    if op == "chunk":
        return _run_chunk(s)
    if op == "chunk_proj":
        return _run_chunk_proj(s)
    if op == "host":
        return _run_host(s)
    if s.graph is not None:
        s.graph.replay()
    else:
        _generate(s, s.pos.next())
    return s.out


def _run_chunk(s):
    pos, per_stream = s.pos.next()
    caches, single = s.caches, len(s.caches) == 1
    for l, (q, out) in enumerate(zip(s.q, s.outs)):
        for i, cache in enumerate(caches):
            k, v = s.kv[l][i]
            if l == 0:
                cache.append(0, k, v, s.types[i], per_stream[i])
            else:
                cache.append(l, k, v)
        if single:
            if l == 0:
                s.cache.evict()
            s.cache.attend(l, q, pos, out)
        else:
            if l == 0:
                binding.evict_batched(caches)
            binding.attend_batched_varlen(caches, l, q, pos, s.n_q, out)
    return s.out


def _run_chunk_proj(s):
    pos, _ = s.pos.next()
    cache, hq = s.cache, s.case["q_heads"]
    for l, (x, out) in enumerate(zip(s.x, s.outs)):
        if l == 0:
            cache.qkv_append(0, x, s.w_qkv[0], hq, s.types[0], pos, s.q1)
            cache.evict()
        else:
            cache.qkv_append(l, x, s.w_qkv[l], hq, None, None, s.q1)
        cache.attend(l, s.q1, pos, s.a1)
        cache.out_proj(s.a1_rows, s.w_o[l], out)
    return s.out


def _generate(s, positions):
    """The pass's generated tokens, layer after layer, and then the eviction that makes room for as many again."""
    cache, proj = s.cache, s.case["op"] == "decode_proj"
    for pos, io in zip(positions, s.io):
        if proj:
            for l, (x, out) in enumerate(io):
                cache.out_proj(x, s.w_qkv[l], s.qkv)
                cache.decode_step(l, s.k1, s.v1, s.type if l == 0 else None, pos, s.q1, s.a1)
                cache.out_proj(s.a1_row, s.w_o[l], out)
        elif len(s.caches) == 1:
            for l, (k, v, q, out) in enumerate(io):
                cache.decode_step(l, k, v, s.type if l == 0 else None, pos, q, out)
        else:
            for l, (k, v, q, out) in enumerate(io):
                binding.decode_step_batched(s.caches, l, k, v, s.type if l == 0 else None, pos, q, out)
    if len(s.caches) == 1:
        cache.evict()
    else:
        binding.evict_batched(s.caches)


def _run_host(s):
    pos, token_pos = s.pos.next()
    cache = s.cache
    cache.append_host(-1, s.kv[0], s.kv[1], s.types, pos)
    cache.evict()
    cache.attend_host(-1, s.q, pos, s.out)
    for p, (k, v, q, out) in zip(token_pos, s.io):
        cache.decode_step_host(-1, k, v, s.type, p, q, out)
    return [s.out, s.tok_out]


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    """Per layer: every stored key and value read once per attention call, new rows read and written once, queries read,
    outputs written; keys that an eviction moves are written back once.  Flops: Q K^T and P V over the visible pairs, and
    the projections."""
    c = case
    L, hq, hk, d, T = c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], c["steps"]
    kept, row, qrow = _retained(c), hk * d * 2, hq * d * 2
    nbytes = flops = 0
    if c["op"] in ("chunk", "chunk_proj", "host"):
        for n in _chunk_lengths(c)[0]:
            # the chunk pushes as much out as it brings, so it attends over what the windows hold
            old = max(0, kept - n)
            pairs = n * old + n * (n + 1) // 2
            nbytes += 2 * kept * row + 4 * n * row + 2 * n * qrow       # K, V once; new K, V in and out; Q in, result out
            nbytes += (kept - c["n_sink"]) * row                        # moved keys written back
            flops += 4 * hq * d * pairs
    if c["op"] in ("decode", "decode_proj", "host"):
        nbytes += c["streams"] * T * (2 * kept * row + 4 * row + 2 * qrow)
        flops += c["streams"] * T * 4 * hq * d * kept
        if c["op"] != "host":
            nbytes += c["streams"] * 2 * c["text_window"] * row         # the text keys that the eviction moves, in and out
    if c["hidden"]:
        n, h = (sum(_chunk_lengths(c)[0]), c["hidden"]) if c["op"] == "chunk_proj" else (T, c["hidden"])
        weights = ((hq + 2 * hk) * d + hq * d) * h
        # a chunk reads the weights once; each generated token needs them all again
        nbytes += 2 * weights * (1 if c["op"] == "chunk_proj" else T) + 4 * n * h
        flops += 2 * n * weights
    return {"bytes": L * nbytes, "flops": L * flops}


def _cost(c):
    w = work(c)
    return w["bytes"] / 6.5e12 + w["flops"] / 1.6e15


def tolerance(case):
    """bf16 keys, weights of the softmax and outputs, fp32 accumulation: each rounding is 2^-9 of its value at most."""
    return {"rel": 1e-2, "max": 0.1}
