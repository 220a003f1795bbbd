"""The work that programs have this library do, as measurable cases.

Each case is one pass of a kind of program, through the public Python names
of ``paper_2608_06849_gb300.aoh``:

  token     one token of a batch through a stack of layers, captured once in a
            CUDA graph and replayed (allocation-free step, caller-owned arena)
  engine    one eager decode step of a serving engine that owns the KV buffer
            and the device lengths (allocation-free step), ragged lengths
  decode    one eager decode step through a cache handle
  generate  a whole small request: reset, prefill, then a few decode steps
  prefill   a whole prompt: reset, then one call or a run of chunks
  h2share   one decode step of an H2Share block: an anchor layer and the reuse
            layers that borrow its positions
  classify  head labels of a whole model from its projection weights
  h2map     group mapping of one reuse layer onto its anchor layer

Shapes are those of the repository's workloads (28/4 and 32/8 heads of 128,
8/2 heads of 64) and generic ones; inputs are N(0, 1) with the first key
scaled by 8 where a prompt starts (an attention sink).

The engine and token programs set the device lengths before every step, so a
pass does the same work each time. A handle's lengths grow by one a pass, which
its contexts and headroom make irrelevant.
"""

import math
import random
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2608_06849_gb300 import aoh

HEADROOM = 16384  # rows a handle cache keeps free past its context


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # batch-1 chat at a short context: 28 launches whose fixed cost counts
        dict(name="token_28l_4k", kind="token", layers=28, batch=1, q_heads=28, kv_heads=4, d_head=128,
             context=4096, sink=128, window=2048, streaming=2),
        # batch-1 step at the longest context, one layer of the 256K stack
        dict(name="engine_b1_256k", kind="engine", batch=1, q_heads=28, kv_heads=4, d_head=128,
             low=262144, high=262144, sink=128, window=4096, streaming=2),
        # continuous batching: 64 sequences of very different lengths
        dict(name="engine_b64_ragged", kind="engine", batch=64, q_heads=32, kv_heads=8, d_head=128,
             low=4096, high=32768, sink=64, window=2048, streaming=4),
        # small-head model (64-wide heads) served in a moderate batch
        dict(name="engine_d64_b8", kind="engine", batch=8, q_heads=32, kv_heads=8, d_head=64,
             low=12001, high=32768, sink=64, window=1024, streaming=4),
        # the largest step: 16 sequences at 128K
        dict(name="decode_b16_128k", kind="decode", batch=16, q_heads=32, kv_heads=8, d_head=128,
             context=131072, sink=128, window=4096, streaming=4),
        # the smallest request: 64-wide heads, a 1K prompt and 32 tokens
        dict(name="generate_d64_1k", kind="generate", batch=1, q_heads=8, kv_heads=2, d_head=64,
             prompt=1024, steps=32, sink=16, window=128, streaming=1),
        # one long prompt in one call
        dict(name="prefill_32k", kind="prefill", batch=1, q_heads=28, kv_heads=4, d_head=128,
             prompt=32768, call=32768, low=32768, sink=128, window=2048, streaming=2, rule=0),
        # the same prompt as a server feeds it, 4K tokens a call
        dict(name="prefill_8x4k", kind="prefill", batch=1, q_heads=28, kv_heads=4, d_head=128,
             prompt=32768, call=4096, low=32768, sink=128, window=2048, streaming=2, rule=0),
        # a padded batch of short prompts of odd lengths
        dict(name="prefill_b8_ragged", kind="prefill", batch=8, q_heads=32, kv_heads=8, d_head=128,
             prompt=2999, call=2999, low=301, sink=64, window=512, streaming=4, rule=0),
        # H2Share block at 128K: one anchor, two reuse layers
        dict(name="h2share_b16_128k", kind="h2share", batch=16, q_heads=32, kv_heads=8, d_head=128,
             context=131072, sink=128, window=4096, streaming=4, reuse=2, top_k=2048),
        # offline, once a model: labels of 28 layers
        dict(name="classify_28l", kind="classify", layers=28, q_heads=28, kv_heads=4, d_head=128, d_model=3584,
             sparsity=50),
        # offline, once a pair of layers
        dict(name="h2map_pair", kind="h2map", q_heads=28, kv_heads=4, d_head=128, d_model=3584, streaming=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds alike often, sizes spread over their ranges."""
    kind = rng.choice(["token", "engine", "engine", "decode", "generate", "prefill", "prefill", "h2share",
                       "classify", "h2map"])
    q_heads, kv_heads = rng.choice([(28, 4), (32, 8), (16, 2), (24, 8), (8, 8), (40, 8)])
    c = dict(kind=kind, batch=1, q_heads=q_heads, kv_heads=kv_heads, d_head=128, sink=rng.choice([0, 16, 64, 128]),
             window=_log_int(rng, 256, 4096), streaming=rng.randint(0, kv_heads))
    if kind == "token":
        c.update(layers=rng.randint(8, 28), batch=rng.choice([1, 1, 2, 4]), context=_log_int(rng, 1000, 32768))
    elif kind == "engine":
        if rng.random() < 0.35:
            q_heads, kv_heads = rng.choice([(32, 8), (8, 2), (28, 4), (16, 8)])
            c.update(q_heads=q_heads, kv_heads=kv_heads, d_head=64, streaming=rng.randint(0, kv_heads))
        high = _log_int(rng, 4096, 131072)
        c.update(batch=max(1, min(64, _log_int(rng, max(1, 131072 // high), max(2, 524288 // high)))), high=high,
                 low=rng.randint(high // 8, high))
    elif kind == "decode":
        c.update(context=_log_int(rng, 65536, 131072), batch=rng.randint(2, 8))
        c.update(streaming=rng.randint(0, kv_heads - 1))
    elif kind == "generate":
        q_heads, kv_heads, d_head = rng.choice([(8, 2, 64), (32, 8, 64), (28, 4, 128), (32, 8, 128)])
        c.update(q_heads=q_heads, kv_heads=kv_heads, d_head=d_head, streaming=rng.randint(0, kv_heads),
                 batch=rng.choice([1, 2]), prompt=_log_int(rng, 200, 4096), steps=rng.randint(8, 32))
    elif kind == "prefill":
        if rng.random() < 0.3:
            q_heads, kv_heads = rng.choice([(32, 8), (8, 2)])
            c.update(q_heads=q_heads, kv_heads=kv_heads, d_head=64, streaming=rng.randint(0, kv_heads))
        # at most the attended work of the long listed prompt, whatever the heads
        longest = int(32768 * math.sqrt(min(1.0, 14 / c["q_heads"])))
        prompt = _log_int(rng, 300, longest)
        form = rng.choice(["one", "chunks", "batch"])
        c.update(prompt=prompt, call=prompt, low=prompt, rule=0)
        if form == "chunks":
            call = rng.choice([1024, 2048, 4096])
            prompt = max(prompt, 2 * call + 1)
            c.update(prompt=prompt, low=prompt, call=call, rule=rng.choice([0, call]))
        elif form == "batch":
            c.update(batch=max(1, min(16, longest // prompt)), low=max(1, prompt // rng.choice([1, 2, 8])))
    elif kind == "h2share":
        c.update(context=_log_int(rng, 65536, 131072), batch=rng.randint(4, 12), streaming=rng.randint(0, kv_heads - 1),
                 reuse=rng.randint(1, 3), top_k=_log_int(rng, 512, 4096))
    elif kind == "classify":
        c = dict(kind=kind, layers=_log_int(rng, 1, 14), q_heads=q_heads, kv_heads=kv_heads,
                 d_head=rng.choice([64, 128]), d_model=rng.choice([512, 1000, 2048, 3584, 4096]),
                 sparsity=rng.choice([25, 50, 75]))
    else:
        c = dict(kind=kind, q_heads=q_heads, kv_heads=kv_heads, d_head=rng.choice([64, 128]),
                 d_model=rng.choice([512, 1000, 2048, 3584, 4096]), streaming=rng.randint(0, kv_heads - 1))
    return c


# ------------------------------------------------------------------ inputs

class State:
    pass


def _gen(seed, tag):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + tag)


def _randn(shape, seed, tag):
    return torch.randn(shape, generator=_gen(seed, tag), device="cuda", dtype=torch.bfloat16)


def _labels(case, seed, layer=0):
    n = case["kv_heads"]
    picked = random.Random(int(seed) * 131 + layer).sample(range(n), case["streaming"])
    return [1 if h in picked else 0 for h in range(n)]


def _past(case, seed, layer, tokens):
    """K and V of a layer's cached tokens, [B, tokens, kv_heads, d_head]."""
    shape = (case["batch"], tokens, case["kv_heads"], case["d_head"])
    k = _randn(shape, seed, 1000 + 10 * layer)
    k[:, 0] *= 8.0
    return k, _randn(shape, seed, 1001 + 10 * layer)


def _step(case, seed, step):
    """q, k, v of one new token of every sequence."""
    B, d = case["batch"], case["d_head"]
    return (_randn((B, case["q_heads"], d), seed, 500000 + 3 * step),
            _randn((B, case["kv_heads"], d), seed, 500001 + 3 * step),
            _randn((B, case["kv_heads"], d), seed, 500002 + 3 * step))


def _prompt(case, seed):
    shape = (case["batch"], case["prompt"])
    q = _randn(shape + (case["q_heads"], case["d_head"]), seed, 900)
    k, v = _past(case, seed, 0, case["prompt"])
    return q, k, v


def _lens(case, seed):
    """Tokens each sequence holds (engine) or each prompt has (prefill)."""
    r = random.Random(int(seed) * 17 + 5)
    high = case["high"] if "high" in case else case["prompt"]
    return [high] + [r.randint(case["low"], high) for _ in range(case["batch"] - 1)]


def _weights(case, seed):
    """Projection weights [layers][heads][d_head][d_model] whose spectra decay,
    each head at its own rate, as trained projections' do."""
    L, dh, dm = case.get("layers", 1), case["d_head"], case["d_model"]
    g = _gen(seed, 77)
    out = []
    for heads in (case["q_heads"], case["kv_heads"]):
        w = torch.empty((L, heads, dh, dm), device="cuda", dtype=torch.bfloat16)
        for layer in range(L):
            mix = torch.randn((heads, dh, dh), generator=g, device="cuda") / math.sqrt(dh)
            rate = 1.0 + 3.0 * torch.rand((heads, 1, 1), generator=g, device="cuda")
            decay = torch.exp(-rate * torch.arange(dh, device="cuda").view(1, 1, dh) / dh)
            base = torch.randn((heads, dh, dm), generator=g, device="cuda") / math.sqrt(dm)
            w[layer] = torch.bmm(mix * decay, base)
        out.append(w)
    return out


def _config(case, max_seq, rule=0):
    return aoh.make_config(case["batch"], case["q_heads"], case["kv_heads"], case["d_head"], max_seq, case["sink"],
                           case["window"], rule)


def _filled_handle(case, seed, layer, tokens, max_seq):
    cache = aoh.Cache(case["batch"], case["q_heads"], case["kv_heads"], case["d_head"], max_seq, case["sink"],
                      case["window"], _labels(case, seed, layer))
    cache.buffer.zero_()
    k, v = _past(case, seed, layer, tokens)
    cache.prefill(None, k, v)
    return cache


def prepare(case, seed):
    s = State()
    s.kind = case["kind"]
    B, d = case.get("batch", 1), case["d_head"]
    if s.kind in ("token", "engine"):
        L = case.get("layers", 1)
        lens = [case["context"]] * B if s.kind == "token" else _lens(case, seed)
        s.max_len = max(lens)
        s.cfg = _config(case, s.max_len + 1)
        s.labels = [_labels(case, seed, layer) for layer in range(L)]
        size = (aoh.aoh_cache_bytes(s.cfg, s.labels[0]) + 255) // 256 * 256
        arena = torch.zeros(L * size, dtype=torch.uint8, device="cuda")
        s.kv = arena.view(torch.int16)
        s.buffers = [arena[i * size:(i + 1) * size] for i in range(L)]
        for layer in range(L):
            k, v = _past(case, seed, layer, s.max_len)
            h = aoh.aoh_cache_init(s.cfg, s.labels[layer], s.buffers[layer])
            aoh.aoh_prefill(None, k, v, s.max_len, lens, h, None)
            torch.cuda.synchronize()
            aoh.aoh_cache_destroy(h)
        s.held = torch.tensor(lens * L, dtype=torch.int32, device="cuda")
        s.lens = s.held.clone()
        s.layer_lens = [s.lens[i * B:(i + 1) * B] for i in range(L)]
        s.inputs = [_step(case, seed, layer) for layer in range(L)]
        s.out = torch.zeros((L, B, case["q_heads"], d), dtype=torch.bfloat16, device="cuda")
        s.outs = [s.out[i] for i in range(L)]
        if s.kind == "token":
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.stream(side):
                _layers(s)
            torch.cuda.current_stream().wait_stream(side)
            with torch.cuda.graph(s.graph):
                _layers(s)
    elif s.kind == "decode":
        s.cache = _filled_handle(case, seed, 0, case["context"], case["context"] + HEADROOM)
        s.kv = s.cache.buffer.view(torch.int16)
        s.q, s.k, s.v = _step(case, seed, 0)
        s.out = torch.zeros_like(s.q)
    elif s.kind == "generate":
        s.cache = aoh.Cache(B, case["q_heads"], case["kv_heads"], d, case["prompt"] + case["steps"], case["sink"],
                            case["window"], _labels(case, seed))
        s.cache.buffer.zero_()
        s.kv = s.cache.buffer.view(torch.int16)
        s.q, s.k, s.v = _prompt(case, seed)
        s.out = torch.zeros_like(s.q)
        s.inputs = [_step(case, seed, i) for i in range(case["steps"])]
        s.out_steps = torch.zeros((case["steps"], B, case["q_heads"], d), dtype=torch.bfloat16, device="cuda")
        s.outs = [s.out_steps[i] for i in range(case["steps"])]
    elif s.kind == "prefill":
        s.cache = aoh.Cache(B, case["q_heads"], case["kv_heads"], d, case["prompt"], case["sink"], case["window"],
                            _labels(case, seed), chunk=case["rule"])
        s.cache.buffer.zero_()
        s.kv = s.cache.buffer.view(torch.int16)
        q, k, v = _prompt(case, seed)
        n = case["call"]
        s.chunks = [tuple(x[:, i:i + n].contiguous() for x in (q, k, v)) for i in range(0, case["prompt"], n)]
        s.seq_lens = _lens(case, seed) if case["low"] < case["prompt"] else None
        s.outs = [torch.zeros_like(c[0]) for c in s.chunks]
    elif s.kind == "h2share":
        n = case["context"]
        s.anchor = _filled_handle(case, seed, 0, n, n + HEADROOM)
        s.anchor.reserve(1, anchor_workspace=True)
        s.reuse = [_filled_handle(case, seed, 1 + i, n, n + HEADROOM) for i in range(case["reuse"])]
        n_r = case["kv_heads"] - case["streaming"]
        s.top_k = case["top_k"]
        s.indices = torch.zeros((B, n_r, s.top_k), dtype=torch.int32, device="cuda")
        s.map = _borrowed(case, seed)
        s.inputs = [_step(case, seed, i) for i in range(1 + case["reuse"])]
        s.out = torch.zeros((1 + case["reuse"], B, case["q_heads"], d), dtype=torch.bfloat16, device="cuda")
        s.outs = [s.out[i] for i in range(1 + case["reuse"])]
        s.kv = [c.buffer.view(torch.int16) for c in [s.anchor] + s.reuse]
    elif s.kind == "classify":
        s.wq, s.wk = _weights(case, seed)
        s.kv_heads, s.sparsity = case["kv_heads"], case["sparsity"]
    else:
        (s.qa, s.ka), (s.qr, s.kr) = ([w[0] for w in x] for x in _pair(case, seed))
        s.la, s.lr = _labels(case, seed, 0), _labels(case, seed, 1)
    return s


def _borrowed(case, seed):
    """The anchor retrieval slot that each reuse retrieval group borrows from."""
    n_r = case["kv_heads"] - case["streaming"]
    r = random.Random(int(seed) * 7 + 3)
    return [r.randrange(n_r) for _ in range(n_r)]


def _pair(case, seed):
    """Weights of an anchor layer and of a reuse layer that resembles it."""
    a, b = _weights(case, seed), _weights(case, seed + 500)
    return a, [(0.8 * x.float() + 0.6 * y.float()).to(torch.bfloat16) for x, y in zip(a, b)]


# ------------------------------------------------------------------ one pass

def _layers(s):
    s.lens.copy_(s.held)
    for cfg_labels, buffer, lens, (q, k, v), out in zip(s.labels, s.buffers, s.layer_lens, s.inputs, s.outs):
        aoh.aoh_decode_step_noalloc(s.cfg, cfg_labels, buffer, lens, s.max_len, q, k, v, out)


def run(s):
    if s.kind == "token":
        s.graph.replay()
        return {"out": s.out, "lens": s.lens, "kv": s.kv}
    if s.kind == "engine":
        _layers(s)
        return {"out": s.out, "lens": s.lens, "kv": s.kv}
    if s.kind == "decode":
        s.cache.decode_step(s.q, s.k, s.v, s.out)
        return {"out": s.out, "kv": s.kv}
    if s.kind == "generate":
        s.cache.reset()
        s.cache.prefill(s.q, s.k, s.v, s.out)
        for (q, k, v), out in zip(s.inputs, s.outs):
            s.cache.decode_step(q, k, v, out)
        return {"out": s.out, "steps": s.out_steps, "kv": s.kv}
    if s.kind == "prefill":
        s.cache.reset()
        for (q, k, v), out in zip(s.chunks, s.outs):
            s.cache.prefill(q, k, v, out, seq_lens=s.seq_lens)
        return {"out": s.outs, "kv": s.kv}
    if s.kind == "h2share":
        q, k, v = s.inputs[0]
        s.anchor.decode_step_anchor(q, k, v, s.outs[0], s.top_k, s.indices)
        for cache, (q, k, v), out in zip(s.reuse, s.inputs[1:], s.outs[1:]):
            cache.decode_step_reuse(q, k, v, out, s.indices, s.top_k, s.map)
        return {"out": s.out, "indices": s.indices, "kv": s.kv}
    if s.kind == "classify":
        labels, er = aoh.aoh_classify(s.wq, s.wk, s.kv_heads, s.sparsity)
        return {"er": np.array(er), "labels": np.array(labels)}
    head_map, sim = aoh.aoh_h2share_map(s.qa, s.ka, s.qr, s.kr, s.la, s.lr)
    return {"map": np.array(head_map), "sim": np.array(sim)}


# ------------------------------------------------------------------ the work

def _decode_work(case, lens, rows=None):
    """Bytes and flops of one decode step over the given lengths: the rows each
    head reads (`rows`: those of a retrieval head, all of them by default), the
    new token's rows read and appended, q and out."""
    d, hq, hk, n_s = case["d_head"], case["q_heads"], case["kv_heads"], case["streaming"]
    n = 0
    for t in lens:
        r = t + 1 if rows is None else min(rows, t + 1)
        n += (hk - n_s) * r + n_s * min(t + 1, case["sink"] + case["window"])
    B = len(lens)
    return (n - B * hk) * d * 4 + B * hk * d * 8 + B * hq * d * 4, n * (hq // hk) * 4 * d


def _seen(case, n, streaming):
    """Attended (query, key) pairs of a prompt of n tokens, one query head."""
    i = np.arange(n, dtype=np.int64)
    if not streaming:
        return int((i + 1).sum())
    rule, S, W = case.get("rule", 0), case["sink"], case["window"]
    start = (i // rule) * rule - W if rule else i - W + 1
    start = np.maximum(start, 0)
    return int((i + 1 - start + np.minimum(S, start)).sum())


def _prefill_work(case, lens):
    d, hq, hk, n_s = case["d_head"], case["q_heads"], case["kv_heads"], case["streaming"]
    g = hq // hk
    nbytes = flops = 0
    for n in lens:
        kept = (hk - n_s) * n + n_s * min(n, case["sink"] + case["window"])
        nbytes += n * hq * d * 4 + n * hk * d * 4 + kept * d * 4
        pairs = (hk - n_s) * g * _seen(case, n, False) + (n_s * g * _seen(case, n, True) if n_s else 0)
        flops += pairs * 4 * d
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "token":
        b, f = _decode_work(case, [case["context"]] * case["batch"])
        b, f = b * case["layers"], f * case["layers"]
    elif kind == "engine":
        b, f = _decode_work(case, _lens(case, 0))
    elif kind == "decode":
        b, f = _decode_work(case, [case["context"]] * case["batch"])
    elif kind == "generate":
        b, f = _prefill_work(case, [case["prompt"]] * case["batch"])
        for i in range(case["steps"]):
            x, y = _decode_work(case, [case["prompt"] + i] * case["batch"])
            b, f = b + x, f + y
    elif kind == "prefill":
        b, f = _prefill_work(case, _lens(case, 0) if case["low"] < case["prompt"] else [case["prompt"]] * case["batch"])
    elif kind == "h2share":
        lens = [case["context"]] * case["batch"]
        b, f = _decode_work(case, lens)
        x, y = _decode_work(case, lens, case["top_k"])
        lists = case["batch"] * (case["kv_heads"] - case["streaming"]) * case["top_k"] * 4
        b, f = b + lists + case["reuse"] * (x + lists), f + case["reuse"] * y
    elif kind == "classify":
        # symmetric Gram matrices, their Cholesky factors, the product of two
        # and its singular values (bidiagonal form: 8/3 n^3)
        n, dh, dm = case["q_heads"] + case["kv_heads"], case["d_head"], case["d_model"]
        f = case["layers"] * (n * (dm * dh * (dh + 1) + dh ** 3 / 3) + case["q_heads"] * (dh ** 3 * 2 / 3 + dh ** 3 * 8 / 3))
        b = case["layers"] * n * dh * dm * 2
    else:
        hq, hk, dh, dm = case["q_heads"], case["kv_heads"], case["d_head"], case["d_model"]
        nq, nk = hq * dh, hk * dh
        f = 2 * dm * (nq * nq + nk * nk) + 2 * dm * 2 * (hq + hk) * dh * dh
        b = 2 * (nq + nk) * dm * 2
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Four times the relative error measured against exact(), by kind."""
    kind = case["kind"]
    if kind == "classify":
        # fp64 throughout: 8e-16 off another fp64 route (QR and a bidiagonal
        # SVD); a few ulps of the sums over d_head singular values
        return {"rel": 1e-14, "max": 1e-13}
    if kind == "h2map":
        # fp32 sums over d_model on the tensor cores: 7e-6 off
        return {"rel": 3e-5, "max": 3e-4}
    if kind == "h2share":
        # a row that ties with the last one taken shifts its list's entries
        return {"rel": 6e-3, "max": 0.06, "differ": 0.01}
    # bf16 outputs and softmax weights: 1.5e-3 to 1.7e-3 off in every case
    return {"rel": 6e-3, "max": 0.06}


# ------------------------------------------------------------------ 64 bits

def _softmax_v(q, k, v, scale, hidden=None):
    """softmax(q k^T scale) v in 64 bits; q [G, n, d], k, v [m, d]."""
    s = torch.matmul(q, k.T) * scale
    if hidden is not None:
        s.masked_fill_(hidden, -math.inf)
    s = torch.exp(s - s.amax(-1, keepdim=True))
    return torch.matmul(s, v) / s.sum(-1, keepdim=True)


def _exact_step(case, labels, k, v, lens, q, k_new, v_new, rows=None):
    """One decode step's outputs [B, q_heads, d]. `rows`: per (sequence, KV
    head) the positions a retrieval head attends to (None: all)."""
    B, d, G = case["batch"], case["d_head"], case["q_heads"] // case["kv_heads"]
    out = torch.zeros((B, case["q_heads"], d), dtype=torch.float64, device="cuda")
    for b in range(B):
        t = int(lens[b])
        for h, streaming in enumerate(labels):
            kk = torch.cat([k[b, :t, h], k_new[b, h][None]]).double()
            vv = torch.cat([v[b, :t, h], v_new[b, h][None]]).double()
            if streaming:
                j = torch.arange(t + 1, device="cuda")
                keep = (j < case["sink"]) | (t - j < case["window"])
                kk, vv = kk[keep], vv[keep]
            elif rows is not None:
                kk, vv = kk[rows[b, h]], vv[rows[b, h]]
            qq = q[b, h * G:(h + 1) * G].double()[:, None]
            out[b, h * G:(h + 1) * G] = _softmax_v(qq, kk, vv, 1 / math.sqrt(d))[:, 0]
    return out


def _exact_prompt(case, labels, q, k, v, lens):
    B, d, G = case["batch"], case["d_head"], case["q_heads"] // case["kv_heads"]
    rule, S, W, block = case.get("rule", 0), case["sink"], case["window"], 1024
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    for b in range(B):
        for h, streaming in enumerate(labels):
            kk, vv = k[b, :, h].double(), v[b, :, h].double()
            for i0 in range(0, lens[b], block):
                i1 = min(lens[b], i0 + block)
                j = torch.arange(i1, device="cuda")
                if streaming:
                    first = (i0 // rule) * rule - W if rule else i0 - W + 1
                    j = j[(j < S) | (j >= first)]
                i = torch.arange(i0, i1, device="cuda")[:, None]
                hidden = j[None] > i
                if streaming:
                    start = (i // rule) * rule - W if rule else i - W + 1
                    hidden |= (j[None] >= S) & (j[None] < start)
                qq = q[b, i0:i1, h * G:(h + 1) * G].double().transpose(0, 1)
                o = _softmax_v(qq, kk[j], vv[j], 1 / math.sqrt(d), hidden)
                out[b, i0:i1, h * G:(h + 1) * G] = o.transpose(0, 1)
    return out


def _exact_er(wq, wk):
    """Effective ranks of one layer's heads (numpy, QR route)."""
    rq = np.linalg.qr(np.swapaxes(wq, 1, 2), mode="r")
    rk = np.linalg.qr(np.swapaxes(wk, 1, 2), mode="r")
    rk = np.repeat(rk, len(rq) // len(rk), axis=0)
    s = np.linalg.svd(np.matmul(rk, np.swapaxes(rq, 1, 2)), compute_uv=False)
    s = np.where(s > s[:, :1] * max(wq.shape[1:]) * np.finfo(np.float64).eps, s, 0.0)
    p = s / s.sum(1, keepdims=True)
    return np.exp(-(p * np.log(np.where(p > 0, p, 1.0))).sum(1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "classify":
        wq, wk = (w.double().cpu().numpy() for w in _weights(case, seed))
        with ThreadPoolExecutor(8) as pool:
            er = list(pool.map(lambda x: _exact_er(*x), zip(wq, wk)))
        return {"er": np.array(er), "labels": None}
    if kind == "h2map":
        (qa, ka), (qr, kr) = ([w[0].double() for w in x] for x in _pair(case, seed))
        G = len(qa) // len(ka)
        ma, mr = ka.repeat_interleave(G, 0), kr.repeat_interleave(G, 0)
        norm = []
        for w, m in ((qa, ma), (qr, mr)):
            norm.append((torch.bmm(w, w.mT) * torch.bmm(m, m.mT)).sum((1, 2)))
        # tr((Wk_a^T Wq_a)^T (Wk_r^T Wq_r)) of every head pair
        num = torch.stack([(torch.matmul(qa[i], qr.mT) * torch.matmul(ma[i], mr.mT)).sum((1, 2))
                           for i in range(len(qa))])
        sim = num / torch.sqrt(norm[0][:, None] * norm[1][None])
        n = len(ka)
        return {"map": None, "sim": sim.view(n, G, n, G).mean((1, 3)).cpu().numpy()}
    if kind in ("generate", "prefill"):
        if work(case)["flops"] > 6e12:
            return None
        q, k, v = _prompt(case, seed)
        lens = _lens(case, seed) if kind == "prefill" and case["low"] < case["prompt"] else [case["prompt"]] * case["batch"]
        labels = _labels(case, seed)
        o = _exact_prompt(case, labels, q, k, v, lens)
        if kind == "prefill":
            return {"out": [o[:, i:i + case["call"]] for i in range(0, case["prompt"], case["call"])], "kv": None}
        steps = []
        for i in range(case["steps"]):
            nq, nk, nv = _step(case, seed, i)
            steps.append(_exact_step(case, labels, k, v, [k.shape[1]] * case["batch"], nq, nk, nv))
            k, v = torch.cat([k, nk[:, None]], 1), torch.cat([v, nv[:, None]], 1)
        return {"out": o, "steps": torch.stack(steps), "kv": None}
    if kind in ("token", "engine", "decode"):
        lens = _lens(case, seed) if kind == "engine" else [case["context"]] * case["batch"]
        out = []
        for layer in range(case.get("layers", 1)):
            k, v = _past(case, seed, layer, max(lens))
            out.append(_exact_step(case, _labels(case, seed, layer), k, v, lens, *_step(case, seed, layer)))
        if kind == "decode":
            return {"out": out[0], "kv": None}
        return {"out": torch.stack(out), "lens": None, "kv": None}
    # h2share
    B, n, d, G = case["batch"], case["context"], case["d_head"], case["q_heads"] // case["kv_heads"]
    lens = [n] * B
    labels = _labels(case, seed, 0)
    k, v = _past(case, seed, 0, n)
    q, nk, nv = _step(case, seed, 0)
    out = [_exact_step(case, labels, k, v, lens, q, nk, nv)]
    heads = [h for h, x in enumerate(labels) if not x]
    picked = torch.empty((B, len(heads), min(case["top_k"], n + 1)), dtype=torch.int64, device="cuda")
    for b in range(B):
        for i, h in enumerate(heads):
            kk = torch.cat([k[b, :, h], nk[b, h][None]]).double()
            p = torch.softmax(q[b, h * G:(h + 1) * G].double() @ kk.T / math.sqrt(d), -1).sum(0)
            picked[b, i] = torch.topk(p, picked.shape[2]).indices
    slots = _borrowed(case, seed)
    for layer in range(1, 1 + case["reuse"]):
        labels = _labels(case, seed, layer)
        k, v = _past(case, seed, layer, n)
        rows, r = {}, 0
        for h, x in enumerate(labels):
            if not x:
                rows.update({(b, h): picked[b, slots[r]] for b in range(B)})
                r += 1
        out.append(_exact_step(case, labels, k, v, lens, *_step(case, seed, layer), rows=rows))
    return {"out": torch.stack(out), "indices": None, "kv": [None] * (1 + case["reuse"])}
