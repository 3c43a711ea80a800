"""What a user of this framework has it do, as cases that can be timed and compared.

One pass of every case is one whole request batch: a handle is opened on the program's own arena, the prompts go
through ``prefill_block`` block by block, the answers through ``decode_step`` token by token, with the evictions the
cadence asks for.  The handle's caches are internal to it; what comes back is the attention output of every call
(each later output is a function of the pairs that were kept) and the caches' final length and position.

``listed`` names a dozen such batches; ``draw`` gives more of the same ranges.
"""
from __future__ import annotations

import math

import torch

from paper_2412_05693_b200 import BatchMaxCache, arena_bytes, workspace_bytes
from paper_2412_05693_b200.binding import Config
from paper_2412_05693_b200.workloads import Inputs, Workload

# Keys of a case (defaults in parentheses):
#   b samples, Hq / Hkv query / KV heads, d head dimension, dtype, s prompt length, B block, K pairs kept,
#   steps decode steps, L (1) layers, heavy ("uniform") where the keys that stand out lie,
#   arm ("blocks"): "blocks" cuts back to K after every block and whenever decoding has grown p pairs above it,
#                   "alg1" is Algorithm 1 as printed (limit K + p, p pairs removed before each block of p tokens and
#                   before each step that would not fit), "once" compresses a single time, after the prompt,
#   p (1) growth above K, rule ("average"), compaction ("stable"), ragged (False) left-padded prompts of unequal
#   length, host (False) inputs and outputs in pinned host memory through the host-fed calls.


def _case(name=None, **kw):
    case = dict(L=1, heavy="uniform", arm="blocks", p=1, rule="average", compaction="stable", ragged=False, host=False,
                dtype="bf16")
    case.update(kw)
    if name is not None:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest call sizes: one layer in single precision, a handful of heads, as in unit tests and debugging
        _case("tiny_f32", b=2, Hq=4, Hkv=4, d=64, dtype="f32", s=512, B=64, K=128, steps=16),
        # one user, one long prompt: every launch has eight caches to work on
        _case("single_prompt", b=1, Hq=32, Hkv=8, d=128, s=4096, B=512, K=1024, steps=64),
        # a small batch through a stack of 32 layers, block by block and token by token
        _case("layer_stack", b=4, Hq=32, Hkv=8, d=128, s=1024, B=512, K=512, steps=16, L=32),
        # the usual serving batch with grouped heads
        _case("serving_batch", b=16, Hq=32, Hkv=8, d=128, s=4096, B=256, K=512, steps=128),
        # summarisation: long prompts, short answers, a batch that fills the GPU
        _case("long_prompts", b=128, Hq=32, Hkv=8, d=128, s=8192, B=512, K=1024, steps=64),
        # multi-head attention (no grouping), heavy positions at the front of the prompt
        _case("multi_head", b=32, Hq=32, Hkv=32, d=128, s=4096, B=1024, K=1024, steps=128, heavy="zipf"),
        # generation at a large batch: most of the time goes into decode steps out of HBM
        _case("large_batch_decode", b=384, Hq=32, Hkv=8, d=128, s=1536, B=512, K=1024, steps=128),
        # Algorithm 1 as printed, with its own p = 64 and the 40-head shape of the paper's larger model
        _case("algorithm1", b=16, Hq=40, Hkv=40, d=128, s=2560, B=1024, K=960, steps=128, arm="alg1", p=64),
        # prompts of unequal length, padded on the left, under the rule with a window of recent pairs; odd sizes
        _case("ragged_recent", b=24, Hq=32, Hkv=8, d=128, s=2901, B=256, K=499, steps=64, rule="sum_recent", ragged=True),
        # unordered caches, small heads in groups of eight, evictions every fourth step; odd sizes
        _case("unordered_d64", b=48, Hq=16, Hkv=2, d=64, s=3001, B=384, K=701, steps=64, compaction="fill", p=4),
        # an evaluation in single precision: grouped heads, one compression after the prompt
        _case("f32_once", b=4, Hq=16, Hkv=4, d=128, dtype="f32", s=1536, B=256, K=512, steps=32, arm="once"),
        # a program whose activations live on the host: every call copies its inputs in and its output back
        _case("host_fed", b=16, Hq=32, Hkv=8, d=128, s=1024, B=256, K=512, steps=32, host=True),
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _heads(rng, d, most_kv=8):
    g = rng.choice([1, 2, 4, 4, 8])
    kv = _between(rng, 1, most_kv)
    return dict(Hq=g * kv, Hkv=kv, d=d)


def _draw_one(rng):
    kind = rng.choice(["f32", "small", "stack", "serving", "serving", "long", "multi_head", "decode", "alg1", "ragged",
                       "unordered", "rule", "host"])
    if kind == "f32":
        once = rng.random() < 0.5
        d = rng.choice([64, 128])
        if once:   # larger, a single compression
            s = _between(rng, 256, 1536)
            return _case(b=_between(rng, 1, 6), **_heads(rng, d, 4), dtype="f32", s=s, B=_between(rng, 48, 320),
                         K=_between(rng, 64, max(64, s // 2)), steps=rng.randint(4, 32), arm="once")
        return _case(b=_between(rng, 1, 3), **_heads(rng, d, 4), dtype="f32", s=_between(rng, 128, 768),
                     B=_between(rng, 24, 128), K=_between(rng, 48, 256), steps=rng.randint(4, 24), p=rng.choice([1, 1, 4]))
    d = rng.choice([128, 128, 64])
    if kind == "small":
        return _case(b=_between(rng, 1, 4), **_heads(rng, d), s=_between(rng, 256, 6000), B=_between(rng, 32, 640),
                     K=_between(rng, 96, 1400), steps=rng.randint(8, 96), p=rng.choice([1, 1, 1, 8]))
    if kind == "stack":
        return _case(b=_between(rng, 1, 12), **_heads(rng, d), s=_between(rng, 128, 1200), B=_between(rng, 64, 600),
                     K=_between(rng, 96, 700), steps=rng.randint(4, 16), L=rng.randint(4, 32))
    if kind == "serving":
        return _case(b=_between(rng, 5, 48), Hq=32, Hkv=rng.choice([4, 8, 8, 16]), d=d, s=_between(rng, 700, 6000),
                     B=_between(rng, 128, 700), K=_between(rng, 200, 1400), steps=rng.randint(16, 128))
    if kind == "long":
        return _case(b=_between(rng, 24, 128), Hq=32, Hkv=8, d=d, s=_between(rng, 2000, 8192), B=_between(rng, 256, 1024),
                     K=_between(rng, 256, 2048), steps=rng.randint(16, 64))
    if kind == "multi_head":
        h = rng.choice([16, 24, 32, 40])
        return _case(b=_between(rng, 4, 32), Hq=h, Hkv=h, d=d, s=_between(rng, 700, 4096), B=_between(rng, 200, 1100),
                     K=_between(rng, 200, 2048), steps=rng.randint(16, 128), heavy=rng.choice(["zipf", "uniform"]))
    if kind == "decode":
        K = _between(rng, 200, 1500)
        return _case(b=_between(rng, 64, 384), Hq=32, Hkv=8, d=d, s=_between(rng, K, K + 600), B=512, K=K,
                     steps=rng.randint(64, 128))
    if kind == "alg1":
        h, p = rng.choice([8, 16, 32, 40]), rng.choice([32, 64, 64, 100])
        limit = _between(rng, 256, 1500)
        return _case(b=_between(rng, 2, 16), Hq=h, Hkv=h, d=d, s=_between(rng, limit, limit + 1200), B=limit, K=limit - p,
                     steps=rng.randint(16, 128), arm="alg1", p=p)
    if kind == "ragged":
        return _case(b=_between(rng, 2, 24), **_heads(rng, d), s=_between(rng, 300, 3000), B=_between(rng, 64, 512),
                     K=_between(rng, 96, 800), steps=rng.randint(8, 64), ragged=True,
                     rule=rng.choice(["average", "sum_recent", "current_query"]))
    if kind == "unordered":
        return _case(b=_between(rng, 2, 64), **_heads(rng, d), s=_between(rng, 300, 4000), B=_between(rng, 64, 700),
                     K=_between(rng, 96, 1200), steps=rng.randint(8, 96), compaction="fill", p=rng.choice([1, 1, 4, 16]))
    if kind == "rule":
        return _case(b=_between(rng, 2, 24), **_heads(rng, d), s=_between(rng, 300, 3000), B=_between(rng, 64, 512),
                     K=_between(rng, 96, 800), steps=rng.randint(8, 64), rule=rng.choice(["sum_recent", "current_query",
                                                                                         "window_pooled", "average_std"]))
    return _case(b=_between(rng, 2, 16), Hq=32, Hkv=8, d=d, s=_between(rng, 200, 1024), B=_between(rng, 64, 300),
                 K=_between(rng, 128, 600), steps=rng.randint(8, 32), host=True)


def _size(case):
    """Rough cost of a case in seconds, for keeping drawn ones below the largest listed one."""
    w = work(case)
    rate = 400e12 if case["dtype"] == "bf16" else 15e12
    calls = case["L"] * (case["steps"] + math.ceil(case["s"] / min(case["B"], case["p"] if case["arm"] == "alg1" else case["B"])))
    return w["flops"] / rate + w["bytes"] / (50e9 if case["host"] else 4e12) + 2e-5 * calls


def draw(rng):
    most = max(_size(c) for c in listed())
    while True:
        case = _draw_one(rng)
        if _size(case) <= most:
            return case


def _calls(case):
    """The calls of one layer: ("prefill", pos0, I, evict_to), ("decode", pos, 1, evict_to), ("evict", 0, 0, target)."""
    s, K, p, arm = case["s"], case["K"], case["p"], case["arm"]
    calls, n, pos = [], 0, 0
    while pos < s:
        if arm == "alg1" and n + 1 > K + p:
            calls.append(("evict", 0, 0, n - p))
            n -= p
        room = K + p - n if arm == "alg1" else s
        I = min(case["B"], s - pos, room)
        keep = K if arm == "blocks" else -1
        calls.append(("prefill", pos, I, keep))
        n, pos = (min(n + I, K) if keep >= 0 else n + I), pos + I
    if arm == "once" and n > K:
        calls.append(("evict", 0, 0, K))
        n = K
    for t in range(case["steps"]):
        if arm == "alg1" and n == K + p:
            calls.append(("evict", 0, 0, n - p))
            n -= p
        full = arm == "blocks" and n + 1 >= K + p
        calls.append(("decode", s + t, 1, K if full else -1))
        n = K if full else n + 1
    return calls


def _growth(case):
    if case["arm"] == "once":   # the whole prompt is cached first
        return max(case["s"] - case["K"], case["steps"], 1)
    return case["p"]


def work(case):
    """Bytes and operations a pass cannot do without: each call reads its inputs and the cached pairs (two rows and
    two 4-byte entries each) once and writes its output and the pairs it adds; 4 d operations per visible
    (query, key) pair.  Pairs moved by a compaction are not counted."""
    e = 2 if case["dtype"] == "bf16" else 4
    Hq, Hkv, d = case["Hq"], case["Hkv"], case["d"]
    row = 2 * d * e + 8
    n = nbytes = pairs = 0
    for kind, _, I, arg in _calls(case):
        if kind == "evict":
            n = min(n, arg)
            continue
        nbytes += 2 * I * Hq * d * e + 2 * I * Hkv * d * e + Hkv * n * row
        if not case["host"]:
            nbytes += Hkv * row * (min(I, arg) if arg >= 0 else I)
        pairs += I * n + I * (I + 1) // 2
        n = min(n + I, arg) if arg >= 0 else n + I
    if case["host"]:   # what crosses the host's link: the inputs one way, the outputs the other
        tokens = case["s"] + case["steps"]
        nbytes = tokens * (2 * Hq + 2 * Hkv) * d * e
    scale = case["b"] * case["L"]
    return {"bytes": scale * nbytes, "flops": scale * Hq * 4 * d * pairs}


def tolerance(case):
    # Measured against the same schedules run in 64 bits, ranking and attention both.  bf16 (outputs and the
    # probabilities on their way into P.V are rounded to 8 bits): relative error 2.1e-3 to 2.4e-3, and up to 5.5e-3
    # (a single value 0.77 off) where two pairs tie at a cut within the rounding of their 32-bit sums and the other one
    # stays.  f32: 2e-7 to 4e-7.
    return {"rel": 2e-2, "max": 0.99} if case["dtype"] == "bf16" else {"rel": 1e-5}


def prepare(case, seed):
    """A program's buffers for one batch: the prompts' and answers' Q/K/V, the outputs, the arena and the workspace."""
    s, steps = case["s"], case["steps"]
    wl = Workload(name="case", b=case["b"], Hq=case["Hq"], Hkv=case["Hkv"], d=case["d"], dtype=case["dtype"], s=s,
                  B=case["B"], K=case["K"], steps=steps, L=case["L"], seed=1009 * seed, heavy=case["heavy"],
                  heavy_count=max(1, round(0.01 * s)))
    calls = _calls(case)
    cfg = Config(batch=wl.b, n_q_heads=wl.Hq, n_kv_heads=wl.Hkv, head_dim=wl.d, kv_max=wl.K, block_max=wl.B,
                 growth=_growth(case), dtype=wl.dtype, n_layers=wl.L, rule=case["rule"], compaction=case["compaction"])
    where = dict(device="cpu", pin_memory=True) if case["host"] else dict(device="cuda")
    n_prompt = sum(c[2] for c in calls if c[0] == "prefill")
    out_prompt = torch.empty(wl.L, wl.b * n_prompt * wl.Hq * wl.d, dtype=wl.torch_dtype, **where)
    out_answer = torch.empty(wl.L, steps, wl.b, wl.Hq, wl.d, dtype=wl.torch_dtype, **where)
    inputs = Inputs(wl, "cuda")
    todo = [[None] * wl.L for _ in calls]
    for layer in range(wl.L):
        at = t = 0
        for i, (kind, pos0, I, arg) in enumerate(calls):
            if kind == "evict":
                todo[i][layer] = (kind, layer, arg)
                continue
            qkv = inputs.block(layer, pos0, I)
            if kind == "decode":
                qkv = tuple(x[:, 0].contiguous() for x in qkv)
                out, t = out_answer[layer, t], t + 1
            else:
                size = qkv[0].numel()
                out, at = out_prompt[layer, at:at + size].view(qkv[0].shape), at + size
            if case["host"]:
                qkv = tuple(x.cpu().pin_memory() for x in qkv)
            todo[i][layer] = (kind, layer, arg, *qkv, pos0, out)
    pads = None
    if case["ragged"]:
        gen = torch.Generator().manual_seed(1009 * seed + 5)
        pads = torch.randint(0, s // 2 + 1, (wl.b,), generator=gen).tolist()
    return {"cfg": cfg, "calls": [c for layers in todo for c in layers], "pads": pads, "host": case["host"],
            "arena": torch.empty(arena_bytes(cfg), dtype=torch.uint8, device="cuda"),
            "workspace": torch.empty(max(256, workspace_bytes(cfg)), dtype=torch.uint8, device="cuda"),
            "out_prompt": out_prompt, "out_answer": out_answer}


def run(state):
    cache = BatchMaxCache(state["cfg"], arena=state["arena"], workspace=state["workspace"])
    if state["pads"] is not None:
        cache.set_left_pad(state["pads"])
    prefill = cache.prefill_block_host if state["host"] else cache.prefill_block
    decode = cache.decode_step_host if state["host"] else cache.decode_step
    for kind, layer, arg, *rest in state["calls"]:
        if kind == "evict":
            cache.evict(arg, layer=layer)
            continue
        q, k, v, pos0, out = rest
        if kind == "prefill":
            prefill(q, k, v, pos0, out=out, evict_to=arg, layer=layer)
        else:
            decode(q, k, v, out=out, evict_to=arg, layer=layer)
    length, position = cache.length()
    cache.close()   # after host-fed calls this waits for their copies
    return {"prompt": state["out_prompt"], "answer": state["out_answer"], "length": length, "position": position}
