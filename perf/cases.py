"""Timed cases of the rollout-decoding library, through its public entry points.

A case is one call (or, for episodes, one loop of calls) that a self-play program makes again and again once its
weights, cache and buffers exist:

  decode    one token for every game of a batch (spiral_decode_step / _logprob): the rollout's inner loop
  nucleus   the same with the evaluation sampler (temperature 0.6, top-p 0.95; spiral_decode_step_nucleus)
  host      the same with token, noise and result in pinned host memory (spiral_decode_step_host)
  append    the observation tokens every game receives between two turns, with the logits behind them (spiral_prefill)
  episodes  games of two turns through the scheduler, from an empty cache to the polled responses (spiral_sched_*)

Decode and append passes roll the games back to where they were (spiral_kv_truncate, host bookkeeping), so that a pass
can be repeated.  Weights, tokens, cached keys/values and noise come from the seed; sizes come from the case alone.

Noise.  The sampler draws argmax(logit / T + noise).  Two correct implementations differ by the rounding of their
activations, about 1e-3 of a logit, and standard Gumbel noise puts the two best scores that close together once in a
thousand draws.  The noise here is Gumbel noise times 64: every entry is read and added as usual, and the draw's margin
is far above rounding, so tokens can be compared as whole numbers.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2506_24119_b200 as sp

PAGE = 16

# Architectures (random weights): the library's test decoder and the three model families it is used with.
MODELS = {
    "tiny": dict(n_layers=2, d_model=256, n_q_heads=4, n_kv_heads=2, head_dim=64, d_ff=688, vocab=4096,
                 rope_theta=1e6, rms_eps=1e-6, qk_norm=0, qkv_bias=0, tied_embed=1),
    "qwen3_4b": dict(n_layers=36, d_model=2560, n_q_heads=32, n_kv_heads=8, head_dim=128, d_ff=9728, vocab=151936,
                     rope_theta=1e6, rms_eps=1e-6, qk_norm=1, qkv_bias=0, tied_embed=1),
    "llama31_8b": dict(n_layers=32, d_model=4096, n_q_heads=32, n_kv_heads=8, head_dim=128, d_ff=14336, vocab=128256,
                       rope_theta=5e5, rms_eps=1e-5, qk_norm=0, qkv_bias=0, tied_embed=0),
    "qwen25_7b": dict(n_layers=28, d_model=3584, n_q_heads=28, n_kv_heads=4, head_dim=128, d_ff=18944, vocab=152064,
                      rope_theta=1e4, rms_eps=1e-6, qk_norm=0, qkv_bias=1, tied_embed=0),
}


def listed():
    return [
        # the smallest call: the test decoder, four games, on the current stream as a first program would call it
        dict(name="decode_tiny_4", kind="decode", model="tiny", n=4, max_batch=4, ctx_lo=64, ctx_hi=160, kv="f16",
             logprob=False, side_stream=False),
        # one game against one opponent: latency of a token
        dict(name="decode_4b_1", kind="decode", model="qwen3_4b", n=1, max_batch=1, ctx_lo=900, ctx_hi=900, kv="f16",
             logprob=False, side_stream=False),
        # the tail of a rollout: most games of a 128-game batch have finished, long ragged contexts
        dict(name="decode_4b_11_of_128", kind="decode", model="qwen3_4b", n=11, max_batch=128, ctx_lo=300, ctx_hi=3000,
             kv="f16", logprob=True, side_stream=True),
        # the benchmark's rollout: 128 games at 512 tokens
        dict(name="decode_4b_128", kind="decode", model="qwen3_4b", n=128, max_batch=128, ctx_lo=512, ctx_hi=512,
             kv="f16", logprob=False, side_stream=True),
        # the largest batches of the multi-turn configuration: early turns, short ragged contexts
        dict(name="decode_4b_213_of_256", kind="decode", model="qwen3_4b", n=213, max_batch=256, ctx_lo=40, ctx_hi=420,
             kv="f16", logprob=True, side_stream=True),
        # the 8B family at its prompt lengths, bf16 pages
        dict(name="decode_8b_29_bf16", kind="decode", model="llama31_8b", n=29, max_batch=64, ctx_lo=1024, ctx_hi=4096,
             kv="bf16", logprob=False, side_stream=True),
        # evaluation of a long-reasoning 7B policy with nucleus sampling
        dict(name="nucleus_7b_18", kind="nucleus", model="qwen25_7b", n=18, max_batch=32, ctx_lo=1024, ctx_hi=15000,
             kv="f16", logprob=False, side_stream=True),
        # a program that keeps tokens and noise on the host
        dict(name="host_4b_96", kind="host", model="qwen3_4b", n=96, max_batch=128, ctx_lo=200, ctx_hi=1000, kv="f16",
             logprob=False, side_stream=True),
        # one game's prompt and observation: time to the first token of a turn
        dict(name="append_4b_1x331", kind="append", model="qwen3_4b", n=1, max_batch=128, ctx_lo=450, ctx_hi=450,
             new_lo=331, new_hi=331, kv="f16", side_stream=False),
        # a dozen games that change turns together, ragged
        dict(name="append_4b_12x40_200", kind="append", model="qwen3_4b", n=12, max_batch=128, ctx_lo=300, ctx_hi=1200,
             new_lo=40, new_hi=200, kv="f16", side_stream=True),
        # a whole batch receives its observations at once: the largest call
        dict(name="append_4b_64x100_500", kind="append", model="qwen3_4b", n=64, max_batch=128, ctx_lo=200, ctx_hi=800,
             new_lo=100, new_hi=500, kv="f16", side_stream=True),
        # everything together: 32 games, two turns each, responses of different lengths
        dict(name="episodes_4b_32x2", kind="episodes", model="qwen3_4b", n=32, max_batch=32, turns=2, new_lo=30,
             new_hi=150, budget_lo=4, budget_hi=16, kv="f16", side_stream=True),
    ]


# ---- sizes that follow from a case ------------------------------------------------------------------------------

def _spread(n, lo, hi, phase=0.0):
    """n lengths over [lo, hi], ragged and the same for every seed."""
    return [lo + int((hi - lo + 1) * ((phase + (i + 1) * 0.6180339887498949) % 1.0)) for i in range(n)]


def _contexts(case):
    return _spread(case["n"], case["ctx_lo"], case["ctx_hi"])


def _observations(case, turn=0):
    return _spread(case["n"], case["new_lo"], case["new_hi"], 0.37 + 0.21 * turn)


def _budgets(case, turn=0):
    return _spread(case["n"], case["budget_lo"], case["budget_hi"], 0.11 + 0.29 * turn)


def _layer_weights(d):
    q, k = d["n_q_heads"] * d["head_dim"], d["n_kv_heads"] * d["head_dim"]
    return d["d_model"] * (q + 2 * k) + q * d["d_model"] + 3 * d["d_model"] * d["d_ff"]


def _kv_token_bytes(d):
    return d["n_layers"] * 2 * d["n_kv_heads"] * d["head_dim"] * 2


def _pages(tokens):
    return -(-tokens // PAGE)


# ---- cases over the whole range ---------------------------------------------------------------------------------

def _log(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    u = rng.random()
    kind = "decode" if u < 0.46 else "append" if u < 0.72 else "nucleus" if u < 0.82 else "host" if u < 0.92 else "episodes"
    side = rng.random() < 0.7
    if kind == "episodes":
        n = _log(rng, 6, 32)
        lo = rng.randint(10, 60)
        b = rng.randint(2, 6)
        return dict(kind=kind, model="qwen3_4b", n=n, max_batch=n + rng.choice([0, 0, 5]), turns=2, new_lo=lo,
                    new_hi=lo + rng.randint(0, 90), budget_lo=b, budget_hi=b + rng.randint(0, 9), kv="f16", side_stream=side)
    if kind == "host":
        model = "qwen3_4b"
    else:
        model = rng.choice(["tiny", "qwen3_4b", "qwen3_4b", "qwen3_4b", "llama31_8b", "qwen25_7b"])
    d = MODELS[model]
    kv = "bf16" if rng.random() < 0.2 else "f16"
    room = 9.5e9 / _kv_token_bytes(d)                   # cached tokens of all games together
    if kind == "append":
        total = _log(rng, 40, 12000 if model in ("tiny", "qwen3_4b") else 6500)      # new tokens of the call
        n = max(1, min(96, _log(rng, 1, 96), total // 12))
        max_batch = max(n, rng.choice([1, 16, 64, 128, 128, 256]))
        if kv == "bf16" or max_batch < 16:                # short observations: these take a decode-shaped step per max_batch
            total = max(n, min(total, 40 * max_batch, 1200))
        mean = total // n
        lo = max(1, int(mean * (rng.uniform(0.4, 1.0) if n > 1 else 1.0)))
        hi = max(lo, 2 * mean - lo)
        ctx_hi = min(_log(rng, 1, 2500), int(room / n) - hi)
        return dict(kind=kind, model=model, n=n, max_batch=max_batch,
                    ctx_lo=max(1, int(ctx_hi * rng.uniform(0.3, 1.0))), ctx_hi=max(1, ctx_hi), new_lo=lo, new_hi=hi, kv=kv,
                    side_stream=side)
    n = _log(rng, 1, 256 if kind == "decode" else 128)
    hi = max(24, min(_log(rng, 40, 15000 if model == "qwen25_7b" else 5000), int(room / n)))
    return dict(kind=kind, model=model, n=n, max_batch=rng.choice([n, max(n, 128), 256]),
                ctx_lo=max(1, int(hi * rng.uniform(0.2, 1.0))), ctx_hi=hi, kv=kv,
                logprob=kind == "decode" and rng.random() < 0.5, side_stream=side)


# ---- inputs -----------------------------------------------------------------------------------------------------

class State:
    """What a program keeps between calls; the library's handles are given back with it."""

    def __init__(self):
        self.ctx = self.kv = self.sched = None

    def __del__(self):
        if self.sched is not None:
            sp.spiral_sched_free(self.sched)
        if self.ctx is not None:
            sp.spiral_free(self.ctx, self.kv)


def _weights(d, gen, final_gain):
    """Random-init weights in the layout the library reads: matrices N(0, 0.02), norm gains 1."""
    def mat(rows, cols):
        return torch.randn(rows, cols, dtype=torch.bfloat16, device="cuda", generator=gen).mul_(0.02)

    def const(n, v=1.0):
        return torch.full((n,), v, dtype=torch.bfloat16, device="cuda")

    L, dm, hd, ff = d["n_layers"], d["d_model"], d["head_dim"], d["d_ff"]
    q, k = d["n_q_heads"] * hd, d["n_kv_heads"] * hd
    return {
        "embed": mat(d["vocab"], dm), "lm_head": None if d["tied_embed"] else mat(d["vocab"], dm),
        "final_norm": const(dm, final_gain), "ln1": [const(dm) for _ in range(L)], "ln2": [const(dm) for _ in range(L)],
        "wqkv": [mat(q + 2 * k, dm) for _ in range(L)],
        "bqkv": [mat(1, q + 2 * k)[0] if d["qkv_bias"] else None for _ in range(L)],
        "q_norm": [const(hd) if d["qk_norm"] else None for _ in range(L)],
        "k_norm": [const(hd) if d["qk_norm"] else None for _ in range(L)],
        "wo": [mat(dm, q) for _ in range(L)], "w_gate_up": [mat(2 * ff, dm) for _ in range(L)],
        "w_down": [mat(dm, ff) for _ in range(L)],
    }


def _noise(n, vocab, gen):
    u = torch.rand(n, vocab, dtype=torch.float32, device="cuda", generator=gen).clamp_(1e-7, 1.0 - 1e-7)
    return u.log_().neg_().log_().mul_(-64.0)


def prepare(case, seed):
    d = MODELS[case["model"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    rng = random.Random(int(seed))
    n, kind = case["n"], case["kind"]
    s = State()
    s.case = case
    s.stream = torch.cuda.Stream() if case["side_stream"] else None
    if kind == "episodes":
        totals = [sum(_observations(case, t)[i] + _budgets(case, t)[i] for t in range(case["turns"])) for i in range(n)]
        room = [t + 1 for t in totals]
    else:
        s.lens = _contexts(case)
        s.new = _observations(case) if kind == "append" else [1] * n
        room = [a + b for a, b in zip(s.lens, s.new)]
    max_ctx = max(room) + PAGE
    # a trained policy at temperature 0.6 keeps some hundred tokens in its nucleus: a larger gain before the LM head
    s.packed = _weights(d, gen, 3.0 if kind == "nucleus" else 1.0)
    s.ctx = sp.spiral_init(d, s.packed, torch.cuda.current_device(), max_batch=case["max_batch"], max_ctx=max_ctx)
    dtype = torch.float16 if case["kv"] == "f16" else torch.bfloat16
    n_pages = sum(_pages(r) for r in room) + n
    s.pool = torch.zeros(n_pages * sp.spiral_kv_page_bytes(d, PAGE) // 2, dtype=dtype, device="cuda")
    s.kv = sp.spiral_kv_alloc(s.ctx, s.pool, PAGE, n, max_ctx, sp.SPIRAL_KV_F16 if case["kv"] == "f16" else sp.SPIRAL_KV_BF16)
    V = d["vocab"]
    if kind == "episodes":
        s.sched = sp.spiral_sched_create(s.ctx, s.kv)
        sp.spiral_sched_collect_logprob(s.sched, True)
        s.obs = [[[rng.randrange(V) for _ in range(k)] for k in _observations(case, t)] for t in range(case["turns"])]
        s.budget = [_budgets(case, t) for t in range(case["turns"])]
        s.noise = [_noise(case["max_batch"], V, gen) for _ in range(4)]
        return s
    # contexts of earlier turns: game ids in no particular order, keys and values of every layer
    s.games = list(range(n))
    rng.shuffle(s.games)
    at = [0]
    for k in s.lens:
        at.append(at[-1] + k)
    shape = (at[-1], d["n_kv_heads"], d["head_dim"])
    for layer in range(d["n_layers"]):
        k = torch.empty(shape, dtype=dtype, device="cuda").uniform_(-2.0, 2.0, generator=gen)
        v = torch.empty(shape, dtype=dtype, device="cuda").uniform_(-1.0, 1.0, generator=gen)
        for i, g in enumerate(s.games):
            sp.spiral_kv_load(s.ctx, s.kv, g, layer, k[at[i]:at[i + 1]], v[at[i]:at[i + 1]])
    # rolled back last game first: freed pages are handed out again in the same order
    s.back_games, s.back_lens = s.games[::-1], s.lens[::-1]
    if kind == "append":
        offs = [0]
        for k in s.new:
            offs.append(offs[-1] + k)
        s.offsets = offs
        s.tokens = torch.randint(0, V, (offs[-1],), dtype=torch.int32, device="cuda", generator=gen)
        s.logits = torch.empty(n, V, dtype=torch.float32, device="cuda")
        return s
    s.tok_in = torch.randint(0, V, (n,), dtype=torch.int32, device="cuda", generator=gen)
    s.gumbel = _noise(n, V, gen)
    s.tok_out = torch.empty(n, dtype=torch.int32, device="cuda")
    s.logprob = torch.empty(n, dtype=torch.float32, device="cuda")
    if kind == "host":
        s.tok_in, s.gumbel, s.tok_out = s.tok_in.cpu().pin_memory(), s.gumbel.cpu().pin_memory(), s.tok_out.cpu().pin_memory()
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------

def _episodes(s):
    n, tick = s.case["n"], 0
    tokens, logprobs = [], []
    games = [sp.spiral_sched_open(s.sched) for _ in range(n)]
    for obs, budget in zip(s.obs, s.budget):
        for g, o, b in zip(games, obs, budget):
            sp.spiral_sched_turn(s.sched, g, o, b)
        got = {}
        while len(got) < n:
            sp.spiral_sched_tick(s.sched, s.noise[tick % len(s.noise)], 1.0, stream=s.stream)
            tick += 1
            while (r := sp.spiral_sched_poll_logprob(s.sched)) is not None:
                got[r[0]] = r
        for g in games:
            tokens += got[g][1]
            logprobs += got[g][2]
    for g in games:
        sp.spiral_sched_close(s.sched, g)
    return {"tokens": np.array(tokens, dtype=np.int32), "logprobs": np.array(logprobs, dtype=np.float32)}


def run(s):
    kind = s.case["kind"]
    if kind == "episodes":
        return _episodes(s)
    if kind == "append":
        sp.spiral_prefill(s.ctx, s.kv, s.games, s.tokens, s.offsets, s.logits, stream=s.stream)
        out = {"logits": s.logits, "cache": s.pool}
    elif kind == "host":
        sp.spiral_decode_step_host(s.ctx, s.kv, s.games, s.tok_in, s.gumbel, 1.0, s.tok_out, stream=s.stream)
        out = {"tokens": s.tok_out, "cache": s.pool}
    elif kind == "nucleus":
        sp.spiral_decode_step_nucleus(s.ctx, s.kv, s.games, s.tok_in, s.gumbel, 0.6, 0.95, s.tok_out, stream=s.stream)
        out = {"tokens": s.tok_out, "cache": s.pool}
    elif s.case["logprob"]:
        sp.spiral_decode_step_logprob(s.ctx, s.kv, s.games, s.tok_in, s.gumbel, 1.0, s.tok_out, s.logprob, stream=s.stream)
        out = {"tokens": s.tok_out, "logprobs": s.logprob, "cache": s.pool}
    else:
        sp.spiral_decode_step(s.ctx, s.kv, s.games, s.tok_in, s.gumbel, 1.0, s.tok_out, stream=s.stream)
        out = {"tokens": s.tok_out, "cache": s.pool}
    sp.spiral_kv_truncate(s.kv, s.back_games, s.back_lens)
    return out


# ---- what a pass cannot do without ------------------------------------------------------------------------------

def _segment_work(d, rows):
    """(bytes, flops) of the layers for rows = [(cached tokens, new tokens)] that share one pass over the weights."""
    kv = _kv_token_bytes(d)
    new = sum(b for _, b in rows)
    keys = sum(b * a + b * (b + 1) / 2 for a, b in rows)          # (query, key) pairs
    return (2 * d["n_layers"] * _layer_weights(d) + kv * sum(a + b for a, b in rows),
            2 * new * d["n_layers"] * _layer_weights(d) + 4 * d["n_layers"] * d["n_q_heads"] * d["head_dim"] * keys)


def _head_work(d, n, noise):
    return 2 * d["vocab"] * d["d_model"] + (4 * n * d["vocab"] if noise else 0), 2 * n * d["vocab"] * d["d_model"]


def work(case):
    d, n = MODELS[case["model"]], case["n"]
    if case["kind"] == "episodes":
        nbytes = flops = 0.0
        lens = [0] * n
        for t in range(case["turns"]):
            obs, budget = _observations(case, t), _budgets(case, t)
            parts = [_segment_work(d, list(zip(lens, obs)))]
            for k in range(max(budget)):          # the observation's last token feeds the first step
                live = [lens[i] + obs[i] + k for i in range(n) if budget[i] > k]
                parts += [_segment_work(d, [(c, 1) for c in live]), _head_work(d, len(live), True)]
            lens = [lens[i] + obs[i] + budget[i] for i in range(n)]
            nbytes += sum(p[0] for p in parts)
            flops += sum(p[1] for p in parts)
        return {"bytes": nbytes, "flops": flops}
    append = case["kind"] == "append"
    new = _observations(case) if append else [1] * n
    a, b = _segment_work(d, list(zip(_contexts(case), new))), _head_work(d, n, not append)
    extra = 4 * n * d["vocab"] if append else 0
    return {"bytes": a[0] + b[0] + extra, "flops": a[1] + b[1]}


def tolerance(case):
    # Activations enter every product as fp16 and cached keys/values are fp16 or bf16 (fp32 accumulation): logits of two
    # correct implementations differ by some 1e-3 (fp16 pages) to 1e-2 (bf16 pages) of their root mean square.
    rel = 1e-2 if case["kv"] == "f16" else 2e-2
    return {"rel": rel, "max": 10 * rel, "differ": 0.005}
