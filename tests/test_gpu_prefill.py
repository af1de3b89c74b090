"""Dense context append (the tensor-core prefill path) against the oracle.

Between two turns the environment appends an observation of tens to hundreds of tokens to every
game's context.  When a call carries more new tokens than one decode-shaped step holds, the
library runs them as dense passes (256-token GEMM tiles, causal block attention).  The checks go
through what the path leaves behind: the logits after the last appended token and the logits of
the decode steps that follow, which read every key and value the append wrote.
"""
import time

import numpy as np
import pytest
import torch

import synth
from harness import TOL_MAX_ABS, TOL_REL_RMS, Pair, compare_logits
from test_gpu_parity import _check, _run_teacher_forced

pytestmark = pytest.mark.gpu


def _append(pair, games, new_tokens):
    """One spiral_prefill call on both sides; returns (worst max|delta|, worst rel rms) of the last-token logits."""
    sp, V = pair.sp, pair.desc["vocab"]
    flat = torch.tensor(sum(new_tokens, []), dtype=torch.int32).cuda()
    offs = np.concatenate([[0], np.cumsum([len(t) for t in new_tokens])]).tolist()
    last = torch.empty(len(games), V, dtype=torch.float32, device="cuda")
    sp.spiral_prefill(pair.ctx, pair.kv, games, flat, offs, last)
    last = last.cpu().numpy()
    worst_abs, worst_rms = 0.0, 0.0
    for i, g in enumerate(games):
        ref = pair.oracle.prefill(pair.oracle_cache(g), new_tokens[i])
        a, r = compare_logits(last[i], ref)
        worst_abs, worst_rms = max(worst_abs, a), max(worst_rms, r)
    return worst_abs, worst_rms


def _decode(pair, games, steps, seed):
    sp, V = pair.sp, pair.desc["vocab"]
    n = len(games)
    tok_out = torch.empty(n, dtype=torch.int32, device="cuda")
    logits = torch.empty(n, V, dtype=torch.float32, device="cuda")
    worst_abs, worst_rms = 0.0, 0.0
    for s in range(steps):
        tok_in = synth.token_ids(seed, 1000 + s, n, V, stream=synth.STREAM_TEACHER)
        noise = synth.gumbel_noise(seed, s, n, V)
        sp.spiral_decode_step(pair.ctx, pair.kv, games, tok_in.cuda(), noise.cuda(), 1.0, tok_out, logits)
        lg = logits.cpu().numpy()
        for i, g in enumerate(games):
            ref = pair.oracle.decode_step(pair.oracle_cache(g), int(tok_in[i]))
            a, r = compare_logits(lg[i], ref)
            worst_abs, worst_rms = max(worst_abs, a), max(worst_rms, r)
    return worst_abs, worst_rms


@pytest.mark.parametrize("shape_name,overrides,chunk", [
    ("tiny_qknorm", {}, 256),                                        # 2 query heads per KV head, head_dim 64
    ("tiny_bias", {}, 512),                                          # 4 per KV head, QKV bias
    ("tiny", dict(n_q_heads=8, n_kv_heads=1, head_dim=128), 256),    # 8 per KV head, head_dim 128
    ("tiny", dict(n_q_heads=2, n_kv_heads=2, head_dim=128), 0),      # no grouping; one pass
    ("tiny", dict(n_q_heads=7, n_kv_heads=1, head_dim=64, d_model=448), 256),   # a group that does not divide 128 rows
])
def test_dense_append_in_several_passes(monkeypatch, shape_name, overrides, chunk):
    """Five games, ragged lengths (one token, below a page, page-aligned, several tiles), a pass size
    that cuts games in the middle: the later pass must find the earlier pass's keys in the pages."""
    if chunk:
        monkeypatch.setenv("SPIRAL_PREFILL_CHUNK", str(chunk))
    desc = synth.shape(shape_name, **overrides)
    lens = [300, 1, 129, 256, 40, 13]
    pair = Pair(desc, max_batch=16, max_ctx=320, n_games=8)
    try:
        games = [5, 0, 3, 7, 1, 2]
        prompts = [synth.token_ids(synth.MASTER_SEED, 900 + i, lens[i], desc["vocab"]).tolist() for i in range(len(games))]
        res = _run_teacher_forced(pair, games, prompts, 4, synth.MASTER_SEED + 21)
        print(shape_name, overrides, "max|d| %.2e rel-rms %.2e agree %.4f" % res[:3], res[3])
        _check(*res)
    finally:
        pair.close()


def test_dense_append_onto_existing_context():
    """Turn structure: append, decode a few tokens, append again at positions that are not page
    aligned, decode again; some games sit out the second append."""
    desc = synth.shape("tiny_qknorm")
    n_games = 6
    pair = Pair(desc, max_batch=16, max_ctx=256, n_games=n_games)
    try:
        V = desc["vocab"]
        games = list(range(n_games))
        obs = [synth.token_ids(11, g, 21 + 7 * g, V).tolist() for g in games]
        launches0 = pair.sp.spiral_launch_count(pair.ctx)
        worst = [_append(pair, games, obs)]
        # one pass = eight kernels per layer plus embedding, row gather, final norm and head -- not one
        # decode-shaped step per 16 tokens
        assert pair.sp.spiral_launch_count(pair.ctx) - launches0 <= 8 * desc["n_layers"] + 6
        worst.append(_decode(pair, games, 3, 31))
        later = [4, 1, 2]
        obs2 = [synth.token_ids(12, g, 50 + 30 * i, V).tolist() for i, g in enumerate(later)]
        worst.append(_append(pair, later, obs2))
        worst.append(_decode(pair, games, 3, 32))
        rc, detail = pair.sp.spiral_last_status(pair.ctx)
        assert rc == 0, detail
        print("append/decode/append/decode:", worst)
        assert max(w[0] for w in worst) <= TOL_MAX_ABS
        assert max(w[1] for w in worst) <= TOL_REL_RMS
    finally:
        pair.close()


@pytest.mark.parametrize("attn", ["mma", "tc1"])
def test_other_attention_kernels_of_the_append_still_available(monkeypatch, attn):
    """SPIRAL_APPEND_ATTN=mma runs the append's attention on mma.sync instead of tcgen05, =tc1 on tcgen05
    with one query tile per CTA and two CTAs per SM: same bars."""
    monkeypatch.setenv("SPIRAL_APPEND_ATTN", attn)
    monkeypatch.setenv("SPIRAL_PREFILL_CHUNK", "256")
    for name, over in [("tiny_bias", {}), ("tiny", dict(n_q_heads=7, n_kv_heads=1, head_dim=128, d_model=448))]:
        desc = synth.shape(name, **over)
        pair = Pair(desc, max_batch=16, max_ctx=320, n_games=4)
        try:
            lens = [300, 17, 130]
            prompts = [synth.token_ids(synth.MASTER_SEED, 950 + i, lens[i], desc["vocab"]).tolist() for i in range(3)]
            res = _run_teacher_forced(pair, [3, 0, 1], prompts, 3, synth.MASTER_SEED + 23)
            _check(*res)
        finally:
            pair.close()


def test_step_shaped_append_still_available(monkeypatch):
    """SPIRAL_PREFILL_DENSE=0 keeps the append on decode-shaped steps (the path of calls that one step holds
    and of contexts without weight copies): same result within the tolerances."""
    monkeypatch.setenv("SPIRAL_PREFILL_DENSE", "0")
    desc = synth.shape("tiny_qknorm")
    pair = Pair(desc, max_batch=24, max_ctx=160, n_games=3)
    try:
        games = [2, 0]
        prompts = [synth.token_ids(synth.MASTER_SEED, 300 + i, 97 - 40 * i, desc["vocab"]).tolist() for i in range(2)]
        res = _run_teacher_forced(pair, games, prompts, 4, synth.MASTER_SEED + 9)
        _check(*res)
    finally:
        pair.close()


def test_dense_append_full_width():
    """Qwen3-4B width (d_model 2560, 32/8 heads of 128, d_ff 9728, 151 936-row head) at three layers,
    so that the oracle can afford observations of the paper's size (hundreds of tokens): two rounds
    of append + decode on three games."""
    desc = synth.shape("qwen3_4b", n_layers=3)
    t0 = time.time()
    pair = Pair(desc, max_batch=16, max_ctx=704, n_games=3, gains=False, generate_on_gpu=True)
    try:
        V = desc["vocab"]
        games = [0, 1, 2]
        obs = [synth.token_ids(13, g, [300, 170, 45][g], V).tolist() for g in games]
        worst = [_append(pair, games, obs)]
        worst.append(_decode(pair, games, 2, 41))
        obs2 = [synth.token_ids(14, g, [40, 300, 10][g], V).tolist() for g in games]
        worst.append(_append(pair, games, obs2))
        worst.append(_decode(pair, games, 2, 42))
        rc, detail = pair.sp.spiral_last_status(pair.ctx)
        assert rc == 0, detail
        print("full width:", worst, "%.0fs" % (time.time() - t0))
        assert max(w[0] for w in worst) <= TOL_MAX_ABS
        assert max(w[1] for w in worst) <= TOL_REL_RMS
    finally:
        pair.close()


@pytest.mark.parametrize("attn", ["tc", "mma"])
def test_dense_append_long_contexts(monkeypatch, attn):
    """Contexts of a few thousand tokens (hundreds of pages per game: the attention kernels' page-id
    windows and ring phases wrap many times), appended in two rounds with decode steps between."""
    monkeypatch.setenv("SPIRAL_APPEND_ATTN", attn)
    desc = synth.shape("tiny_bias")
    pair = Pair(desc, max_batch=16, max_ctx=2500, n_games=2)
    try:
        V = desc["vocab"]
        games = [1, 0]
        obs = [synth.token_ids(19, g, [2049, 700][i], V).tolist() for i, g in enumerate(games)]
        worst = [_append(pair, games, obs)]
        worst.append(_decode(pair, games, 2, 51))
        obs2 = [synth.token_ids(20, g, [40, 301][i], V).tolist() for i, g in enumerate(games)]
        worst.append(_append(pair, games, obs2))
        worst.append(_decode(pair, games, 2, 52))
        rc, detail = pair.sp.spiral_last_status(pair.ctx)
        assert rc == 0, detail
        print("long contexts (%s):" % attn, worst)
        assert max(w[0] for w in worst) <= TOL_MAX_ABS
        assert max(w[1] for w in worst) <= TOL_REL_RMS
    finally:
        pair.close()


@pytest.mark.parametrize("overrides,lens", [
    ({}, [44, 1, 45, 130, 89]),                                                      # 2 heads per group: 44 positions per block
    (dict(n_q_heads=7, n_kv_heads=1, head_dim=64, d_model=448), [12, 13, 300, 25]),  # 12 per block, rows left over
    (dict(n_q_heads=8, n_kv_heads=1, head_dim=128), [11, 12, 64, 200]),              # 11 per block
    (dict(n_q_heads=2, n_kv_heads=2, head_dim=128), [88, 89, 176, 177]),             # 88 per block
])
def test_dense_append_with_bf16_pages(overrides, lens):
    """bf16 pages take the mma.sync attention with queries and weights in two bf16 parts; lengths around its query blocks."""
    desc = synth.shape("tiny", **overrides)
    pair = Pair(desc, max_batch=8, max_ctx=320, n_games=8, kv_bf16=True)
    try:
        games = [5, 0, 3, 7, 1][:len(lens)]
        prompts = [synth.token_ids(synth.MASTER_SEED, 970 + i, lens[i], desc["vocab"]).tolist() for i in range(len(games))]
        launches0 = pair.sp.spiral_launch_count(pair.ctx)
        res = _run_teacher_forced(pair, games, prompts, 3, synth.MASTER_SEED + 25)
        assert pair.sp.spiral_launch_count(pair.ctx) - launches0 < 6 * (9 * desc["n_layers"] + 6)     # dense, not 8 tokens a step
        print(overrides, "max|d| %.2e rel-rms %.2e agree %.4f" % res[:3], res[3])
        _check(*res)
    finally:
        pair.close()


@pytest.mark.parametrize("overrides,new", [
    ({}, [1, 40, 129]),                                                    # 128 positions per query block
    (dict(n_q_heads=7, n_kv_heads=1, head_dim=64, d_model=448), [37, 3]),  # rows left over in both tiles
    (dict(n_q_heads=8, n_kv_heads=1, head_dim=128), [33, 16, 50]),         # 32 positions per query block
])
def test_dense_append_cut_along_the_keys(overrides, new):
    """Few query blocks behind long contexts: several CTAs share one, at cuts inside the context and inside the new tokens."""
    desc = synth.shape("tiny", **overrides)
    pair = Pair(desc, max_batch=2, max_ctx=1300, n_games=2)
    try:
        V = desc["vocab"]
        worst = [_append(pair, [1], [synth.token_ids(41, 0, 700, V).tolist()])]
        for i, k in enumerate(new):
            worst.append(_append(pair, [1, 0], [synth.token_ids(42, i, k, V).tolist(), synth.token_ids(43, i, 190 + i, V).tolist()]))
        worst.append(_decode(pair, [0, 1], 2, 44))
        rc, detail = pair.sp.spiral_last_status(pair.ctx)
        assert rc == 0, detail
        print("cut along the keys:", overrides, worst)
        assert max(w[0] for w in worst) <= TOL_MAX_ABS
        assert max(w[1] for w in worst) <= TOL_REL_RMS
    finally:
        pair.close()


@pytest.mark.parametrize("total", [33, 256, 257, 1024, 1025, 2049])
def test_dense_append_at_the_edges_of_its_gemms(total):
    """Token counts around a 256-row tile, around the limits up to which partial sums and narrow tiles are considered, and
    11 k blocks (d_ff 688) in stages of two."""
    desc = synth.shape("tiny")
    pair = Pair(desc, max_batch=8, max_ctx=1200, n_games=3)
    try:
        V, games = desc["vocab"], [2, 0, 1]
        lens = [total // 2, total // 3, total - total // 2 - total // 3]
        worst = [_append(pair, games, [synth.token_ids(51, i, k, V).tolist() for i, k in enumerate(lens)])]
        worst.append(_decode(pair, games, 2, 52))
        rc, detail = pair.sp.spiral_last_status(pair.ctx)
        assert rc == 0, detail
        print("append of", total, worst)
        assert max(w[0] for w in worst) <= TOL_MAX_ABS
        assert max(w[1] for w in worst) <= TOL_REL_RMS
    finally:
        pair.close()


@pytest.mark.parametrize("overrides,lens", [
    ({}, [64, 3, 129, 40]),                                                          # 2 heads per group, head_dim 64
    (dict(n_q_heads=8, n_kv_heads=2, head_dim=128), [33, 50, 16, 100]),              # 32 positions per query block
    (dict(n_q_heads=7, n_kv_heads=1, head_dim=64, d_model=448), [37, 18, 19, 70]),   # a group that does not divide 128 rows
])
def test_dense_append_in_place_of_steps_loses_no_precision(monkeypatch, overrides, lens):
    """A context for few games appends in dense passes what it would otherwise append in decode-shaped steps, whose queries
    and softmax weights are in two parts (22 bits).  One layer without an MLP, so that the attention is what differs.
    Bound: a value that differs by d before it is rounded to fp16 (steps of u = 2^-10.5) differs by sqrt(d u) rms after it,
    because a share d / u of the values rounds the other way.  Another order of sums, d = 2^-20, gives 2^-15.3 in the cached
    keys and values, that 2^-12.9 in the attention's output, and that, half of the residual stream, 2^-12.2 in the LM
    head's input; 2^-12 is allowed.  A single fp16 rounding of queries and weights gave 2^-11.5 to 2^-11.2 here."""
    desc = synth.shape("tiny_qknorm", n_layers=1, **overrides)
    w = synth.perturb_gains(synth.make_weights(desc))
    w["w_down"][0].zero_()
    V, out = desc["vocab"], {}
    prompts = [synth.token_ids(61, i, k, V).tolist() for i, k in enumerate(lens)]
    games = [3, 0, 2, 1]
    for dense in ("0", "1"):
        monkeypatch.setenv("SPIRAL_PREFILL_DENSE", dense)
        pair = Pair(desc, max_batch=8, max_ctx=320, n_games=4, weights_cpu=w)
        try:
            rows = []
            for part in range(2):               # onto nothing, then onto the cached first half
                new = [p[:len(p) // 2] if part == 0 else p[len(p) // 2:] for p in prompts]
                flat = torch.tensor(sum(new, []), dtype=torch.int32).cuda()
                offs = np.concatenate([[0], np.cumsum([len(t) for t in new])]).tolist()
                last = torch.empty(4, V, dtype=torch.float32, device="cuda")
                pair.sp.spiral_prefill(pair.ctx, pair.kv, games, flat, offs, last)
                rows.append(last.cpu().numpy().astype(np.float64))
            out[dense] = np.concatenate(rows)
        finally:
            pair.close()
    rel = np.sqrt(((out["0"] - out["1"]) ** 2).sum() / (out["0"] ** 2).sum())
    print(overrides, "dense against steps: rel %.2e" % rel)
    assert rel <= 2.0 ** -12


@pytest.mark.parametrize("d_ff", [688, 200, 704])
def test_first_appends_on_a_side_stream(d_ff):
    """Calls that make or enlarge the append workspace, on a stream that the legacy default stream does not wait for: with a
    d_ff that is no multiple of 64 the activations are cleared before they are written."""
    desc = synth.shape("tiny", d_ff=d_ff)
    pair = Pair(desc, max_batch=8, max_ctx=1500, n_games=2)
    try:
        V, stream = desc["vocab"], torch.cuda.Stream()
        for i, k in enumerate((33, 300, 900)):
            new = [synth.token_ids(91 + i, g, k // 2 + g, V).tolist() for g in range(2)]
            flat = torch.tensor(sum(new, []), dtype=torch.int32).cuda()
            last = torch.empty(2, V, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            pair.sp.spiral_prefill(pair.ctx, pair.kv, [1, 0], flat, [0, len(new[0]), len(new[0]) + len(new[1])], last, stream)
            stream.synchronize()
            for j, g in enumerate((1, 0)):
                a, r = compare_logits(last[j].cpu().numpy(), pair.oracle.prefill(pair.oracle_cache(g), new[j]))
                assert a <= TOL_MAX_ABS and r <= TOL_REL_RMS
    finally:
        pair.close()


def test_shorter_appends_do_not_allocate_again():
    """What a call allocates serves every call with no more tokens, also one whose GEMM plans leave more partial sums or whose
    attention is cut along the keys: at this shape 1024 tokens leave 6 MB more of them than 1792."""
    desc = synth.shape("llama31_8b", n_layers=1, vocab=4096)
    V = desc["vocab"]
    last = torch.empty(2, V, dtype=torch.float32, device="cuda")
    tokens = synth.token_ids(95, 0, 2048, V).cuda()
    for measured in (False, True):                   # (the first context has the kernels loaded, which takes memory, too)
        pair = Pair(desc, max_batch=16, max_ctx=2100, n_games=2, gains=False, generate_on_gpu=True)
        try:
            sp = pair.sp

            def append(k):
                sp.spiral_prefill(pair.ctx, pair.kv, [0, 1], tokens[:k], [0, k // 2, k], last)
                torch.cuda.synchronize()

            append(1792)                             # the largest
            append(40)                               # few query blocks behind 896 tokens: cut
            free = torch.cuda.mem_get_info()[0]
            sp.spiral_kv_truncate(pair.kv, [0, 1], [0, 0])
            for k in (1024, 1700, 640, 300, 172, 40, 17):
                append(k)
                assert not measured or torch.cuda.mem_get_info()[0] == free, k
                sp.spiral_kv_truncate(pair.kv, [0, 1], [0, 0])
            assert sp.spiral_last_status(pair.ctx)[0] == 0
        finally:
            pair.close()


@pytest.mark.parametrize("overrides,room,games,each", [
    ({}, 20 << 20, 8, 500),
    (dict(d_model=1024, n_q_heads=16, d_ff=8192), 6 << 20, 2, 40),       # 256 rows of workspace: more than 10 MB
])
def test_append_on_a_gpu_with_little_room(overrides, room, games, each):
    """Where the workspace of one long pass does not fit, the call takes shorter passes; where none fits, steps."""
    desc = synth.shape("tiny", **overrides)
    warm = Pair(desc, max_batch=24, max_ctx=600, n_games=games)          # (loads the kernels)
    pair = Pair(desc, max_batch=24, max_ctx=600, n_games=games)
    hog = None
    try:
        V = desc["vocab"]
        _append(warm, list(range(games)), [synth.token_ids(96, g, 40, V).tolist() for g in range(games)])
        _decode(warm, list(range(games)), 1, 98)
        new = [synth.token_ids(97, g, each + g, V).tolist() for g in range(games)]
        flat = torch.tensor(sum(new, []), dtype=torch.int32).cuda()
        offs = np.concatenate([[0], np.cumsum([len(t) for t in new])]).tolist()
        last = torch.empty(games, V, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        pair.sp.spiral_prefill(pair.ctx, pair.kv, list(range(games)), flat, offs, last)
        torch.cuda.synchronize()
        del hog
        for g in range(games):
            a, r = compare_logits(last[g].cpu().numpy(), pair.oracle.prefill(pair.oracle_cache(g), new[g]))
            assert a <= TOL_MAX_ABS and r <= TOL_REL_RMS
        assert pair.sp.spiral_last_status(pair.ctx)[0] == 0
    finally:
        warm.close()
        pair.close()
        torch.cuda.empty_cache()
