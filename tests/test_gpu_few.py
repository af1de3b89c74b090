"""The one-kernel decode step for up to eight games (csrc/step_few.cuh) against the kernel-per-operation step of the same
context.  The latter is what a step takes while kernel classes are being timed (spiral_profile); it is itself compared with the
oracle by the other parity tests, as this path is wherever they decode eight games or fewer.

Tolerance: both paths round the same activations to fp16 and the same keys and values to the cache's type and add in fp32 in
different orders, so their logits differ by what a flipped rounding here and there makes of them: a part of the 1e-2 that either
may be away from the oracle.  4e-3 of the root mean square (measured: 4e-4 to 2e-3), keys and values of the new token 2e-3."""
import pytest
import torch

import synth
from harness import TOL_REL_RMS, Pair

pytestmark = pytest.mark.gpu

REL, REL_KV = 0.4 * TOL_REL_RMS, 2e-3


def _step_both(pair, lens, seed, scale=None):
    """One step for games that hold lens[i] tokens, on either path: (logits, the new tokens' cache bytes, launches) of each."""
    sp, desc, n = pair.sp, pair.desc, len(lens)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    pair.pool.zero_()
    games = list(range(n))[::-1]
    for layer in range(desc["n_layers"]):
        for g, k in zip(games, lens):
            if k == 0:
                continue
            kv = [torch.empty(k, desc["n_kv_heads"], desc["head_dim"], device="cuda").uniform_(-2, 2, generator=gen).to(pair.kv_dtype) for _ in range(2)]
            sp.spiral_kv_load(pair.ctx, pair.kv, g, layer, kv[0], kv[1])
    tok_in = torch.randint(0, desc["vocab"], (n,), dtype=torch.int32, device="cuda", generator=gen)
    noise = torch.zeros(n, desc["vocab"], device="cuda")
    tok_out = torch.empty(n, dtype=torch.int32, device="cuda")
    before = pair.pool.clone()
    out = []
    for timed in (1, 0, 0):
        sp.spiral_profile(pair.ctx, timed)
        pair.pool.copy_(before)
        logits = torch.empty(n, desc["vocab"], device="cuda")
        l0 = sp.spiral_launch_count(pair.ctx)
        sp.spiral_decode_step(pair.ctx, pair.kv, games, tok_in, noise, 1.0, tok_out, logits)
        torch.cuda.synchronize()
        launches = sp.spiral_launch_count(pair.ctx) - l0
        assert sp.spiral_last_status(pair.ctx) == (0, 0)
        out.append((logits, (pair.pool.view(pair.kv_dtype).float() - before.view(pair.kv_dtype).float()), launches))
        sp.spiral_kv_truncate(pair.kv, games[::-1], lens[::-1])          # (last first: the same pages are handed out again)
    assert torch.equal(out[1][0], out[2][0]) and torch.equal(out[1][1], out[2][1])      # nothing depends on which CTA is first
    return out[0], out[1]


def _close(a, b, rel):
    return float((a.double() - b.double()).norm() / a.double().norm()) <= rel


@pytest.mark.parametrize("name,over,lens,bf16", [
    ("tiny", {}, [0], False),                                                   # the first token of an empty game
    ("tiny_qknorm", {}, [15, 16, 17, 31], False),                               # last, first and second row of a page
    ("tiny_qknorm", {}, [1, 600, 3, 250, 16, 48, 2, 90], True),                 # eight games, items shared by CTAs
    ("tiny_bias", {}, [33, 0, 400], False),
    ("tiny", dict(n_q_heads=8, n_kv_heads=1, head_dim=128), [700, 20], False),  # 8 heads per KV head, head_dim 128
    ("tiny", dict(n_q_heads=7, n_kv_heads=1, head_dim=64, d_model=448), [64, 65, 5, 6, 7], True),
    ("tiny", dict(n_q_heads=16, n_kv_heads=16, head_dim=64, d_model=1024, d_ff=5000), [40, 41, 42, 43, 44, 45, 46, 47], False),
    ("qwen3_4b", dict(n_layers=2), [900], False),                               # an item over several CTAs
    ("qwen3_4b", dict(n_layers=2), [100, 31, 32, 33, 500, 1], False),
    ("llama31_8b", dict(n_layers=2, vocab=4096), [64, 1000, 17], True),
    ("qwen25_7b", dict(n_layers=2, vocab=4096), [5, 80, 1500, 16, 48, 47, 49, 300], False),
])
def test_one_kernel_step_against_kernel_per_operation(name, over, lens, bf16):
    desc = synth.shape(name, **over)
    pair = Pair(desc, max_batch=8, max_ctx=1600, n_games=8, kv_bf16=bf16, generate_on_gpu=desc["d_model"] > 1024)
    try:
        per_op, one = _step_both(pair, lens, 5)
        assert one[2] == 2 and per_op[2] > 2        # the layers and the LM head
        assert _close(per_op[0], one[0], REL)
        assert _close(per_op[1], one[1], REL_KV)
    finally:
        pair.close()


@pytest.mark.parametrize("factor", [2.0 ** -14, 2.0 ** 10])
def test_rows_that_change_their_size(factor):
    """Activations are stored times a power of two that follows the row's previous norm.  Embeddings 2^14 times smaller (2^10
    times larger) than the layers' output make the residual grow (or, relative to it, hardly change) past the window in which
    that is exact; the rows then have to be stored again."""
    desc = synth.shape("tiny_qknorm", tied_embed=0)
    w = synth.perturb_gains(synth.make_weights(desc))
    w["embed"] = (w["embed"].float() * factor).to(torch.bfloat16)
    pair = Pair(desc, max_batch=8, max_ctx=128, n_games=8, weights_cpu=w)
    try:
        per_op, one = _step_both(pair, [20, 64, 3], 9)
        assert one[2] == 2
        assert _close(per_op[0], one[0], REL)
        assert _close(per_op[1], one[1], REL_KV)
    finally:
        pair.close()


def test_nine_games_take_the_kernels_per_operation():
    desc = synth.shape("tiny_qknorm")
    pair = Pair(desc, max_batch=9, max_ctx=64, n_games=9)
    try:
        per_op, other = _step_both(pair, [5 + i for i in range(9)], 3)
        assert other[2] == per_op[2] > 2
        assert torch.equal(per_op[0], other[0])
    finally:
        pair.close()
