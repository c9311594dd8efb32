"""Attention kernels through whole decode steps: prompt lengths around the edges of key tiles and 16-key groups, query rows around
the edges of a 128-row tile, suffix depths around the edges of suffix tiles, against the oracle's full recompute."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle.decoder import Decoder
from paper_2605_26606_b200 import binding as B
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import RolloutEngine

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,prompt,rows,depth,half", [(wl.SMALL_BF16, 1, 1, 2, True), (wl.SMALL_BF16, 16, 63, 18, True),
                                                          (wl.SMALL_QKNORM_BF16, 63, 64, 5, True), (wl.SMALL_BF16, 64, 65, 3, False),
                                                          (wl.SMALL_QKNORM_BF16, 65, 2, 34, True), (wl.SMALL_BF16, 191, 129, 3, True),
                                                          (wl.SMALL_BF16, 600, 3, 66, True), (wl.TINY_BF16, 130, 40, 18, True),
                                                          # prompts past the length up to which few rows read them themselves
                                                          (wl.SMALL_BF16, 1024, 3, 17, True), (wl.SMALL_BF16, 1025, 3, 17, True), (wl.TINY_BF16, 1100, 20, 17, True)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_decode_logits_at_attention_tile_edges(cuda_device, model, prompt, rows, depth, half):
    ensure_built()
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=2, prompt_len_lo=prompt, prompt_len_hi=prompt, group_size=rows,
                            n_pilot=rows, max_new=depth + 1, cap_lo=depth + 1, cap_hi=depth + 1, data_seed=5, forced_explicit=None)
    weights = wl.gen_weights(model, seed=4, threads=4, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=2 * rows, max_prefill_tokens=2 * prompt, half_gemm=half)
    steps = sorted({0, depth // 2, depth - 1})
    eng.record_pilot_logits = {s: None for s in steps}
    got = eng.pilot_commit_step(w, batch)
    dec = Decoder(model, weights)
    for p, i in {(0, 0), (1, rows - 1), (1, rows // 2)}:
        toks = got["tokens"][p][i]
        pt = batch.prompt_tokens[batch.prompt_offsets[p]:batch.prompt_offsets[p + 1]]
        want = dec.forward_full(np.concatenate([pt, toks[:-1]]))
        for s in steps:
            logits, rp, rr = eng.record_pilot_logits[s]
            row = int(np.flatnonzero((rp == p) & (rr == i))[0])
            assert np.max(np.abs(logits[row].cpu().numpy() - want[prompt + s])) <= 5e-2, (p, i, s)


@pytest.mark.parametrize("model,prompt,rows,depth,half", [(wl.SMALL_BF16, 600, 150, 3, True), (wl.SMALL_QKNORM_BF16, 40, 150, 66, True),
                                                          (wl.SMALL_BF16, 300, 160, 35, False), (wl.SMALL_BF16, 64, 300, 18, True),
                                                          (wl.TINY_BF16, 130, 160, 34, True)], ids=lambda v: getattr(v, "name", str(v)))
def test_decode_logits_where_suffix_items_are_claimed(cuda_device, model, prompt, rows, depth, half):
    """600 to 1,200 (row, KV head) items, where B200 has room for 592 pairs of warps: four to an item up to one and a half rounds of pairs, two beyond.
    Suffixes of one to five tiles, so some warps have none; long prompts beside short suffixes, so items are finished before the shared-prefix
    records are there.  (Fewer items, other head counts and ragged caps: below.)"""
    test_decode_logits_at_attention_tile_edges(cuda_device, model, prompt, rows, depth, half)


_heads = lambda base, hq, hkv: dataclasses.replace(base, name=f"{base.name}-{hq}-{hkv}", n_q_heads=hq, n_kv_heads=hkv)


@pytest.mark.parametrize("model,rows,prompts,caps", [(wl.SMALL_BF16, 150, (600, 1000), (2, 20)),                    # 640 items
                                                     (wl.SMALL_QKNORM_BF16, 110, (700, 1500), (3, 70)),              # 448
                                                     (_heads(wl.SMALL_BF16, 12, 2), 300, (500, 900), (2, 24)),       # 1,280; six query heads per KV head
                                                     (_heads(wl.SMALL_QKNORM_BF16, 32, 8), 30, (500, 900), (20, 40)),   # 512; four
                                                     (_heads(wl.SMALL_BF16, 16, 2), 160, (400, 800), (2, 40)),       # 640; eight
                                                     (_heads(wl.TINY_BF16, 16, 2), 110, (300, 700), (2, 50)),        # 448, head_dim 64
                                                     (_heads(wl.TINY_BF16, 8, 2), 160, (300, 700), (2, 50))],        # 640, head_dim 64
                         ids=lambda v: getattr(v, "name", str(v)))
def test_claimed_suffix_items_give_the_same_bits_whenever_they_finish(cuda_device, model, rows, prompts, caps):
    """Ragged groups of long prompts beside short suffixes: some items are finished before the shared-prefix records are there and are
    merged later, others at once, and which is a matter of timing.  Tokens, log-probabilities and every K and V (layer 1's are made of layer
    0's attention outputs) are the same in every run, and with the kernels in plain stream order (mask 0: all merged at once); a few
    rollouts are compared with the oracle."""
    ensure_built()
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=2, prompt_len_lo=prompts[0], prompt_len_hi=prompts[1], group_size=rows,
                            n_pilot=rows, max_new=caps[1], cap_lo=caps[0], cap_hi=caps[1], data_seed=5, forced_explicit=None)
    weights = wl.gen_weights(model, seed=4, threads=4, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=2 * rows, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    eng.collect_logprobs = True
    eng.pilot_commit_step(w, batch)                       # (the arena exists now)
    want = None
    for mask in (0, 63, 63, 63, 63, 63):
        B.pc_set_dependent_launch(eng.ctx, mask)
        eng.suffix_kv.zero_()
        out = eng.pilot_commit_step(w, batch)
        got = (eng.tokens.clone(), eng.logprobs.clone(), eng.suffix_kv.view(torch.int16).clone())
        want = want or got
        for name, a, b in zip(("tokens", "log-probabilities", "K and V"), got, want):
            assert torch.equal(a, b), (mask, name)
    logp, dec = want[1].cpu().numpy().reshape(2, rows, w.max_new), Decoder(model, weights)
    for p, i in {(0, 0), (1, rows - 1), (1, rows // 2)}:
        toks = out["tokens"][p][i]
        pt = batch.prompt_tokens[batch.prompt_offsets[p]:batch.prompt_offsets[p + 1]]
        logits = dec.forward_full(np.concatenate([pt, toks[:-1]]))[len(pt) - 1:].astype(np.float64)
        ref = logits[np.arange(len(toks)), toks] - np.logaddexp.reduce(logits, axis=1)
        assert np.max(np.abs(logp[p, i, :len(toks)] - ref)) <= 1e-1        # two logits' worth of 5e-2


@pytest.mark.parametrize("model,prompt,rows", [(wl.SMALL_BF16, 4096, 3), (wl.SMALL_BF16, 4097, 3), (wl.TINY_BF16, 1280, 20), (wl.TINY_BF16, 1281, 20),
                                               (wl.SMALL_QKNORM_BF16, 1281, 20), (wl.SMALL_BF16, 1025, 50)], ids=lambda v: getattr(v, "name", str(v)))
def test_decode_logits_on_both_sides_of_the_longest_prompt_rows_read_themselves(cuda_device, model, prompt, rows):
    """4,096 tokens with four CTAs to a (row, KV head), 1,280 with two, 1,024 with one."""
    test_decode_logits_at_attention_tile_edges(cuda_device, model, prompt, rows, 17, True)


def test_few_rows_read_a_long_prompt_once_per_group(cuda_device):
    """Prompts of 40 tokens and one of 1,500: on average they are short enough for every row to read its own, but the long one is not.  The
    step then has the shared-prefix kernel, one launch per layer more than a step of short prompts; logits against the oracle."""
    ensure_built()
    model, rows, steps = wl.SMALL_BF16, 30, 4
    weights = wl.gen_weights(model, seed=4, threads=4, gain_jitter=0.1)
    eng = RolloutEngine(model, weights, max_rows=4 * rows, max_prefill_tokens=1700)
    eng.use_graphs = False
    dec, launches = Decoder(model, weights), {}
    for longest in (40, 1500):
        w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=4, prompt_len_lo=longest, prompt_len_hi=longest, group_size=rows,
                                n_pilot=rows, max_new=steps + 1, cap_lo=steps + 1, cap_hi=steps + 1, data_seed=5, forced_explicit=None)
        batch = wl.gen_batch(w)
        lens = np.array([40, 40, longest, 40], np.int32)
        keep = np.concatenate([np.arange(o, o + n) for o, n in zip(batch.prompt_offsets, lens)])
        batch = dataclasses.replace(batch, prompt_lens=lens, prompt_offsets=np.r_[0, np.cumsum(lens)].astype(np.int32), prompt_tokens=batch.prompt_tokens[keep])
        eng.load_batch(w, batch)
        eng.prefill()
        eng.record_pilot_logits = {steps - 1: None}
        before = B.pc_launch_count()
        prompts, rollouts = np.repeat(np.arange(4), rows), np.tile(np.arange(rows), 4)
        eng.run_stage(prompts, rollouts, record_logits=eng.record_pilot_logits)
        launches[longest] = B.pc_launch_count() - before
        eng.check_error_flag()
        logits = eng.record_pilot_logits[steps - 1][0].cpu().numpy()
        toks = eng.tokens.cpu().numpy().reshape(4, rows, w.max_new)
        for p in (1, 2):
            pt = batch.prompt_tokens[batch.prompt_offsets[p]:batch.prompt_offsets[p + 1]]
            want = dec.forward_full(np.concatenate([pt, toks[p, 3, :-1]]), last_only=True)[0]
            assert np.max(np.abs(logits[p * rows + 3] - want)) <= 5e-2, p
    assert launches[1500] - launches[40] == steps * model.n_layers, launches


def test_probabilities_round_below_their_maximum(cuda_device):
    """Half rounds a probability finest just below the row's largest, which is 1 and exact.  64 keys of one kind, then 200 whose score is
    higher by log2(1.00044): as 1.00044 they would round to 1, a relative error of 4.4e-4 in every output; as 1, beside 0.99956 for
    the others, they lose nothing.  Layer 1's V reads the outputs back: three half roundings each (rms 2^-11 / sqrt 3, zero mean), so the
    mean error over 256 of them has a deviation of 3e-5 at most."""
    ensure_built()
    model = dataclasses.replace(wl.SMALL_QKNORM_BF16, name="two-kinds-of-keys", qk_norm=False, tied_embed=False, rms_eps=1e-12)
    weights, rng = wl.gen_weights(model, seed=4, threads=4), np.random.default_rng(0)
    d, hd = model.d_model, model.head_dim
    zero = {n: np.zeros_like(weights[n]) for n in weights.names() if n.startswith("layers.") and "norm" not in n}
    e = np.zeros((model.vocab, d), np.float32)
    e[:, :128] = 2.0                                        # rms 1; the other coordinates receive the attention's outputs
    e[0, 0] = -2.0                                          # token 0: the first kind of key, any other: the second
    zero["layers.0.wq"][hd // 2 - 1::hd, 1] = 0.5           # the slowest rotary pair: q = 1 and k = -+ 0.00249 at every position
    zero["layers.0.wk"][hd // 2 - 1::hd, 0] = 0.001244
    c = (1 + rng.integers(0, 128, model.kv_dim) / 128).astype(np.float32)
    zero["layers.0.wv"][:, 0] = zero["layers.0.wv"][:, 1] = c / 4            # V = 0 for the first kind, c for the second
    zero["layers.0.wo"][128 + np.arange(384), np.arange(384)] = 0.25
    zero["layers.1.wv"][np.arange(256), 128 + np.arange(256)] = 1.0
    for name, a in {**zero, "embed": e}.items():
        weights.put(name, a, True)
    tokens = np.r_[np.zeros(64, np.int32), np.full(200, 7, np.int32)]
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=1, prompt_len_lo=264, prompt_len_hi=264, group_size=2, n_pilot=2,
                            max_new=2, cap_lo=2, cap_hi=2, data_seed=5, forced_explicit=None)
    batch = dataclasses.replace(wl.gen_batch(w), prompt_tokens=tokens)
    eng = RolloutEngine(model, weights, max_rows=2, max_prefill_tokens=264)
    eng.pilot_commit_step(w, batch)
    _, kv = Decoder(model, weights).forward_full(tokens, return_kv=True, last_only=True)
    got = eng.prompt_kv[1, 1, :, 263].contiguous().view(torch.float16).cpu().numpy().astype(np.float64).reshape(-1)
    want = kv[1][1][263].reshape(-1)
    off = float(np.mean(got / want - 1))
    print(f"mean relative error {off:.2e}")
    assert np.min(want) > 0.1 and abs(off) <= 1e-4, off
