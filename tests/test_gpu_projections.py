"""The weight-on-lanes projections (gemm_wt.cuh) through whole decode steps: row counts around the edges of their tiles, K splits
and epilogue chunks, against the oracle's full recompute."""
import dataclasses

import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2605_26606_b200 import binding as B
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import RolloutEngine

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu

WIDE = dataclasses.replace(wl.SMALL_BF16, name="wide-bf16", d_model=1536, n_q_heads=12, n_kv_heads=2, d_ff=1088, vocab=1003)


NARROW = dataclasses.replace(wl.SMALL_BF16, name="narrow-bf16", d_model=192)        # one and a half feature tiles


@pytest.mark.parametrize("model,rows,half", [(wl.SMALL_BF16, 1, True), (NARROW, 33, True), (NARROW, 33, False), (wl.SMALL_BF16, 15, True), (wl.SMALL_QKNORM_BF16, 17, True),
                                             (WIDE, 33, True), (WIDE, 129, True), (WIDE, 257, True), (WIDE, 300, False),
                                             (wl.SMALL_QKNORM_BF16, 47, False), (WIDE, 1100, True)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_decode_logits_at_tile_edges(cuda_device, model, rows, half):
    ensure_built()
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=1, prompt_len_lo=5, prompt_len_hi=5, group_size=rows,
                            n_pilot=rows, max_new=4, cap_lo=4, cap_hi=4, data_seed=3, forced_explicit=None)
    weights = wl.gen_weights(model, seed=2, threads=4, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=rows, max_prefill_tokens=5, half_gemm=half)
    eng.record_pilot_logits = {1: None, 2: None}
    got = eng.pilot_commit_step(w, batch)
    dec = Decoder(model, weights)
    for i in sorted({0, rows - 1, rows // 2, rows // 3}):
        toks = got["tokens"][0][i]
        want = dec.forward_full(np.concatenate([batch.prompt_tokens, toks[:-1]]))
        for s in (1, 2):
            logits, _, rr = eng.record_pilot_logits[s]
            row = int(np.flatnonzero(rr == i)[0])
            assert np.max(np.abs(logits[row].cpu().numpy() - want[5 + s])) <= 5e-2, (i, s)


@pytest.mark.parametrize("prompt_len", [255, 4200])
def test_logits_after_a_prefill_of_many_row_tiles(cuda_device, prompt_len):
    ensure_built()
    model = wl.SMALL_BF16
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=1, prompt_len_lo=prompt_len, prompt_len_hi=prompt_len, group_size=3,
                            n_pilot=3, max_new=3, cap_lo=3, cap_hi=3, data_seed=3, forced_explicit=None)
    weights = wl.gen_weights(model, seed=2, threads=4, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=3, max_prefill_tokens=prompt_len)
    eng.record_pilot_logits = {1: None}
    got = eng.pilot_commit_step(w, batch)
    want = Decoder(model, weights).forward_full(np.concatenate([batch.prompt_tokens, got["tokens"][0][0][:-1]]))
    logits, _, rr = eng.record_pilot_logits[1]
    row = int(np.flatnonzero(rr == 0)[0])
    assert np.max(np.abs(logits[row].cpu().numpy() - want[prompt_len + 1])) <= 5e-2


UNTIED = dataclasses.replace(wl.SMALL_BF16, name="untied-bf16", tied_embed=False, qkv_bias=False)
WIDE_MLP = dataclasses.replace(UNTIED, name="wide-mlp-bf16", d_model=1536, n_q_heads=12, d_ff=8960, vocab=1003)      # CTA pairs from 200 rows on


def _scaled(model, factors):
    weights = wl.gen_weights(model, seed=2, threads=4, gain_jitter=0.1)
    for name, k in factors.items():
        weights.put(name, weights[name] * np.float32(2.0 ** k), True)        # exact in bfloat16
    return weights


def _pilot(model, weights, rows, fused_sampler=0):
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=1, prompt_len_lo=5, prompt_len_hi=5, group_size=rows,
                            n_pilot=rows, max_new=4, cap_lo=4, cap_hi=4, data_seed=3, forced_explicit=None)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=rows, max_prefill_tokens=5)
    B.pc_set_fused_sampler(eng.ctx, fused_sampler)
    if not fused_sampler:
        eng.record_pilot_logits = {1: None, 2: None}
    got = eng.pilot_commit_step(w, batch)                                     # raises when the device error flag is set
    logits = {} if fused_sampler else {s: eng.record_pilot_logits[s][0].cpu().numpy() for s in (1, 2)}
    return batch, got["tokens"][0], logits


def _worst(model, weights, batch, tokens, logits):
    dec, rows = Decoder(model, weights), len(logits[1])
    worst = 0.0
    for i in sorted({0, rows - 1, rows // 2}):
        want = dec.forward_full(np.concatenate([batch.prompt_tokens, tokens[i][:-1]]))
        worst = max([worst] + [float(np.max(np.abs(logits[s][i] - want[5 + s]))) for s in (1, 2)])
    return worst


@pytest.mark.parametrize("rows", [3, 300])
@pytest.mark.parametrize("matrices,values", [(12, 6), (-8, -8)], ids=["large", "small"])
def test_residual_stream_of_any_size(cuda_device, rows, matrices, values):
    """Everything that is added to the residual stream times 2^k, eps times 2^2k: the same logits.  At 2^18 the stream is beyond half's
    largest value, at 2^-16 (rms 1e-6) its spacing of 2^-24 is 4 % of it.  The factors keep what else is stored as half in its
    normal range: at 2^-8 the rms of the matrices is 8e-5, of the SwiGLU outputs 6e-4 and of V 2e-3, where a spacing of 2^-24 (rms
    rounding error 1.7e-8) adds at most 2.2e-4 to the 1.4e-4 of an ordinary rounding.  So the error grows less than three times."""
    ensure_built()
    k = matrices + values
    ordinary = _worst(UNTIED, _scaled(UNTIED, {}), *_pilot(UNTIED, _scaled(UNTIED, {}), rows))
    model = dataclasses.replace(UNTIED, rms_eps=UNTIED.rms_eps * 4.0 ** k)
    factors = {"embed": k}
    for l in range(model.n_layers):
        factors.update({f"layers.{l}.wo": matrices, f"layers.{l}.w_down": matrices, f"layers.{l}.wv": values, f"layers.{l}.w_up": values})
    weights = _scaled(model, factors)
    worst = _worst(model, weights, *_pilot(model, weights, rows))
    print(f"max |dlogit| {worst:.5f}, of the ordinary model {ordinary:.5f}")
    assert worst <= 3 * ordinary, (worst, ordinary)


@pytest.mark.parametrize("model,rows,grown", [(UNTIED, 3, {"layers.0.w_up": 6, "layers.0.w_down": 14}), (UNTIED, 130, {"layers.0.w_up": 6, "layers.0.w_down": 14}),
                                              (UNTIED, 3, {"layers.1.w_up": 14, "layers.1.w_down": 18}), (UNTIED, 130, {"layers.1.w_up": 14, "layers.1.w_down": 18}),
                                              (WIDE_MLP, 256, {})],
                         ids=["into-qkv-3", "into-qkv-130", "into-lm-head-3", "into-lm-head-130", "into-cta-pairs-256"])
def test_rows_that_outgrow_their_operand(cuda_device, model, rows, grown):
    """The residual stream grows 2^20-fold and more within a sublayer (layer 0's attention, then an MLP): the next operand does not
    hold the rows and their products come from the stream itself.  Six roundings of 2^-11 on logits of rms 0.45 (0.78 with 1,536
    features), 4.5 standard deviations: 2.5e-3 (4.3e-3); asserted with a factor 4."""
    ensure_built()
    bound = 1e-2 * (model.d_model / 512) ** 0.5
    model = dataclasses.replace(model, rms_eps=1e-20)
    weights = _scaled(model, {"embed": -20, **grown})
    batch, tokens, logits = _pilot(model, weights, rows)
    worst = _worst(model, weights, batch, tokens, logits)
    print(f"max |dlogit| {worst:.5f}")
    assert worst <= bound, worst
    assert np.array_equal(np.stack(_pilot(model, weights, rows, fused_sampler=1)[1]), np.stack(tokens))
