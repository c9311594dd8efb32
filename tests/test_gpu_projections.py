"""The weight-on-lanes projections (gemm_wt.cuh) through whole decode steps: row counts around the edges of their tiles, K splits
and epilogue chunks, against the oracle's full recompute."""
import dataclasses

import numpy as np
import pytest

from oracle.decoder import Decoder
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
