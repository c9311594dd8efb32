"""Attention kernels through whole decode steps: prompt lengths around the edges of key tiles and 16-key groups, query rows around
the edges of a 128-row tile, suffix depths around the edges of suffix tiles, against the oracle's full recompute."""
import dataclasses

import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import RolloutEngine

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,prompt,rows,depth,half", [(wl.SMALL_BF16, 1, 1, 2, True), (wl.SMALL_BF16, 16, 63, 18, True),
                                                          (wl.SMALL_QKNORM_BF16, 63, 64, 5, True), (wl.SMALL_BF16, 64, 65, 3, False),
                                                          (wl.SMALL_QKNORM_BF16, 65, 2, 34, True), (wl.SMALL_BF16, 191, 129, 3, True),
                                                          (wl.SMALL_BF16, 600, 3, 66, True), (wl.TINY_BF16, 130, 40, 18, True)],
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
