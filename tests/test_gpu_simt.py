"""The float32 kernels at the edges of their tiles: row counts around 8 / 16 / 64, K and vocabulary sizes that are no multiple of a
block, position counts around the chunks of the attention kernel, every bucket of query heads per KV head."""
import dataclasses

import numpy as np
import pytest

from oracle.decoder import Decoder
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import RolloutEngine

from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,kv,hd,d,ff,vocab,prompt,rows", [(1, 1, 64, 8, 8, 5, 1, 1), (4, 2, 64, 256, 688, 2048, 63, 9), (6, 2, 128, 72, 200, 1003, 65, 17),
                                                                (8, 1, 64, 264, 40, 333, 8, 65), (5, 1, 128, 136, 64, 4097, 130, 3),
                                                                (2, 1, 64, 64, 128, 2048, 3, 520)])
def test_float32_logits_at_tile_edges(cuda_device, heads, kv, hd, d, ff, vocab, prompt, rows):
    ensure_built()
    model = wl.ModelShape("edge-f32", 2, d, heads, kv, hd, ff, vocab, dtype=wl.DTYPE_F32, qk_norm=True, qkv_bias=True)
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=1, prompt_len_lo=prompt, prompt_len_hi=prompt, group_size=rows,
                            n_pilot=rows, max_new=11, cap_lo=11, cap_hi=11, data_seed=5, forced_explicit=None)
    weights = wl.gen_weights(model, seed=4, threads=4, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=rows, max_prefill_tokens=prompt)
    eng.record_pilot_logits = {s: None for s in (0, 7, 9)}
    got = eng.pilot_commit_step(w, batch)
    dec = Decoder(model, weights)
    for i in {0, rows - 1, rows // 2}:
        toks = got["tokens"][0][i]
        want = dec.forward_full(np.concatenate([batch.prompt_tokens, toks[:-1]]))
        for s in (0, 7, 9):
            logits, _, rr = eng.record_pilot_logits[s]
            row = int(np.flatnonzero(rr == i)[0])
            assert np.max(np.abs(logits[row].cpu().numpy() - want[prompt + s])) <= 1e-4, (i, s)
