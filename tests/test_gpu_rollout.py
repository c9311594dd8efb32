"""End-to-end parity of the CUDA rollout path with the CPU oracle (through the C ABI)."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import rollout as orollout
from oracle import stats as ostats
from oracle.decoder import Decoder
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import RolloutEngine

from gpu_util import ensure_built, oracle_group_tokens, teacher_forced_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built(cuda_device):
    ensure_built()


def _compare_step(got, want, w):
    P, G = w.n_prompts, w.group_size
    assert np.array_equal(got["status"], want["status"]) and np.array_equal(got["extra"], want["extra"])
    assert np.array_equal(got["evict"], want["evict"])
    assert got["n_selected"] == want["n_selected"] and got["total_rollouts"] == want["total_rollouts"]
    assert np.array_equal(got["generated"], want["generated"])
    for p in range(P):
        for i in range(G):
            if want["generated"][p, i]:
                assert np.array_equal(got["tokens"][p][i], want["tokens"][p][i]), (p, i)
    assert np.array_equal(got["rewards"], want["rewards"])
    for key in ("pilot_n", "pilot_success", "union_n", "union_success"):
        assert np.array_equal(got[key], want[key]), key
    for key in ("pilot_mean", "pilot_var", "union_mean", "union_var"):
        assert np.max(np.abs(got[key] - want[key])) < 1e-6, key
    assert np.max(np.abs(got["advantages"] - want["advantages"])) < 1e-5


@pytest.mark.parametrize("variant", ["config0", "all_mid", "bt1", "k_eq_G", "ragged"])
def test_config0_free_running_step_is_bit_exact(variant):
    """Tiny fp32 decoder: tokens, rewards, counts, statuses and allocations identical; advantages within 1e-5."""
    w = wl.WORKLOADS["config0"]
    b_t = None
    if variant == "all_mid":
        w = dataclasses.replace(w, forced_explicit=((0, 0.5), (1, 0.5), (2, 0.45), (3, 0.55)))
    elif variant == "bt1":
        w = dataclasses.replace(w, forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.5)), sample_seed=99)
        b_t = 1
    elif variant == "k_eq_G":
        w = dataclasses.replace(w, n_pilot=8)                     # GRPO-style: every rollout in one stage
    elif variant == "ragged":
        w = dataclasses.replace(w, n_prompts=5, prompt_len_lo=1, prompt_len_hi=40, cap_lo=1, cap_hi=16, data_seed=3,
                                forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.5), (4, 0.5)))
    weights = wl.gen_weights(w.model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(w.model, weights)
    want = orollout.pilot_commit_step(dec, w, batch, b_t=b_t)
    eng = RolloutEngine(w.model, weights, max_rows=w.n_prompts * w.group_size, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    got = eng.pilot_commit_step(w, batch, b_t=b_t)
    _compare_step(got, want, w)
    if variant in ("all_mid", "ragged"):
        assert np.any(want["status"] == ostats.COMMIT)


def test_config0_teacher_forced_logits_within_1e_4():
    w = wl.WORKLOADS["config0"]
    weights = wl.gen_weights(w.model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(w.model, weights)
    P, G = w.n_prompts, w.group_size
    prompts, rollouts = np.repeat(np.arange(P), G), np.tile(np.arange(G), P)
    ref = oracle_group_tokens(dec, w, batch, prompts, rollouts)
    eng = RolloutEngine(w.model, weights, max_rows=P * G, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    worst, n_cmp, n_exempt = teacher_forced_compare(eng, w, batch, ref, prompts, rollouts, logit_tol=1e-4, gap_tol=1e-3)
    assert n_cmp == P * G * 16 and n_exempt <= 2


@pytest.mark.parametrize("half_gemm", [True, False], ids=["half-operands", "bf16-operands"])
@pytest.mark.parametrize("model", [wl.TINY_BF16, wl.SMALL_BF16, wl.SMALL_QKNORM_BF16], ids=lambda m: m.name)
def test_small_bf16_models_teacher_forced(model, half_gemm):
    """bf16 storage: logits within 5e-2; sampled token identical wherever the oracle's top-two gap exceeds 1e-1.
    Both operand modes of the GEMMs: IEEE half (the engine's default) and bfloat16 value + rounding remainder."""
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=3, prompt_len_lo=5, prompt_len_hi=70,
                            group_size=6, n_pilot=2, max_new=12, cap_lo=3, cap_hi=12, data_seed=11,
                            forced_explicit=None)
    weights = wl.gen_weights(model, seed=1, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(model, weights)
    P, G = w.n_prompts, w.group_size
    prompts, rollouts = np.repeat(np.arange(P), G), np.tile(np.arange(G), P)
    ref = oracle_group_tokens(dec, w, batch, prompts, rollouts)
    eng = RolloutEngine(model, weights, max_rows=P * G, max_prefill_tokens=int(batch.prompt_offsets[-1]), half_gemm=half_gemm)
    worst, n_cmp, n_exempt = teacher_forced_compare(eng, w, batch, ref, prompts, rollouts, logit_tol=5e-2, gap_tol=1e-1)
    assert n_cmp == int(batch.caps.sum())


@pytest.mark.parametrize("spec", ["qkv=256x2,o=256x3,dn=256x4,gu=64x1,lm=64x1", "qkv=64x1,o=64x1,dn=64x8,gu=256x1,lm=256x1",
                                  "qkv=128x2,o=128x2,dn=128x4,gu=128x1"])
def test_forced_gemm_plans_stay_within_tolerance(spec):
    """pc_set_gemm_plan: the rows-on-lanes kernels with a forced tile width and K-split stay within the tolerance of the oracle; a bad
    spec is refused."""
    from paper_2605_26606_b200 import binding as B
    model = wl.SMALL_BF16
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=3, prompt_len_lo=5, prompt_len_hi=70,
                            group_size=6, n_pilot=2, max_new=12, cap_lo=3, cap_hi=12, data_seed=11, forced_explicit=None)
    weights = wl.gen_weights(model, seed=1, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(model, weights)
    P, G = w.n_prompts, w.group_size
    prompts, rollouts = np.repeat(np.arange(P), G), np.tile(np.arange(G), P)
    ref = oracle_group_tokens(dec, w, batch, prompts, rollouts)
    eng = RolloutEngine(model, weights, max_rows=P * G, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    B.pc_set_gemm_plan(eng.ctx, spec)
    worst, n_cmp, _ = teacher_forced_compare(eng, w, batch, ref, prompts, rollouts, logit_tol=5e-2, gap_tol=1e-1)
    assert n_cmp == int(batch.caps.sum())
    for bad in ("qkv=96x1", "zz=64x1", "dn=64x0", "dn=64"):
        with pytest.raises(B.PcError):
            B.pc_set_gemm_plan(eng.ctx, bad)
    B.pc_set_gemm_plan(eng.ctx, None)


def test_run_twice_is_deterministic_and_batch_invariant():
    """Same inputs give bit-identical tokens; a rollout's tokens do not depend on its batch mates."""
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=wl.TINY_BF16, n_pilot=8)
    weights = wl.gen_weights(w.model, seed=0, threads=2)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(w.model, weights, max_rows=64, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    a = eng.pilot_commit_step(w, batch)
    b = eng.pilot_commit_step(w, batch)
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i])
    w2 = dataclasses.replace(w, n_pilot=2, forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.5)))
    c = eng.pilot_commit_step(w2, wl.gen_batch(w2))
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            if c["generated"][p, i]:
                assert np.array_equal(a["tokens"][p][i], c["tokens"][p][i])


def test_bf16_many_rows_long_prefix_long_suffix():
    """Several query tiles per group, prompt longer than the K/V ring of the group kernel, suffix longer than the
    ring of the suffix kernel, several work items per warp, ragged tails everywhere."""
    model = wl.SMALL_BF16
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=2, prompt_len_lo=197, prompt_len_hi=333,
                            group_size=70, n_pilot=70, max_new=140, cap_lo=90, cap_hi=140, data_seed=5, forced_explicit=None)
    weights = wl.gen_weights(model, seed=2, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(model, weights)
    P, G = w.n_prompts, w.group_size
    prompts, rollouts = np.repeat(np.arange(P), G), np.tile(np.arange(G), P)
    ref = oracle_group_tokens(dec, w, batch, prompts, rollouts)
    eng = RolloutEngine(model, weights, max_rows=P * G, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    worst, n_cmp, n_exempt = teacher_forced_compare(eng, w, batch, ref, prompts, rollouts, logit_tol=5e-2, gap_tol=1e-1)
    assert n_cmp == int(batch.caps.sum())


@pytest.mark.parametrize("model", [wl.TINY, wl.SMALL_BF16], ids=lambda m: m.name)
def test_graph_replay_equals_step_by_step(model):
    """pc_decode_run (captured steps replayed from a device-resident schedule) against one pc_decode_step per step."""
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=5, prompt_len_lo=3, prompt_len_hi=50, group_size=9,
                            n_pilot=3, max_new=40, cap_lo=1, cap_hi=40, data_seed=21,
                            forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.0), (4, 0.5)))
    weights = wl.gen_weights(model, seed=0, threads=2)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=45, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    eng.use_graphs = False
    a = eng.pilot_commit_step(w, batch)
    eng.use_graphs = True
    b = eng.pilot_commit_step(w, batch)
    assert np.array_equal(a["status"], b["status"]) and np.any(a["status"] == ostats.COMMIT)
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            if a["generated"][p, i]:
                assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i])
    assert np.array_equal(a["advantages"], b["advantages"])


@pytest.mark.parametrize("base", [wl.QWEN3_8B, wl.QWEN3_14B], ids=lambda m: m.name)
def test_qwen3_widths_two_layers_teacher_forced(base):
    """The 8B / 14B layer shapes (d 4096 / 5120, 32/8 and 40/8 heads, QK-norm, untied head, theta 1e6) with two layers and a
    reduced vocabulary, so that the oracle stays cheap: logits within 5e-2, tokens identical outside the 1e-1 gap."""
    model = dataclasses.replace(base, name=base.name + "-2l", n_layers=2, vocab=8192)
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=2, prompt_len_lo=40, prompt_len_hi=90, group_size=5,
                            n_pilot=5, max_new=6, cap_lo=2, cap_hi=6, data_seed=4, forced_explicit=None)
    weights = wl.gen_weights(model, seed=3, threads=4)
    batch = wl.gen_batch(w)
    dec = Decoder(model, weights)
    P, G = w.n_prompts, w.group_size
    prompts, rollouts = np.repeat(np.arange(P), G), np.tile(np.arange(G), P)
    ref = oracle_group_tokens(dec, w, batch, prompts, rollouts)
    eng = RolloutEngine(model, weights, max_rows=P * G, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    worst, n_cmp, n_exempt = teacher_forced_compare(eng, w, batch, ref, prompts, rollouts, logit_tol=5e-2, gap_tol=1e-1)
    assert n_cmp == int(batch.caps.sum())


def test_behaviour_logprobs_along_free_running_rollouts():
    """log pi(o_t) of every sampled token (Eq. 2's denominator), config 0: tokens are identical to the oracle's, so its
    logits give the expected log-probabilities position by position."""
    from oracle.logprob import token_logprob
    w = dataclasses.replace(wl.WORKLOADS["config0"], forced_explicit=((0, 0.0), (1, 0.5), (2, 0.45), (3, 1.0)))
    weights = wl.gen_weights(w.model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    dec = Decoder(w.model, weights)
    eng = RolloutEngine(w.model, weights, max_rows=w.n_prompts * w.group_size, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    eng.collect_logprobs = True
    out = eng.pilot_commit_step(w, batch)
    assert np.any(out["status"] == ostats.COMMIT)
    n_checked = 0
    for p in range(w.n_prompts):
        idx = [i for i in range(w.group_size) if out["generated"][p, i]]
        ref = oracle_group_tokens(dec, w, batch, [p] * len(idx), idx)
        for i in idx:
            toks, logs = ref[(p, i)]
            assert np.array_equal(toks, out["tokens"][p][i])
            for s, t in enumerate(toks):
                assert abs(out["logprobs"][p, i, s] - token_logprob(logs[s], int(t), w.temperature)) < 1e-4
                n_checked += 1
    assert n_checked == int(batch.caps[out["generated"]].sum())


def test_bound_pass_equals_separate_passes_of_the_same_engine():
    """Section 3.4 binding: commit rollouts of batch A's survivors and pilot rollouts of batch B in one decode batch are
    token for token what separate passes produce (A's prompt KV is taken over, not recomputed)."""
    w = dataclasses.replace(wl.WORKLOADS["config0"], n_prompts=4, prompt_len_lo=5, prompt_len_hi=40, cap_lo=3, cap_hi=16,
                            forced_explicit=((0, 0.5), (1, 0.0), (2, 0.5), (3, 0.5)), data_seed=31)
    wb = dataclasses.replace(w, data_seed=32, n_prompts=3, forced_explicit=None)
    weights = wl.gen_weights(w.model, seed=0, threads=2)
    batch_a, batch_b = wl.gen_batch(w), wl.gen_batch(wb)
    P, G, k = w.n_prompts, w.group_size, w.n_pilot
    eng = RolloutEngine(w.model, weights, max_rows=64, max_prefill_tokens=int(batch_a.prompt_offsets[-1] + batch_b.prompt_offsets[-1]))
    # separate passes
    full_a = eng.pilot_commit_step(w, batch_a)
    commit_a = np.flatnonzero(full_a["status"] == ostats.COMMIT)
    assert 0 < len(commit_a) < P
    full_b = eng.pilot_commit_step(wb, batch_b)
    # bound: A's pilot pass, then one pass with A's commit rows and B's pilot rows
    eng.load_batch(w, batch_a)
    eng.prefill()
    eng.run_stage(np.repeat(np.arange(P), k), np.tile(np.arange(k), P))
    bound = eng.bound_pass(w, batch_a, commit_a, batch_b)
    assert len(bound["a"]) == len(commit_a) * (G - k) and len(bound["b"]) == wb.n_prompts * k
    for (p, i), t in bound["a"].items():
        assert np.array_equal(t, full_a["tokens"][p][i]), (p, i)
    for (p, i), t in bound["b"].items():
        assert np.array_equal(t, full_b["tokens"][p][i]), (p, i)


@pytest.mark.parametrize("data_seed,sample_seed", [(0, 1234), (1, 1234), (2, 7), (3, 99), (4, 2**40 + 5), (5, 1234), (6, 31), (7, 8)])
def test_config0_free_running_seed_sweep_is_bit_exact(data_seed, sample_seed):
    """config0 over eight (data seed, sampling seed) pairs.  (The workload's default data seed is 6 because it is the first
    one, with prompts 0 and 3 forced to tau = 0 / 1, whose batch has a prompt that passes the pilot filter, so that the
    commit stage runs; several seeds of this sweep, 0 among them, commit nothing.)"""
    w = dataclasses.replace(wl.WORKLOADS["config0"], data_seed=data_seed, sample_seed=sample_seed)
    weights = wl.gen_weights(w.model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    want = orollout.pilot_commit_step(Decoder(w.model, weights), w, batch)
    eng = RolloutEngine(w.model, weights, max_rows=w.n_prompts * w.group_size, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    _compare_step(eng.pilot_commit_step(w, batch), want, w)


def _bound_setup(model, seed_a, seed_b, forced_a, sample_seed=1234):
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=4, prompt_len_lo=5, prompt_len_hi=40, cap_lo=3, cap_hi=16,
                            forced_explicit=forced_a, data_seed=seed_a, sample_seed=sample_seed)
    wb = dataclasses.replace(w, data_seed=seed_b, n_prompts=3, forced_explicit=None)
    return w, wb, wl.gen_batch(w), wl.gen_batch(wb)


def test_bound_pass_tokens_equal_the_oracle_rollouts():
    """Section 3.4 binding against the oracle: every rollout of the bound pass (commit rollouts of batch A's survivors, pilot
    rollouts of batch B) is token for token the rollout the oracle generates for that (prompt, rollout) on its own --
    counter-based keys make a rollout independent of the batch it is decoded in."""
    w, wb, batch_a, batch_b = _bound_setup(wl.TINY, 31, 32, ((0, 0.5), (1, 0.0), (2, 0.5), (3, 0.5)))
    weights = wl.gen_weights(w.model, seed=0, threads=2, gain_jitter=0.1)
    dec = Decoder(w.model, weights)
    P, G, k = w.n_prompts, w.group_size, w.n_pilot
    want_a = orollout.pilot_commit_step(dec, w, batch_a)
    commit_a = np.flatnonzero(want_a["status"] == ostats.COMMIT)
    assert 0 < len(commit_a) < P
    eng = RolloutEngine(w.model, weights, max_rows=64, max_prefill_tokens=int(batch_a.prompt_offsets[-1] + batch_b.prompt_offsets[-1]))
    eng.load_batch(w, batch_a)
    eng.prefill()
    eng.run_stage(np.repeat(np.arange(P), k), np.tile(np.arange(k), P))
    bound = eng.bound_pass(w, batch_a, commit_a, batch_b)
    assert len(bound["a"]) == len(commit_a) * (G - k) and len(bound["b"]) == wb.n_prompts * k
    for (p, i), t in bound["a"].items():
        assert np.array_equal(t, want_a["tokens"][p][i]), (p, i)
    for p in range(wb.n_prompts):
        pt = batch_b.prompt_tokens[batch_b.prompt_offsets[p]:batch_b.prompt_offsets[p + 1]]
        want = orollout.generate_group(dec, pt, p, list(range(k)), batch_b.caps[p, :k], wb.sample_seed, wb.temperature)
        for i in range(k):
            assert np.array_equal(bound["b"][(p, i)], want[i]), (p, i)


def test_bound_pass_bf16_logits_against_full_recompute():
    """The bound pass on the tensor-core path: the logits of every decode step of the mixed batch against the oracle's full
    recompute over (prompt + the GPU's own tokens), 5e-2; drawn tokens identical outside the 1e-1 gap."""
    from oracle import sampler as osampler
    model = wl.SMALL_BF16
    w, wb, batch_a, batch_b = _bound_setup(model, 41, 42, ((0, 0.5), (1, 0.5), (2, 0.0), (3, 0.5)), sample_seed=7)
    weights = wl.gen_weights(model, seed=5, threads=2, gain_jitter=0.1)
    dec = Decoder(model, weights)
    P, G, k = w.n_prompts, w.group_size, w.n_pilot
    eng = RolloutEngine(model, weights, max_rows=64, max_prefill_tokens=int(batch_a.prompt_offsets[-1] + batch_b.prompt_offsets[-1]))
    full_a = eng.pilot_commit_step(w, batch_a)
    commit_a = np.flatnonzero(full_a["status"] == ostats.COMMIT)
    assert 0 < len(commit_a) < P
    eng.load_batch(w, batch_a)
    eng.prefill()
    eng.run_stage(np.repeat(np.arange(P), k), np.tile(np.arange(k), P))
    n_steps = int(max(batch_a.caps.max(), batch_b.caps.max())) - 1
    eng.record_pilot_logits = {s: None for s in range(n_steps)}
    bound = eng.bound_pass(w, batch_a, commit_a, batch_b)
    rec = eng.record_pilot_logits
    eng.record_pilot_logits = None
    nA = len(commit_a)
    worst, n_cmp = 0.0, 0
    cases = [(j, int(p), i, batch_a, bound["a"][(int(p), i)]) for j, p in enumerate(commit_a) for i in range(k, G)]
    cases += [(nA + p, p, i, batch_b, bound["b"][(p, i)]) for p in range(wb.n_prompts) for i in range(k)]
    for row_prompt, key_prompt, i, batch, toks in cases:
        pt = batch.prompt_tokens[batch.prompt_offsets[key_prompt]:batch.prompt_offsets[key_prompt + 1]]
        Lp = len(pt)
        if len(toks) < 2:
            continue
        want = dec.forward_full(np.concatenate([pt, toks[:-1]]))
        for s in range(len(toks) - 1):                         # decode step s consumed token s and produced the logits of token s + 1
            logits, rp, rr = rec[s]
            row = int(np.flatnonzero((rp == row_prompt) & (rr == i))[0])
            got = logits[row].cpu().numpy()
            worst = max(worst, float(np.max(np.abs(got - want[Lp + s]))))
            tok_o, gap = osampler.sample(want[Lp + s], w.temperature, w.sample_seed, key_prompt, i, s + 1)
            if gap > 1e-1:
                assert int(toks[s + 1]) == tok_o, (key_prompt, i, s, gap)
            n_cmp += 1
    assert n_cmp > 50 and worst <= 5e-2, (n_cmp, worst)


@pytest.mark.parametrize("model", [wl.SMALL_BF16, wl.SMALL_QKNORM_BF16, wl.TINY_BF16], ids=lambda m: m.name)
def test_persistent_decode_kernel_equals_one_kernel_per_operation(model):
    """pc_set_decode_mode: the persistent kernel (phases separated by grid barriers) runs the arithmetic of the form with one
    kernel per operation (pc_set_fused_epilogues 0) in the same order, so a free-running Pilot-Commit step gives identical tokens and identical recorded logits; a
    missed barrier or a stale tile would show up as a difference."""
    from paper_2605_26606_b200 import binding as B
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=5, prompt_len_lo=3, prompt_len_hi=90, group_size=40,
                            n_pilot=8, max_new=40, cap_lo=1, cap_hi=40, data_seed=21,
                            forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.0), (4, 0.5)))
    weights = wl.gen_weights(model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=200, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    B.pc_set_fused_epilogues(eng.ctx, 0)              # the persistent kernel shares its arithmetic with the one-kernel-per-operation form
    outs, logits = [], []
    for mode in (0, 1, 1):
        B.pc_set_decode_mode(eng.ctx, mode)
        eng.record_pilot_logits = {s: None for s in (0, 5, 17)}
        outs.append(eng.pilot_commit_step(w, batch))
        logits.append({s: v[0].clone() for s, v in eng.record_pilot_logits.items()})
    eng.record_pilot_logits = None
    a = outs[0]
    assert np.any(a["status"] == ostats.COMMIT)
    for b, lg in zip(outs[1:], logits[1:]):
        assert np.array_equal(a["status"], b["status"])
        for p in range(w.n_prompts):
            for i in range(w.group_size):
                if a["generated"][p, i]:
                    assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i]), (p, i)
        for s in lg:
            assert torch.equal(lg[s], logits[0][s]), s
        assert np.array_equal(a["advantages"], b["advantages"])


@pytest.mark.parametrize("model,group_size", [(wl.SMALL_BF16, 40), (wl.SMALL_QKNORM_BF16, 40), (wl.SMALL_BF16, 90)],
                         ids=["small-batch-kernels", "qk-norm", "fused-epilogues"])
def test_dependent_launch_of_the_projections_changes_no_bit(model, group_size):
    """pc_set_dependent_launch: a projection launched as a programmatic dependent sets itself up and requests weight tiles
    while the kernel before it still runs, and waits for that kernel before it reads activations.  Tokens, recorded logits
    and advantages of a free-running Pilot-Commit step must be identical with the switch on (every projection and the shared-prefix attention), on for the
    gate/up projection only, on for the attention kernel only, and off; a projection that read its operand early would show up as a difference.  The
    90-rollout groups take the commit stage above 256 rows, to other tilings and to the suffix kernel that merges inside a warp."""
    from paper_2605_26606_b200 import binding as B
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=5, prompt_len_lo=3, prompt_len_hi=90, group_size=group_size,
                            n_pilot=8, max_new=40, cap_lo=1, cap_hi=40, data_seed=21,
                            forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.0), (4, 0.5)))
    weights = wl.gen_weights(model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=5 * group_size, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    outs, logits = [], []
    for mask in (0, 63, 4, 32, 63):
        B.pc_set_dependent_launch(eng.ctx, mask)
        eng.record_pilot_logits = {s: None for s in (0, 5, 17)}
        outs.append(eng.pilot_commit_step(w, batch))
        logits.append({s: v[0].clone() for s, v in eng.record_pilot_logits.items()})
    eng.record_pilot_logits = None
    a = outs[0]
    assert np.any(a["status"] == ostats.COMMIT)
    for b, lg in zip(outs[1:], logits[1:]):
        assert np.array_equal(a["status"], b["status"])
        for p in range(w.n_prompts):
            for i in range(w.group_size):
                if a["generated"][p, i]:
                    assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i]), (p, i)
        for s in lg:
            assert torch.equal(lg[s], logits[0][s]), s
        assert np.array_equal(a["advantages"], b["advantages"])


def test_new_schedules_and_token_buffers_reuse_the_captured_steps():
    """pc_decode_run keys its captured steps on shapes and arenas only: running the same step again (fresh schedule tensors, a
    fresh token buffer, another sampling seed) captures nothing new, and a bad row index is caught on the device."""
    from paper_2605_26606_b200 import binding as B
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=wl.SMALL_BF16, n_prompts=5, prompt_len_lo=3, prompt_len_hi=50, group_size=9,
                            n_pilot=3, max_new=40, cap_lo=1, cap_hi=40, data_seed=21,
                            forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.0), (4, 0.5)))
    weights = wl.gen_weights(w.model, seed=0, threads=2)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(w.model, weights, max_rows=45, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    a = eng.pilot_commit_step(w, batch)
    n1 = B.pc_capture_count(eng.ctx)
    assert n1 > 0
    keep = [eng.tokens, eng._keep_schedule]              # keep the old buffers alive so that the allocator hands out new addresses
    b = eng.pilot_commit_step(w, batch)
    assert B.pc_capture_count(eng.ctx) == n1
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            if a["generated"][p, i]:
                assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i])
    c = eng.pilot_commit_step(dataclasses.replace(w, sample_seed=77), batch)
    assert B.pc_capture_count(eng.ctx) == n1
    assert any(not np.array_equal(a["tokens"][p][0], c["tokens"][p][0]) for p in range(w.n_prompts))
    del keep
    # a row that names a prompt outside the per-prompt arrays is switched off and flagged instead of read
    eng.load_batch(w, batch)
    eng.prefill()
    sch_prompts = np.array([1], dtype=np.int64)
    longest = np.argsort(-batch.caps[1])[:2]                          # two rollouts of prompt 1 with several decode steps
    assert batch.caps[1, longest[1]] > 2
    eng.run_stage(sch_prompts, longest[:1])                           # a valid one-row stage first
    eng.check_error_flag()
    B.pc_set_index_bounds(eng.ctx, w.n_prompts, 8)                   # token buffer "of 8 cells": every row_tok_index is beyond it
    eng.use_graphs = False
    eng.run_stage(sch_prompts, longest[1:])
    assert int(eng.err_flag.item()) == 4                             # DEV_ERR_GROUP_RANGE
    eng.err_flag.zero_()


def test_half_operands_out_of_range_are_saturated_and_flagged():
    """IEEE-half GEMM operands: with gate / up matrices scaled until the SwiGLU output passes 65504 the step still ends with
    in-range tokens and the device error flag holds DEV_ERR_HALF_RANGE (5) -- no silent inf / NaN logits."""
    model = wl.SMALL_BF16
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=2, prompt_len_lo=5, prompt_len_hi=20, group_size=4,
                            n_pilot=4, max_new=6, cap_lo=3, cap_hi=6, data_seed=2, forced_explicit=None)
    weights = wl.gen_weights(model, seed=1, threads=2)
    weights.put("layers.0.w_gate", weights["layers.0.w_gate"] * 64.0, True)
    weights.put("layers.0.w_up", weights["layers.0.w_up"] * 4096.0, True)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=8, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    eng.load_batch(w, batch)
    status, n_tok = eng.run_device()
    torch.cuda.synchronize()
    assert int(eng.err_flag.item()) == 5
    toks = eng.tokens.cpu().numpy().reshape(w.n_prompts, w.group_size, w.max_new)
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            t = toks[p, i, :batch.caps[p, i]]
            assert t.min() >= 0 and t.max() < model.vocab
    assert torch.isfinite(eng.last_logits).all()
    eng.err_flag.zero_()
    # the same model inside the range raises nothing
    weights2 = wl.gen_weights(model, seed=1, threads=2)
    eng2 = RolloutEngine(model, weights2, max_rows=8, max_prefill_tokens=int(batch.prompt_offsets[-1]))
    eng2.pilot_commit_step(w, batch)


@pytest.mark.parametrize("vocab,half_gemm", [(4096, True), (20004, True), (20004, False)], ids=["narrow-tiles", "wide-tiles-ragged-vocab", "bf16-operands"])
def test_sampler_in_the_lm_head_epilogue_draws_the_same_tokens(vocab, half_gemm):
    """pc_set_fused_sampler: the Gumbel-max draw inside the LM-head GEMM (no logits stored) against the stand-alone sampler on
    stored logits, free running over a whole Pilot-Commit step: every token identical, and the oracle's tokens wherever its
    top-two gap is clear (checked teacher-forced by the tests above for the stored-logits path)."""
    from paper_2605_26606_b200 import binding as B
    model = dataclasses.replace(wl.SMALL_BF16, name=f"small-bf16-v{vocab}", vocab=vocab)
    w = dataclasses.replace(wl.WORKLOADS["config0"], model=model, n_prompts=5, prompt_len_lo=3, prompt_len_hi=90, group_size=40,
                            n_pilot=8, max_new=30, cap_lo=1, cap_hi=30, data_seed=23,
                            forced_explicit=((0, 0.5), (1, 0.5), (2, 0.5), (3, 0.0), (4, 0.5)))
    weights = wl.gen_weights(model, seed=0, threads=2, gain_jitter=0.1)
    batch = wl.gen_batch(w)
    eng = RolloutEngine(model, weights, max_rows=200, max_prefill_tokens=int(batch.prompt_offsets[-1]), half_gemm=half_gemm)
    outs = []
    for fused in (0, 1):
        B.pc_set_fused_sampler(eng.ctx, fused)
        n0 = B.pc_launch_count()
        outs.append(eng.pilot_commit_step(w, batch))
    a, b = outs
    assert np.array_equal(a["status"], b["status"]) and np.any(a["status"] == ostats.COMMIT)
    n_tok = 0
    for p in range(w.n_prompts):
        for i in range(w.group_size):
            if a["generated"][p, i]:
                assert np.array_equal(a["tokens"][p][i], b["tokens"][p][i]), (p, i)
                n_tok += len(a["tokens"][p][i])
    assert n_tok > 1000
    assert np.array_equal(a["advantages"], b["advantages"])
