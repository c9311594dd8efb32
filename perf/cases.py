"""The calls a program built on this framework spends its time in, at the sizes it makes them.

A training step of group rollout generation is: one shared prefill of the sampling batch, then hundreds to thousands of
decode steps over the live rollouts (their number falls as rollouts end), then the rewards, statistics, allocation and
advantages.  The listed cases follow the repository's own configurations (workloads.WORKLOADS): the sizes of one whole
step on the float32 configuration, the prefill and the decode steps of the 1.5B, 8B and 14B shapes at the row counts and
suffix depths the pilot, commit and all-rollouts stages go through.

bfloat16 rollouts that sample freely for long cannot be compared between two correct implementations (one last-bit
difference in a logit sooner or later draws another token), so the decode cases run a short window of consecutive steps
from a given depth, as pc_decode_run replays them, and hand back the token (and log-probability) buffers the window updates.
"""
import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_2605_26606_b200 import binding as B
from paper_2605_26606_b200 import workloads as wl
from paper_2605_26606_b200.engine import STEP_DESC_DTYPE, RolloutEngine

MODELS = {m.name: m for m in (wl.TINY, wl.QWEN25_1P5B, wl.QWEN3_8B, wl.QWEN3_14B)}
# What the workspace of a program on this model is sized for: concurrent rollouts, packed prompt tokens of one prefill
CAPACITY = {wl.QWEN25_1P5B.name: (2048, 16384), wl.QWEN3_8B.name: (512, 4096), wl.QWEN3_14B.name: (256, 2048)}
SAMPLE_SEED = 1234


# ----------------------------------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------------------------------
def _step(prompts, group, pilot, prompt_lo, prompt_hi, cap_lo, cap_hi):
    return dict(kind="step", model=wl.TINY.name, prompts=prompts, group=group, pilot=pilot, prompt_lo=prompt_lo, prompt_hi=prompt_hi,
                cap_lo=cap_lo, cap_hi=cap_hi)


def _prefill(model, prompts, lo, hi):
    return dict(kind="prefill", model=model.name, prompts=prompts, prompt_lo=lo, prompt_hi=hi)


def _decode(model, rows, groups, group_size, suffix, steps, prompt_lo=256, prompt_hi=1024, half=True, logprobs=False, logits=False):
    """rows: live rollouts at the first step; groups x group_size: what the stage started with."""
    return dict(kind="decode", model=model.name, rows=rows, groups=groups, group_size=group_size, suffix=suffix, steps=steps,
                prompt_lo=prompt_lo, prompt_hi=prompt_hi, half=half, logprobs=logprobs, logits=logits)


def listed():
    q15, q8 = wl.QWEN25_1P5B, wl.QWEN3_8B
    return [
        # what follows the generation: rewards, statistics, allocation and advantages of a sampling batch; the smallest call
        dict(kind="groups", prompts=512, group=16, pilot=8, name="groups_512x16"),
        # one whole Pilot-Commit step through the engine, float32, everything counted: upload, schedules, prefill, both stages,
        # read-back.  config 0 as it stands, and a larger ragged batch
        dict(_step(4, 8, 2, 32, 32, 16, 16), name="step_f32_config0"),
        dict(_step(24, 16, 4, 16, 96, 24, 96), name="step_f32_ragged"),
        # shared prefill: one prompt arriving alone (odd length), and config 2's whole sampling batch
        dict(_prefill(q15, 1, 351, 351), name="prefill_1x351"),
        dict(_prefill(q15, 16, 256, 1024), name="prefill_16x256-1024"),
        # decode steps of the 1.5B shape.  The tail of a stage (few long rollouts left), config 1's pilot with the behaviour
        # log-probabilities a policy update needs, config 2's pilot with some rollouts ended, its commit stage (few large groups)
        # deep into the rollouts, and all 2048 rollouts at once
        dict(_decode(q15, 16, 9, 16, 1100, 8), name="decode_16@1100"),
        dict(_decode(q15, 71, 32, 4, 256, 8, 256, 256, logprobs=True), name="decode_71@256_logprob"),
        dict(_decode(q15, 237, 16, 16, 512, 8), name="decode_237@512"),
        dict(_decode(q15, 336, 3, 112, 900, 8), name="decode_336@900"),
        dict(_decode(q15, 2048, 16, 128, 512, 8), name="decode_2048@512"),
        # bfloat16 operands, one step whose logits the caller keeps (scoring given tokens)
        dict(_decode(q15, 112, 1, 112, 300, 1, half=False, logits=True), name="score_112@300_bf16"),
        # config 3's pilot stage on the 8B shape
        dict(_decode(q8, 64, 8, 8, 300, 8, 512, 512), name="decode_8b_64@300"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_any(rng):
    kind = rng.choice(["groups", "step", "prefill", "decode", "decode", "decode", "decode", "decode"])
    if kind == "groups":
        group = rng.choice([8, 16, 64, 128])
        return dict(kind="groups", prompts=_log_int(rng, 4, 4096), group=group, pilot=group // rng.choice([2, 4, 8]))
    if kind == "step":
        group = rng.choice([4, 8, 16, 32])
        cap_hi, p_hi = _log_int(rng, 8, 96), _log_int(rng, 8, 128)
        return _step(_log_int(rng, 2, 32), group, max(1, group // rng.choice([2, 4])), max(4, p_hi // rng.choice([1, 2, 4])), p_hi,
                     max(2, cap_hi // rng.choice([1, 2, 4])), cap_hi)
    if kind == "prefill":
        hi = _log_int(rng, 64, 1024)
        return _prefill(wl.QWEN25_1P5B, _log_int(rng, 1, 16), max(16, hi // rng.choice([1, 2, 4])), hi)
    model = MODELS[rng.choice([wl.QWEN25_1P5B.name] * 7 + [wl.QWEN3_8B.name] * 2 + [wl.QWEN3_14B.name])]
    rows = _log_int(rng, 8, CAPACITY[model.name][0])
    groups = min(rows, rng.choice([1, 3, 4, 8, 16, 32]))
    hi = _log_int(rng, 64, 1024)
    half, logits = rng.random() < 0.85 or model is not wl.QWEN25_1P5B, rng.random() < 0.15
    return _decode(model, rows, groups, min(-(-rows // groups) + rng.choice([0, 1, 7]), CAPACITY[model.name][0] // groups + 1),
                   _log_int(rng, 16, 1536), 1 if logits else 8, max(16, hi // rng.choice([1, 2, 4])), hi, half,
                   not logits and rng.random() < 0.3, logits)


def draw(rng):
    most = [work(c) for c in listed()]
    top_bytes, top_flops = max(w["bytes"] for w in most), max(w["flops"] for w in most)
    while True:
        c = _draw_any(rng)
        w = work(c)
        if w["bytes"] <= top_bytes and w["flops"] <= top_flops:
            return c


# ----------------------------------------------------------------------------------------------------------------
# what a program keeps: weights, context and workspace of one model
# ----------------------------------------------------------------------------------------------------------------
_KEPT = {}


def _keep(key, make):
    if key not in _KEPT:
        _KEPT.clear()                       # one model at a time, like a program that serves one
        torch.cuda.empty_cache()
        _KEPT[key] = make()
    return _KEPT[key]


@dataclasses.dataclass
class _Model:
    shape: wl.ModelShape
    ctx: B.Context
    error: torch.Tensor


def _random_model(m, half):
    """Random-init weights N(0, 0.02) of a bf16 shape made on the GPU, in the layout pc_create takes."""
    g = torch.Generator(device="cuda").manual_seed(0)

    def matrix(rows, cols, as_half=half):
        t = torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=g)
        return t.to(torch.float16) if as_half else t

    ones = lambda n: torch.ones(n, dtype=torch.float32, device="cuda")
    L, d, qkv = range(m.n_layers), m.d_model, m.q_dim + 2 * m.kv_dim
    embed = matrix(m.vocab, d, False)
    head = (embed.to(torch.float16) if half else None) if m.tied_embed else matrix(m.vocab, d)
    bias = [torch.empty(qkv, dtype=torch.float32, device="cuda").normal_(0.0, 0.02, generator=g) for _ in L] if m.qkv_bias else None
    gains = [ones(m.head_dim) for _ in L] if m.qk_norm else None
    desc = B.ModelDesc(m.n_layers, d, m.n_q_heads, m.n_kv_heads, m.head_dim, m.d_ff, m.vocab, m.rms_eps, m.rope_theta, m.dtype,
                       int(m.tied_embed), int(m.qk_norm), int(m.qkv_bias), int(half))
    ctx = B.pc_create(desc, embed, head, ones(d), [ones(d) for _ in L], [matrix(qkv, d) for _ in L], bias, gains, gains,
                      [matrix(d, m.q_dim) for _ in L], [ones(d) for _ in L], [matrix(2 * m.d_ff, d) for _ in L],
                      [matrix(d, m.d_ff) for _ in L])
    rows, tokens = CAPACITY[m.name]
    space = torch.empty(B.pc_workspace_bytes(ctx, rows, tokens), dtype=torch.uint8, device="cuda")
    error = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.pc_set_workspace(ctx, space, rows, tokens, error)
    return _Model(m, ctx, error)


def _model(case):
    m, half = MODELS[case["model"]], bool(case.get("half", True))
    return _keep((m.name, half), lambda: _random_model(m, half))


def _workload(case, seed):
    return wl.Workload("case", MODELS[case["model"]], case["prompts"], case["prompt_lo"], case["prompt_hi"], case["group"], case["pilot"],
                       case["cap_hi"], case["cap_lo"], case["cap_hi"], 0.3, data_seed=seed, sample_seed=SAMPLE_SEED)


# ----------------------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------------------
def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype=dtype)


def _arena(m, slots, gen=None):
    """A KV arena (K and V as IEEE half); with a generator, filled with values of the size the shape's projections give."""
    t = torch.empty((m.n_layers, 2, m.n_kv_heads, slots, m.head_dim), dtype=torch.float16, device="cuda")
    return t if gen is None else t.normal_(0.0, 1.0 if m.qk_norm else 0.8, generator=gen)


def _prompt_lens(r, case, n):
    return r.integers(case["prompt_lo"], case["prompt_hi"] + 1, n)


def prepare(case, seed):
    r = np.random.default_rng([seed, 17])
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return {"groups": _prepare_groups, "step": _prepare_step, "prefill": _prepare_prefill, "decode": _prepare_decode}[case["kind"]](
        case, seed, r, gen)


def _prepare_groups(case, seed, r, gen):
    P, G, k, V, width = case["prompts"], case["group"], case["pilot"], wl.QWEN25_1P5B.vocab, 4      # width: token cells per rollout
    # success rates of Beta(1/2, 1/2), three in ten prompts all wrong or all right
    tau = np.sin(0.5 * math.pi * r.random(P)) ** 2
    forced = r.random(P) < 0.3
    tau[forced] = (r.random(P) < 0.5)[forced]
    i32 = lambda: torch.zeros(P, dtype=torch.int32, device="cuda")
    f32 = lambda n=P: torch.zeros(n, dtype=torch.float32, device="cuda")
    count = lambda n: torch.full((P,), n, dtype=torch.int32, device="cuda")
    return dict(run=_run_groups, P=P, G=G, tokens=_dev(r.integers(0, V, P * G * width), torch.int32),
                last=_dev(np.arange(P * G) * width + r.integers(0, width, P * G), torch.int64),
                threshold=_dev(np.repeat(np.floor(tau * V), G), torch.int32), start=_dev(np.arange(P) * G, torch.int32),
                pilot=count(k), union=count(G), rewards=f32(P * G), n=i32(), success=i32(), mean=f32(), var=f32(), status=i32(),
                extra=i32(), evict=i32(), selected=torch.zeros(1, dtype=torch.int32, device="cuda"),
                total=torch.zeros(1, dtype=torch.int64, device="cuda"), union_n=i32(), union_success=i32(), union_mean=f32(),
                union_var=f32(), advantage=f32(P * G), params=B.AllocParams(0.125, 0.75, 1.0, G - k, max(1, P // 2)))


def _prepare_step(case, seed, r, gen):
    w = _workload(case, seed)
    weights = lambda: wl.gen_weights(w.model, seed=0)
    rows = w.n_prompts * max(w.n_pilot, w.n_commit)
    tokens = w.n_prompts * w.prompt_len_hi
    eng = _keep((w.model.name, rows, tokens), lambda: RolloutEngine(w.model, weights(), max_rows=rows, max_prefill_tokens=tokens))
    return dict(run=_run_step, eng=eng, workload=w, batch=wl.gen_batch(w))


def _prepare_prefill(case, seed, r, gen):
    k = _model(case)
    m, P = k.shape, case["prompts"]
    offsets = np.r_[0, np.cumsum(_prompt_lens(r, case, P))]
    total, slots = int(offsets[-1]), P * case["prompt_hi"]           # the arena has room for the longest prompts there may be
    return dict(run=_run_prefill, model=k, P=P, total=total, slots=slots, longest=int(np.diff(offsets).max()),
                tokens=_dev(r.integers(0, m.vocab, total), torch.int32), offsets=_dev(offsets, torch.int32),
                start=_dev(offsets[:-1], torch.int64), kv=_arena(m, slots).zero_(), logits=torch.empty((P, m.vocab), device="cuda"))


def _prepare_decode(case, seed, r, gen):
    k = _model(case)
    m, P, R, s0, n = k.shape, case["groups"], case["rows"], case["suffix"], case["steps"]
    cap = s0 + n + 1
    # which rollouts of which groups are still live, and how long each goes on (a few end inside the window)
    full = P * max(case["group_size"], -(-R // P))
    live = np.sort(r.choice(full, R, replace=False))
    prompt, rollout = live // (full // P), live % (full // P)
    left = r.integers(1, 1536, R)
    lens = _prompt_lens(r, case, P)
    starts = np.cumsum(lens) - lens
    steps, flat, bounds = np.zeros(n, STEP_DESC_DTYPE), [], []
    n_rows = n_bounds = 0
    for j in range(n):
        rows = np.flatnonzero(left > j) if (left > j).any() else np.array([0])
        p = prompt[rows]
        b = np.r_[np.flatnonzero(np.r_[True, p[1:] != p[:-1]]), len(p)]
        steps[j] = (len(rows), len(b) - 1, int(np.diff(b).max()), 0, n_rows, n_bounds)
        flat.append(np.stack([p, rollout[rows], np.full(len(rows), s0 + j), rows * cap, rows * cap + s0 + j]))
        bounds.append(b)
        n_rows, n_bounds = n_rows + len(rows), n_bounds + len(b)
    flat = np.concatenate(flat, axis=1)
    steps = np.ascontiguousarray(steps)
    s = dict(run=_run_score if case["logits"] else _run_decode, model=k, P=P, n=n, steps=steps,
             steps_dev=_dev(steps.view(np.uint8).reshape(-1), torch.uint8), prompt=_dev(flat[0], torch.int32),
             rollout=_dev(flat[1], torch.int32), step=_dev(flat[2], torch.int32), kv_start=_dev(flat[3], torch.int64),
             tok_index=_dev(flat[4], torch.int64), bounds=_dev(np.concatenate(bounds), torch.int32), prompt_len=_dev(lens, torch.int32),
             prompt_start=_dev(starts, torch.int64), prompt_slots=int(lens.sum()), suffix_slots=R * cap,
             prompt_kv=_arena(m, int(lens.sum()), gen), suffix_kv=_arena(m, R * cap, gen),
             tokens=torch.randint(0, m.vocab, (R * cap,), dtype=torch.int32, device="cuda", generator=gen),
             logprobs=None, logits=None, sample=B.SampleParams(1.0, SAMPLE_SEED))
    if case["logprobs"]:                    # what the rollouts' tokens so far were drawn with: about -ln V
        s["logprobs"] = torch.empty(R * cap, device="cuda").normal_(-math.log(m.vocab), 0.8, generator=gen)
    if case["logits"]:
        s["logits"] = torch.empty((int(steps["n_rows"][0]), m.vocab), device="cuda")
    return s


# ----------------------------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------------------------
def run(state):
    return state["run"](state)


def _run_groups(s):
    P = s["P"]
    B.pc_reward_last_token(P * s["G"], s["tokens"], s["last"], s["threshold"], s["rewards"])
    B.pc_group_stats(P, s["rewards"], s["start"], s["pilot"], s["n"], s["success"], s["mean"], s["var"])
    B.pc_allocate(P, s["success"], s["n"], s["params"], s["status"], s["extra"], s["evict"], s["selected"], s["total"])
    B.pc_group_stats(P, s["rewards"], s["start"], s["union"], s["union_n"], s["union_success"], s["union_mean"], s["union_var"])
    B.pc_grpo_advantage(P, s["rewards"], s["start"], s["union"], s["status"], s["advantage"])
    return [s[k] for k in ("rewards", "n", "success", "mean", "var", "status", "extra", "evict", "selected", "total", "union_n",
                           "union_success", "union_mean", "union_var", "advantage")]


def _run_step(s):
    got = s["eng"].pilot_commit_step(s["workload"], s["batch"])
    keys = ("rewards", "generated", "pilot_n", "pilot_success", "pilot_mean", "pilot_var", "status", "extra", "evict", "n_selected",
            "total_rollouts", "union_n", "union_success", "union_mean", "union_var", "advantages", "generated_tokens")
    return {"tokens": s["eng"].tokens, **{k: got[k] for k in keys}}


def _run_prefill(s):
    B.pc_prefill_shared(s["model"].ctx, s["P"], s["tokens"], s["offsets"], s["total"], s["longest"], s["kv"], s["slots"], s["start"],
                        s["logits"])
    return s["kv"], s["logits"]


def _run_decode(s):
    ctx = s["model"].ctx
    B.pc_set_index_bounds(ctx, s["P"], s["tokens"].numel())
    B.pc_set_logprob_buffer(ctx, s["logprobs"])
    B.pc_decode_run(ctx, s["n"], s["steps"].ctypes.data_as(ctypes.c_void_p), s["steps_dev"], s["prompt"], s["rollout"], s["step"],
                    s["kv_start"], s["tokens"], s["tok_index"], s["bounds"], s["prompt_len"], s["prompt_kv"], s["prompt_slots"],
                    s["prompt_start"], s["suffix_kv"], s["suffix_slots"], s["sample"])
    return s["tokens"], s["logprobs"]


def _run_score(s):
    ctx, d = s["model"].ctx, s["steps"][0]
    B.pc_set_index_bounds(ctx, s["P"], s["tokens"].numel())
    B.pc_set_logprob_buffer(ctx, None)
    B.pc_decode_step(ctx, int(d["n_rows"]), s["prompt"], s["rollout"], s["step"], s["kv_start"], s["tokens"], s["tok_index"],
                     int(d["n_groups"]), s["bounds"], int(d["max_group_rows"]), s["prompt_len"], s["prompt_kv"], s["prompt_slots"],
                     s["prompt_start"], s["suffix_kv"], s["suffix_slots"], s["logits"], None)
    return s["logits"]


# ----------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------------------------------
def _decode_work(m, rows, groups, suffix, prompt_len, logits):
    """One decode step: the matrices once, every suffix once, every group's prompt once, the new K/V and what is handed back."""
    params = m.weight_bytes_per_decode_step() // m.elem_bytes
    kv = m.kv_bytes_per_token * (rows * (suffix + 2) + groups * prompt_len)
    return (m.weight_bytes_per_decode_step() + kv + rows * (4 * m.vocab if logits else 8),
            2.0 * rows * params + 4.0 * rows * m.q_dim * m.n_layers * (suffix + 1 + prompt_len))


def _prefill_work(m, prompts, mean_len):
    tokens = prompts * mean_len
    nbytes = m.n_layers * m.layer_params() * m.elem_bytes + m.vocab * m.d_model * m.elem_bytes + tokens * m.kv_bytes_per_token + 4 * prompts * m.vocab
    return nbytes, 2.0 * tokens * m.n_layers * m.layer_params() + 2.0 * tokens * mean_len * m.q_dim * m.n_layers + 2.0 * prompts * m.vocab * m.d_model


def work(case):
    if case["kind"] == "groups":
        n = case["prompts"] * case["group"]
        return {"bytes": 24 * n + 80 * case["prompts"], "flops": 20 * n}
    m, mean_len = MODELS[case["model"]], (case["prompt_lo"] + case["prompt_hi"]) / 2
    if case["kind"] == "prefill":
        b, f = _prefill_work(m, case["prompts"], mean_len)
        return {"bytes": b, "flops": f}
    if case["kind"] == "step":
        # the pilot stage and, for about half of the prompts, the commit stage
        b, f = _prefill_work(m, case["prompts"], mean_len)
        cap = (case["cap_lo"] + case["cap_hi"]) / 2
        for prompts, each in ((case["prompts"], case["pilot"]), (case["prompts"] // 2, case["group"] - case["pilot"])):
            if prompts * each:
                x, y = _decode_work(m, prompts * each, prompts, cap / 2, mean_len, False)
                b, f = b + x * (cap - 1), f + y * (cap - 1)
        return {"bytes": b, "flops": f}
    b, f = _decode_work(m, case["rows"], case["groups"], case["suffix"], mean_len, case["logits"])
    return {"bytes": b * case["steps"], "flops": f * case["steps"]}


def tolerance(case):
    if case["kind"] in ("groups", "step"):
        return {"rel": 1e-5}                # float32; tokens, counts and decisions stay the same
    if case["kind"] == "prefill":
        return {"rel": 1e-2}
    # 16-bit operands: a logit moves by up to about 1 % of the logits' spread (2 % where the operands are bfloat16), so now
    # and then the two best perturbed scores of a row change places, and the rollout goes on with the other token
    return {"rel": 1e-2 if case["half"] else 2e-2, "differ": 5e-3}
