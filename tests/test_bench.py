"""bench.py's host-side tables (no GPU: events are stand-ins)."""
import types

import pytest

import bench
from paper_2605_26606_b200 import binding as B
from paper_2605_26606_b200 import workloads as wl

EVENT_MS = 0.0027


class _Event:
    def __init__(self, at):
        self.at = at

    def elapsed_time(self, other):
        return other.at - self.at


def _samples(durations):
    """Marks as the library records them: every mark costs EVENT_MS, an operation between two marks its duration on top."""
    t, at = 0.0, {}
    for name in B.PROFILE_MARKS:
        t += durations.get(name, 0.0) + EVENT_MS
        at[name] = t
    return [([_Event(at[n]) for n in B.PROFILE_MARKS], 64, 1000)] * 2


@pytest.mark.parametrize("model,half,absent", [(wl.QWEN25_1P5B, True, {"norm_attn", "qkv_post", "attn_merge", "norm_mlp"}),
                                               (wl.QWEN25_1P5B, False, {"norm_attn", "qkv_post", "attn_merge"}),
                                               (wl.TINY_BF16, True, {"attn_merge"}), (wl.TINY, False, {"attn_prefix", "attn_merge"})],
                         ids=["half", "bfloat16", "head-dim-64", "float32"])
def test_phase_table_leaves_out_the_events_themselves(model, half, absent):
    """An operation that runs inside another kernel has no line, and no line holds the cost of the two events around it."""
    ms = {"qkv": 0.012, "group": 0.009, "suffix": 0.020, "o": 0.008, "norm_mlp": 0.004, "gate_up": 0.015, "down": 0.011, "lm_head": 0.090, "sample": 0.060}
    if "norm_mlp" in absent:
        ms.pop("norm_mlp")
    if "attn_prefix" in absent:
        ms.pop("group")
    eng = types.SimpleNamespace(profile_samples=_samples(ms), model=model, half_gemm=half)
    per_sample, avg, est = bench.phase_table(eng, B, model.n_layers)
    assert not absent & set(avg) and len(per_sample) == 2
    assert avg["attn_suffix"] == pytest.approx(0.020) and avg["gate_up_gemm"] == pytest.approx(0.015) and avg["sampler"] == pytest.approx(0.060)
    assert est["qkv_gemm"] == pytest.approx(0.012 * model.n_layers) and est["lm_head"] == pytest.approx(0.090)
    assert sum(est.values()) == pytest.approx(sum(v * (1 if k in ("lm_head", "sample") else model.n_layers) for k, v in ms.items()))
