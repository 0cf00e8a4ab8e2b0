"""Decode with the rows split evenly over a wave of warps, the parts of a segment merged by the last warp to finish:
one sequence far longer than the rest, few segments, in every head dimension and type, over open spans and rings that
wrap, layer by layer of a call over several, and with the static scratch.  Every output against the fp64 oracle; the
plan is told from the others of its mode by its rows per tile and its warps."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import harness
import oracle as orc
import oracle.workload as ow
import paper_2310_08152_gb300 as kvc
from synth import workloads as wl

from _parity import compare, run_workload

pytestmark = pytest.mark.gpu


def _long_short(d, dtype, rot=0, M=1, long=4500, spans=False):
    """One sequence of `long` tokens and one of 70, 8 heads: the long segments are past what a cluster of 8 takes."""
    w = wl.opt13b(b=2, L=64, M=M)
    k, sp = wl.block_kinds(2 * long, 32) if spans else (np.zeros(long, np.uint8), [])
    ks, ss = wl.block_kinds(70, 8)
    return dataclasses.replace(w, H=8, d=d, dtype=dtype, rotary_dim=rot, scale=1.0 / math.sqrt(d), prompt_kinds=[k, ks],
                               prompt_spans=[sp, ss], name=f"long-short-d{d}-{dtype}-r{rot}")


def _is_split(plan, d):
    # 2 rows per lane of 16 (d_head 64, 80) or 8 row groups, a warp per 30 rows or so
    return plan["mode"] == 0 and plan["tile_rows"] == (32 if d <= 80 else 16) and plan["workers"] > 1000


@pytest.mark.parametrize("d,dtype,rot,policy", [
    (64, "f16", 0, orc.POLICY_PAPER), (64, "bf16", 64, orc.POLICY_KEEP_CL), (80, "f16", 80, orc.POLICY_PAPER),
    (80, "bf16", 0, orc.POLICY_PAPER), (96, "f16", 32, orc.POLICY_KEEP_CL), (96, "bf16", 96, orc.POLICY_PAPER),
    (128, "f16", 128, orc.POLICY_PAPER), (128, "bf16", 0, orc.POLICY_KEEP_CL)])
def test_split_rows(d, dtype, rot, policy):
    """Three steps: a <CL>, which sees itself, and two tokens in its open span, whose <CL> row is hidden from them
    under the paper policy; the segments of the long sequence in some 150 parts each."""
    run, _ = run_workload(_long_short(d, dtype, rot), steps=3, policy=policy)
    assert _is_split(run.cache.last_decode_plan, d), run.cache.last_decode_plan


def test_split_rows_after_a_compaction():
    run, _ = run_workload(_long_short(64, "f16", spans=True), steps=3)
    assert _is_split(run.cache.last_decode_plan, 64), run.cache.last_decode_plan


@pytest.mark.parametrize("d,dtype,slot", [(64, "f16", 4502), (80, "bf16", 6000), (128, "f16", 5000)])
def test_split_rows_of_a_ring(d, dtype, slot):
    """Local Attention windows of 4,500 and 70 rows in rings whose end comes two rows, 1,500 or 500 into the window."""
    w = dataclasses.replace(_long_short(d, dtype), prompt_kinds=[np.zeros(9000, np.uint8), np.zeros(140, np.uint8)],
                            prompt_spans=[[], []], gen_kind=lambda s, g: 0)
    run = harness.Runner(w, 3, kvc.POLICY_LOCAL, local_ratio=0.5, capacity=[slot, 100])
    run.load_prompt()
    out = torch.empty(w.M, w.b, w.H, w.d, dtype=torch.float32, device="cuda")
    for g in range(3):
        run.step(run.make_step_inputs(g), out)
        torch.cuda.synchronize()
        compare(out[0].cpu().numpy(), ow.expected_local_decode(w, g + 1, 0, [0, 1], 0.5), f"step {g}")
        assert _is_split(run.cache.last_decode_plan, d), run.cache.last_decode_plan
    assert run.cache.device_status() == 0


@pytest.mark.parametrize("d,dtype", [(64, "f16"), (96, "bf16")])
def test_split_rows_layer_by_layer_and_with_the_static_scratch(d, dtype):
    """A call over three layers launches each, as the calls for one layer do; the static scratch, which keeps the last
    call's parts and counters, gives the same bits twice."""
    w = dataclasses.replace(_long_short(d, dtype, M=3), gen_kind=lambda s, g: 0)
    run = harness.Runner(w, 1)
    run.load_prompt()
    inp = run.make_step_inputs(0)
    run.append_only(inp)
    l0 = run.cache.launch_count
    many = run.cache.decode_attention_layers(inp.q, w.scale)
    assert run.cache.launch_count == l0 + w.M
    assert _is_split(run.cache.last_decode_plan, d), run.cache.last_decode_plan
    other = torch.full((3, w.M, w.b, w.H, w.d), float("nan"), device="cuda")
    for m in range(w.M):
        kvc.kvc_decode_attention(run.cache.handle, m, inp.q[m], w.scale, other[0, m])
        for rep in (1, 2):
            kvc.kvc_decode_attention_static_scratch(run.cache.handle, m, inp.q[m], w.scale, other[rep, m])
            assert _is_split(run.cache.last_decode_plan, d), run.cache.last_decode_plan
    torch.cuda.synchronize()
    for x in other:
        assert torch.equal(x, many)
    for m in range(w.M):
        compare(many[m].cpu().numpy(), ow.expected_decode(w, 1, m, [0, 1]), f"layer {m}")
    assert run.cache.device_status() == 0
