"""Decode with a CTA or a cluster of CTAs per (layer, sequence, head) segment, or several consecutive
segments per CTA.  Every output against the fp64 oracle at the sizes where the split can
go wrong: clusters of 8, 4 and 2, rows just below, at and above a tile, CTAs of a cluster without rows,
rings that wrap, open spans, the small shape, several segments per CTA, and unbalanced segments."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import harness
import oracle as orc
import oracle.workload as ow
from synth import workloads as wl

from _parity import compare, run_workload

pytestmark = pytest.mark.gpu


def _with(w, **kw):
    d = kw.get("d", w.d)
    return dataclasses.replace(w, scale=1.0 / math.sqrt(d), name="-".join([w.name] + [f"{k}{v}" for k, v in kw.items()]), **kw)


def _lengths(lens, M=1):
    """Prompts of the given lengths, spans of 32 in every 64 tokens."""
    w = wl.opt13b(b=len(lens), L=64, M=M)
    made = [wl.block_kinds(n, 32) for n in lens]
    return dataclasses.replace(w, prompt_kinds=[k for k, _ in made], prompt_spans=[s for _, s in made], name=f"lens{lens}")


# workload, steps, rows per tile and warps (None: not looked at) of the plan after the last step
CASES = [
    ("cluster of 8", lambda: wl.opt13b(b=1, L=4000, M=1), 3, 128, 32 * 8 * 4),
    ("cluster of 4, d 80 rotary", lambda: wl.rope3b(32, b=2, L=2048, M=1), 3, 128, 64 * 4 * 4),
    ("cluster of 2, bf16, d 128", lambda: _with(wl.opt13b(b=4, L=1000, M=1), dtype="bf16", d=128), 3, 64, 128 * 2 * 4),
    ("cluster of 4, a short sequence", lambda: _lengths([3000, 40]), 3, 128, 64 * 4 * 4),
    ("about a tile of rows, two layers", lambda: wl.opt13b_uncompressed(b=2, L=126, M=2), 3, 128, 128 * 4),
    ("about a tile of rows, d 96", lambda: _with(wl.opt13b_uncompressed(b=2, L=62, M=1), d=96, rotary_dim=32), 3, 64, 64 * 4),
    ("small shape", lambda: wl.opt13b(b=12, L=200, M=1), 3, 64, 384 * 2),
    ("small shape, d 80 bf16 rotary", lambda: _with(wl.rope3b(32, b=11, L=180, M=1), dtype="bf16"), 3, 64, 352 * 2),
    ("several segments per CTA", lambda: wl.opt13b(b=21, L=900, M=1), 3, 128, 224 * 4),
    ("a segment per CTA, many waves, d 128", lambda: _with(wl.opt13b_uncompressed(b=40, L=170, M=2), d=128), 2, 64, 2560 * 4),
    ("unbalanced, beyond a wave", lambda: wl.ragged(b=20, lmin=300, lmax=2000, M=1, steps=4), 3, 128, 640 * 4),
    ("unbalanced, short, two per CTA", lambda: wl.ragged(b=21, lmin=60, lmax=400, M=1, steps=4), 3, 64, 336 * 2),
    ("unbalanced, short, d 80, two per CTA", lambda: _with(wl.ragged(b=21, lmin=60, lmax=400, M=1, steps=4), d=80), 3, 128, 336 * 4),
    ("unbalanced layers in one launch", lambda: wl.ragged(b=12, lmin=300, lmax=2000, M=2, steps=4), 3, 128, 768 * 4),
]


@pytest.mark.parametrize("name,make,steps,tile,warps", CASES, ids=[c[0] for c in CASES])
def test_cta_per_segment(name, make, steps, tile, warps):
    run, _ = run_workload(make(), steps=steps)
    plan = run.cache.last_decode_plan
    assert plan["mode"] in (0, 1, 4), plan
    assert plan["tile_rows"] == tile and (warps is None or plan["workers"] == warps), plan


def test_ring_that_wraps_over_a_cluster():
    """A Local Attention window cut over a cluster of 4 CTAs, its ring's end inside one CTA's rows."""
    w = wl.opt13b_local(b=2, L=1700, M=1)
    run = harness.Runner(w, steps=3)
    run.load_prompt()
    out = torch.empty(w.M, w.b, w.H, w.d, dtype=torch.float32, device="cuda")
    for g in range(3):
        run.step(run.make_step_inputs(g), out)
        torch.cuda.synchronize()
        ref = ow.expected_local_decode(w, g + 1, 0, [0, 1], float(np.float32(0.5)))
        compare(out[0].cpu().numpy(), ref, f"step {g}")
    plan = run.cache.last_decode_plan
    assert plan["workers"] == 64 * 4 * 4, plan
    assert run.cache.device_status() == 0


def test_open_span_hidden_row_in_every_part():
    """A span opened while generating: its <CL> row, hidden under the paper policy, among the last rows of a
    cluster's last CTA."""
    for policy in (orc.POLICY_PAPER, orc.POLICY_KEEP_CL):
        w = wl.opt13b(b=2, L=1600, M=1)
        run_workload(w, steps=4, policy=policy)


# (hidden from the query at row 1600 by an open <CL> or by a closed span not freed yet, which of the two sequences)
# A cluster of 4 takes rows 0-400, 401-801, 802-1202 and 1203-1600 of 1,601.
HIDDEN = [[("open", 400), ("open", 401)], [("open", 801), ("open", 802)], [("open", 1202), ("open", 1203)],
          [("open", 0), ("open", 1599)], [("span", 390, 420), ("span", 0, 401)], [("span", 300, 1500), ("span", 401, 802)],
          [("span", 1202, 1599), ("span", 1201, 1204)]]


@pytest.mark.parametrize("policy", [orc.POLICY_PAPER, orc.POLICY_KEEP_CL])
@pytest.mark.parametrize("hidden", HIDDEN, ids=str)
def test_hidden_rows_at_the_ctas_of_a_cluster(hidden, policy):
    """Hidden rows at every CTA's first and last row, across two CTAs' rows, and all rows of one or two CTAs."""
    kinds = [np.zeros(1600, np.uint8) for _ in hidden]
    for k, (what, *at) in zip(kinds, hidden):
        k[at[0]] = wl.CL
        if what == "span":
            k[at[1]] = wl.CR
    w = dataclasses.replace(wl.opt13b(b=2, L=64, M=1), prompt_kinds=kinds, prompt_spans=[[], []], gen_kind=lambda s, g: 0)
    run = harness.Runner(w, 1, policy)
    run.load_prompt()
    inp = run.make_step_inputs(0)
    run.append_only(inp)
    out = run.cache.decode_attention(0, inp.q[0], w.scale)
    plan = run.cache.last_decode_plan
    assert plan["workers"] == 64 * 4 * 4, plan
    compare(out.cpu().numpy(), ow.expected_decode(w, 1, 0, [0, 1], None, policy), str(hidden))
    assert run.cache.device_status() == 0


def _few_long(d, dtype, b, short, n_long, factor, M):
    """Prompts of about `short` tokens and n_long of `factor` times that, no spans."""
    rng = np.random.default_rng(b + short)
    lens = rng.integers(int(0.7 * short), int(1.3 * short), b)
    lens[rng.permutation(b)[:n_long]] = factor * short
    w = wl.opt13b(b=b, L=64, M=M)
    return dataclasses.replace(w, d=d, dtype=dtype, scale=1.0 / math.sqrt(d), prompt_kinds=[np.zeros(n, np.uint8) for n in lens],
                               prompt_spans=[[] for _ in lens], gen_kind=lambda s, g: 0, name=f"few-long-d{d}")


# few long sequences among many: the plan, and its rows per tile, of one call for all layers
FEW_LONG = [
    ("d 64, wide", lambda: _few_long(64, "f16", 90, 900, 1, 8, 24), 4, 128),
    ("d 80 bf16, wide", lambda: _few_long(80, "bf16", 90, 700, 1, 8, 24), 4, 96),
    ("d 96, wide", lambda: _few_long(96, "f16", 160, 300, 1, 7, 24), 4, 32),
    ("d 128 bf16, wide", lambda: _few_long(128, "bf16", 120, 250, 1, 8, 24), 4, 32),
    ("d 64, narrow", lambda: _few_long(64, "f16", 220, 200, 1, 8, 24), 4, 32),
    ("d 64, too long a sequence", lambda: _few_long(64, "f16", 60, 300, 1, 12, 24), 0, 32),
    ("d 64, longer than a CTA's share", lambda: _few_long(64, "f16", 18, 1500, 1, 4, 1), 0, 32),
    ("d 64, within a CTA's share of two layers", lambda: _few_long(64, "f16", 18, 1500, 1, 4, 2), 4, 128),
]


@pytest.mark.parametrize("name,make,mode,tile", FEW_LONG, ids=[c[0] for c in FEW_LONG])
def test_a_few_long_sequences_over_layers(name, make, mode, tile):
    """Runs of whole segments per warp, cut by rows, in the wide and the narrow shape, and the layers one by one
    where a warp would hold too much: the first, a middle and the last layer against the oracle."""
    w = make()
    run = harness.Runner(w, steps=1)
    run.load_prompt()
    out = torch.full((w.M, w.b, w.H, w.d), float("nan"), dtype=torch.float32, device="cuda")
    inp = run.make_step_inputs(0)
    run.append_only(inp)
    run.cache.decode_attention_layers(inp.q, w.scale, out=out)
    plan = run.cache.last_decode_plan
    assert plan["mode"] == mode and plan["tile_rows"] == tile, plan
    lens = [k.size for k in w.prompt_kinds]
    seqs, heads = [int(np.argmax(lens)), int(np.argmin(lens)), w.b - 1], [0, 31]
    assert torch.isfinite(out).all()
    for m in (0, w.M // 2, w.M - 1):
        compare(out[m].cpu().numpy()[seqs][:, heads], ow.expected_decode(w, 1, m, seqs, heads, orc.POLICY_PAPER), f"layer {m}")
    assert run.cache.device_status() == 0


# balanced segments too short for a CTA each: mode (2: one warp a segment, 3: several), rows per tile
SHORT = [
    ("d 80, several a warp", lambda: _with(wl.opt13b_uncompressed(b=40, L=400, M=2), d=80), 3, 32),
    ("d 96, one wide warp each", lambda: _with(wl.opt13b_uncompressed(b=22, L=250, M=1), d=96), 2, 32),
    ("d 96, several a wide warp", lambda: _with(wl.opt13b_uncompressed(b=40, L=250, M=2), d=96, dtype="bf16"), 3, 32),
    ("d 96, several a narrow warp", lambda: _with(wl.opt13b_uncompressed(b=40, L=170, M=2), d=96), 3, 16),
    ("d 128, several a wide warp", lambda: _with(wl.opt13b_uncompressed(b=43, L=250, M=2), d=128), 3, 32),
]


@pytest.mark.parametrize("d,dtype,rot,b,L,M,mode", [(96, "f16", 32, 40, 500, 2, 3), (128, "bf16", 64, 43, 470, 2, 3), (96, "bf16", 96, 22, 500, 1, 2)])
@pytest.mark.parametrize("policy", [orc.POLICY_PAPER, orc.POLICY_KEEP_CL])
def test_whole_segments_per_wide_warp_with_an_open_span(d, dtype, rot, b, L, M, mode, policy):
    """Compacted prompts, rotary positions, and a span opened while generating, whose <CL> row the paper policy hides."""
    run, _ = run_workload(_with(wl.opt13b(b=b, L=L, M=M), d=d, dtype=dtype, rotary_dim=rot), steps=3, policy=policy,
                          seqs=[0, b // 2, b - 1], heads=[0, 31])
    plan = run.cache.last_decode_plan
    assert plan["mode"] == mode and plan["tile_rows"] == 32, plan


def test_whole_segments_per_wide_warp_of_rings():
    """Windows of 250 rows, the ring's end at another row in each step."""
    w = _with(wl.opt13b_local(b=40, L=500, M=2), d=96)
    run = harness.Runner(w, steps=4, capacity_slack=9)
    run.load_prompt()
    out = torch.empty(w.M, w.b, w.H, w.d, dtype=torch.float32, device="cuda")
    for g in range(4):
        run.step(run.make_step_inputs(g), out)
        torch.cuda.synchronize()
        assert run.cache.last_decode_plan["mode"] == 3 and run.cache.last_decode_plan["tile_rows"] == 32
        for m in range(w.M):
            ref = ow.expected_local_decode(w, g + 1, m, [0, 20, 39], float(np.float32(0.5)), [0, 31])
            compare(out[m].cpu().numpy()[[0, 20, 39]][:, [0, 31]], ref, f"step {g} layer {m}")
    assert run.cache.device_status() == 0


@pytest.mark.parametrize("name,make,mode,tile", SHORT, ids=[c[0] for c in SHORT])
def test_whole_segments_per_warp(name, make, mode, tile):
    run, _ = run_workload(make(), steps=2, seqs=[0, 7, 21], heads=[0, 13, 31])
    plan = run.cache.last_decode_plan
    assert plan["mode"] == mode and plan["tile_rows"] == tile, plan
