"""Benchmark: decode steps over a sentinel-compressed KV cache on GB300.

One step = one pass of the whole hot path over a batch: append the new token's K/V rows (all layers),
single-query decode attention for every layer over the kept rows, and compaction of the span a <CR>
just closed.  Workload (default): the ragged stress cache, the largest one that fits one GPU (M=24,
H=32, d_head=64, fp16, b=128, prompts of U[256, 8192] tokens with half of them enclosed in sampled
spans, each sequence opening and closing one span during decode), seeded synthetic inputs already
resident in HBM.  Every step reads ~50 GB, far more than L2.  Beside the headline, the decode and
compaction roofline fractions of the OPT-1.3B-, OPT-2.7B- and 3B-rotary-shaped caches are measured in
the same run (`per_workload`).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME] [--impl kvc|reference]

Prints one JSON line (rank 0).  Multi-GPU (torchrun): every rank runs its own replica (the path
shards by sequence with no exchange); value = tokens of all ranks / max time over ranks.
"""
from __future__ import annotations

import argparse
import collections
import dataclasses
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "compressed-KV decode-attention tokens/s; achieved HBM GB/s vs ~8 TB/s peak"
UNIT = "tokens/s"
FALLBACK_HBM_GBS = 6800.0


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=128)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--workload", default="ragged",
                    help="headline workload (default: the ragged stress cache, the largest single-GPU one)")
    ap.add_argument("--per-workload", default="opt1.3b,opt2.7b,rope3b_I19,rope3b_I32,rope3b_I45",
                    help="workloads whose decode and compaction fractions are reported beside the headline "
                         "('' for none)")
    ap.add_argument("--per-workload-steps", type=int, default=16)
    ap.add_argument("--impl", default="kvc", choices=["kvc", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--e2e-reps", type=int, default=3, help="timed end-to-end windows (median reported)")
    ap.add_argument("--cpu-seconds", type=float, default=10.0, help="budget of the CPU-baseline sample")
    ap.add_argument("--layers", type=int, default=0, help="override the layer count (small profiling runs)")
    ap.add_argument("--ragged-lengths", default="",
                    help="LMIN,LMAX: prompt-length range of the ragged workload (small profiling runs)")
    ap.add_argument("--capacity-sweep", action="store_true",
                    help="largest batch under a KV-memory cap per compression ratio, and its throughput")
    ap.add_argument("--caps", default="12,24,180", help="KV-memory caps in GB for --capacity-sweep")
    ap.add_argument("--ratios", default="0,0.5,0.8,0.9", help="compression ratios for --capacity-sweep")
    ap.add_argument("--prefill-only", action="store_true",
                    help="only time the masked prefill of the workload's prompt (one JSON line per mode)")
    ap.add_argument("--prefill-block", type=int, default=-1,
                    help="with --prefill-only: block size (0 = one go; default: both 0 and 512)")
    return ap.parse_args()


def measured_hbm_peak():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            j = json.load(f)
        return float(j["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def measured_tensor_peak():
    """Dense 16-bit tensor-core TFLOP/s measured by a cuBLAS bf16 GEMM (burst); f16 runs at the same
    dense rate on these tensor cores."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            j = json.load(f)
        return float(j["bf16_tflops"]), "measured (bf16 GEMM burst; same dense rate for f16)"
    except Exception:
        return 1900.0, "fallback"


def kernel_source_hash() -> str:
    """Hash of the decode kernel's source: its device helpers, the kernel and its launcher."""
    csrc = os.path.join(ROOT, "paper_2310_08152_gb300/csrc")
    text = open(os.path.join(csrc, "kernels.cu")).read()
    marks = [("// a5 + a6: decode", "cudaError_t launch_append_t")]
    h = hashlib.sha256()
    h.update(open(os.path.join(csrc, "device_common.cuh")).read().encode())
    for a, b in marks:
        i = text.index(a)
        h.update(text[i:text.index(b, i)].encode())
    return h.hexdigest()[:16]


def recorded_traffic(workload: str, bytes_per_launch: float):
    """DRAM bytes (read + write) per decode launch from a committed ncu capture taken on this kernel
    source: the capture's DRAM bytes per algorithmic byte, scaled to this run's algorithmic bytes per
    launch (the capture is a smaller case of the same plan; the ratio, not the size, carries over)."""
    p = os.path.join(ROOT, "profiles", "decode_traffic.json")
    try:
        with open(p) as f:
            j = json.load(f)
    except Exception:
        return None
    rec = j.get(workload)
    if not rec or rec.get("kernel_source_hash") != kernel_source_hash():
        return None
    return rec["dram_bytes_per_algorithmic_byte"] * bytes_per_launch


class ClockSampler:
    """SM clock and clock-event (throttle) reasons sampled every 50 ms while the timed region runs.

    Sampling NVML every 2 ms slowed the end-to-end steps by about 10 % (the GPU's own time, with copies
    on two more streams); every 50 ms had no measurable effect.

    Reads NVML (libnvidia-ml) through ctypes; falls back to `nvidia-smi -lms` when NVML is not
    loadable.  Only reads state; changes nothing on the GPU."""

    REASONS = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown", 0x40: "hw_thermal_slowdown",
               0x80: "hw_power_brake_slowdown"}

    def __init__(self, gpu_index: int, period_s: float = 0.05):
        self.gpu = gpu_index
        self.period = period_s
        self.samples = []
        self.thread = None
        self.proc = None
        self.nvml = None
        try:
            import ctypes

            lib = ctypes.CDLL("libnvidia-ml.so.1")
            if lib.nvmlInit_v2() == 0:
                dev = ctypes.c_void_p()
                if lib.nvmlDeviceGetHandleByIndex_v2(ctypes.c_uint(gpu_index), ctypes.byref(dev)) == 0:
                    self.nvml = (lib, dev)
        except Exception:
            self.nvml = None

    def _read(self):
        import ctypes

        lib, dev = self.nvml
        clk, mx, rs = ctypes.c_uint(), ctypes.c_uint(), ctypes.c_ulonglong()
        if lib.nvmlDeviceGetClockInfo(dev, 1, ctypes.byref(clk)) != 0:
            return None
        lib.nvmlDeviceGetMaxClockInfo(dev, 1, ctypes.byref(mx))
        fn = getattr(lib, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            getattr(lib, "nvmlDeviceGetCurrentClocksThrottleReasons")
        fn(dev, ctypes.byref(rs))
        return clk.value, mx.value, rs.value

    def _loop(self):
        while not self._stop:
            r = self._read()
            if r:
                self.samples.append(r)
            time.sleep(self.period)

    def start(self):
        import threading

        self._stop = False
        if self.nvml:
            self.thread = threading.Thread(target=self._loop, daemon=True)
            self.thread.start()
            return
        fields = ("index,clocks.sm,clocks.max.sm,clocks_event_reasons.hw_slowdown,"
                  "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
                  "clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={fields}",
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        self._stop = True
        if self.thread is not None:
            self.thread.join()
            if not self.samples:
                return None
            sm = [c for c, _, _ in self.samples]
            reasons = set()
            for _, _, r in self.samples:
                for bit, name in self.REASONS.items():
                    if r & bit:
                        reasons.add(name)
            return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(m for _, m, _ in self.samples),
                    "reasons": sorted(reasons), "samples": len(sm), "source": "nvml"}
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 7:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[3:7]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm), "source": "nvidia-smi"}


# ------------------------------------------------------------------------------------------------
# CPU oracle timing (the reported CPU baseline, and the reference arm)
# ------------------------------------------------------------------------------------------------

class OracleSample:
    """Full-length masked decode of a set of layers for every sequence of the workload, by the fp64
    oracle on the host cores.  K/V of those layers are generated once for the whole capacity (not
    timed)."""

    def __init__(self, w, steps_total: int, layers=(0,)):
        import oracle
        import oracle.workload as ow

        self.oracle, self.ow, self.w, self.layers = oracle, ow, w, list(layers)
        self.K, self.V = {}, {}
        for m in self.layers:
            self.K[m], self.V[m] = [], []
            for s in range(w.b):
                T = int(w.prompt_len[s]) + steps_total
                K, V = ow.kv_bits(w, m, s, T)
                self.K[m].append(K)
                self.V[m].append(V)
        self.threads = oracle.max_threads()

    def time_step(self, g: int, layer: int = 0) -> float:
        """Seconds the oracle takes for one layer of decode step g (query = generated token g)."""
        w, ow = self.w, self.ow
        kinds_l, pos_l, K_l, V_l, q_l = [], [], [], [], []
        for s in range(w.b):
            kinds, pos = ow.history(w, s, g + 1)
            T = kinds.size
            kinds_l.append(kinds)
            pos_l.append(pos)
            K_l.append(np.ascontiguousarray(self.K[layer][s][:, :T]))
            V_l.append(np.ascontiguousarray(self.V[layer][s][:, :T]))
            q_l.append(ow.q_bits(w, layer, s, T - 1))
        q = np.stack(q_l)
        t0 = time.perf_counter()
        self.oracle.masked_decode(kinds_l, pos_l, K_l, V_l, q, w.dtype, w.scale, rot=w.rotary_dim,
                                  base=w.rope_base)
        return time.perf_counter() - t0

    def tokens_per_s(self, seconds_per_layer: float) -> float:
        return self.w.b / (seconds_per_layer * self.w.M)


def cpu_baseline(w, steps_total: int, budget_s: float):
    samp = OracleSample(w, steps_total)
    times = []
    t_start = time.perf_counter()
    g = 0
    while True:
        times.append(samp.time_step(g % steps_total))
        g += 1
        if time.perf_counter() - t_start >= budget_s or g >= steps_total:
            break
    per_layer = sum(times) / len(times)
    return {"value": samp.tokens_per_s(per_layer), "unit": UNIT, "cores": samp.threads, "kind": "oracle",
            "sample": f"fp64 oracle, full-length masked decode of layer 0 for all {w.b} sequences at {len(times)} "
                      f"decode steps (mean {per_layer * 1e3:.1f} ms per layer), scaled by M={w.M} layers; "
                      "K/V generation not timed"}


# All layers of a step are timed when their K/V history fits this many bytes of host memory; beyond
# it (the 2.7B- and 3B-shaped caches, the ragged one) one layer per step is timed and scaled by M.
REFERENCE_ALL_LAYERS_BYTES = 8 << 30


# ------------------------------------------------------------------------------------------------
# arms
# ------------------------------------------------------------------------------------------------

def dist_setup(n_gpus: int):
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world != n_gpus and world > 1:
        raise SystemExit(f"--gpus {n_gpus} but WORLD_SIZE={world}")
    return rank, world, local


def reference_layers(w, steps_total: int):
    """Layers the reference arm times per step, and the bytes of the whole K/V history (all layers)."""
    hist_bytes = 2 * 2 * w.M * w.H * w.d * int((w.prompt_len + steps_total).sum())
    return (list(range(w.M)) if hist_bytes <= REFERENCE_ALL_LAYERS_BYTES else [0]), hist_bytes


def run_reference(args, w):
    """The reference arm: the fp64 oracle on the host cores, full-length masked decode of every
    sequence under the paper's mask.  A step times every layer when the whole K/V history fits
    REFERENCE_ALL_LAYERS_BYTES of host memory, else layer 0 alone (layers are independent and
    processed identically) and the step's all-layer time is extrapolated by M.  ms_per_step is the
    host time the timed layers took, so ms_per_step x steps is what ran; with a sampled step the line
    says so (extrapolated, layers_timed_per_step) and gives the extrapolated step time beside it."""
    rank, world, _ = dist_setup(args.gpus)
    if rank != 0:
        return
    steps_total = args.warmup + args.steps
    layers, hist_bytes = reference_layers(w, steps_total)
    samp = OracleSample(w, steps_total, layers)
    for g in range(args.warmup):
        samp.time_step(g, layers[0])
    step_s = []
    for k in range(args.steps):
        step_s.append(sum(samp.time_step(args.warmup + k, m) for m in layers))
    per_layer = sum(step_s) / (len(step_s) * len(layers))
    value = samp.tokens_per_s(per_layer)
    sampled = len(layers) < w.M
    what = (f"every layer ({w.M})" if not sampled else
            f"layer 0 of {w.M} (the {hist_bytes / 2**30:.0f} GiB K/V history does not fit the host budget), "
            f"scaled by M")
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": sum(step_s) / len(step_s) * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded counter-based generator)",
        "config": workload_config(w),
        "extrapolated": sampled, "layers_timed_per_step": len(layers),
        "ms_per_step_all_layers": per_layer * w.M * 1e3,
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": samp.threads, "kind": "oracle",
                         "sample": f"each step: fp64 oracle full-length masked decode of all {w.b} sequences, "
                                   f"{what}; K/V generation not timed"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def workload_config(w):
    L = w.prompt_len
    return {"workload": f"{w.name}: {w.note}", "M": w.M, "H": w.H, "d_head": w.d, "b": w.b,
            "prompt_len": int(L[0]) if np.all(L == L[0]) else f"{int(L.min())}..{int(L.max())}",
            "kv_dtype": w.dtype, "accum": "f32", "rope": bool(w.rotary_dim), "parallelism": "replicas",
            "l2": "inputs larger than L2 (every step reads GBs of distinct K/V rows)"}


def aggregate(local_tokens: int, local_elapsed: float, device=None):
    """Whole-job tokens (sum over ranks) and elapsed time (max over ranks); identity on one rank."""
    import torch
    import torch.distributed as dist

    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return local_tokens, local_elapsed
    t = torch.tensor([float(local_elapsed)], dtype=torch.float64, device=device)
    n = torch.tensor([float(local_tokens)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(n, op=dist.ReduceOp.SUM)
    return int(n.item()), float(t.item())


def time_prompt_compaction(run, w):
    """Frees every prompt span in one go (one compaction over all sequences and layers) and reports
    the row-move bandwidth: bytes = 2 (read + write) x moved rows x row bytes x M x 2 (K, V) x H,
    over the device time of the two kernels (the library's events before the scan, between the
    kernels and after the row moves).  call_ms is the whole call measured from an idle stream: it
    also holds the host's planning of the compaction, which a decode loop overlaps with the GPU."""
    import torch

    import paper_2310_08152_gb300 as kvc

    kvc.kvc_set_compaction_timing(run.cache.handle, True)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    run.compress_prompt()
    e1.record()
    torch.cuda.synchronize()
    call_ms = e0.elapsed_time(e1)
    scan_ms = move_ms = None
    if any(w.prompt_spans[s] for s in range(w.b)):  # else nothing was compacted (no spans)
        scan_ms, move_ms = kvc.kvc_last_compaction_ms(run.cache.handle)
    kvc.kvc_set_compaction_timing(run.cache.handle, False)
    ln = run.cache.lengths()[0]
    moved = 0
    for s in range(w.b):
        if w.prompt_spans[s]:
            first = min(a for a, _ in w.prompt_spans[s])  # first dropped row: nothing before it moves
            moved += int(ln[s]) - first
    nbytes = 2 * moved * w.d * 2 * w.M * 2 * w.H
    peak, kind = measured_hbm_peak()
    ms = (scan_ms + move_ms) if scan_ms is not None else None
    gbs = nbytes / (ms * 1e-3) / 1e9 if ms else None
    move_gbs = nbytes / (move_ms * 1e-3) / 1e9 if move_ms else None
    return {"kernels": "compact_scan_kernel + compact_move_kernel", "moved_rows_per_stream": moved,
            "bytes": nbytes, "ms": ms, "scan_ms": scan_ms, "move_ms": move_ms, "call_ms": call_ms,
            "achieved": gbs, "peak": peak, "unit": "GB/s", "frac": (gbs / peak) if gbs else None,
            "frac_of_8tbs": gbs / 8000.0 if gbs else None,
            "move_frac": (move_gbs / peak) if move_gbs else None, "peak_kind": kind}


def time_prompt_write_time_freeing(w, steps_total, dev):
    """The same prompts ingested with write-time freeing (spans never stored, nothing to compact):
    the append calls' time, against append + compaction of the one-go path."""
    import torch

    import harness

    run = harness.Runner(w, steps_total, device=dev)
    ev = []
    run.load_prompt(mode="free", timer=ev)
    torch.cuda.synchronize()
    ms = sum(a.elapsed_time(b) for a, b in ev)
    stored = int(run.cache.lengths()[0].sum())
    del run
    torch.cuda.empty_cache()
    return {"mode": "write-time freeing (kvc_append_free_closed)", "append_ms": ms,
            "rows_written_per_stream": stored, "rows_in_prompt_per_stream": int(w.prompt_len.sum())}


def prefill_work(w, block: int):
    """FLOPs of one layer's masked prefill over the prompt, summed over sequences and heads:
    (algorithmic) 4 d per visible (query, key) pair -- q.k and p.v over exactly the rows the mask
    leaves (Sec. 3.1) -- and (executed) 4 d x 128 x keys per key tile the kernel runs: of each
    128-query tile over the rows that no span hides before it, the interior of a span it begins in
    and its own rows, in tiles of 128, 112 or 64 keys.  The visible counts follow the per-row bounds
    of the library's host book: query iq sees rows i <= iq with hid(i) >= iq, a <CL> query only
    itself."""
    import paper_2310_08152_gb300 as kvc

    L = w.prompt_len
    book = kvc.Book(w.b, L + 1)
    start = np.zeros(w.b, np.int64)
    pairs = keys = 0
    kt = 128 if w.d > 80 else 64 if w.dtype == "bf16" else {64: 128, 80: 112}[w.d]
    while (start < L).any():
        n = L - start if block <= 0 else np.minimum(L - start, block)
        kinds = np.concatenate([w.prompt_kinds[s][start[s]:start[s] + n[s]] for s in range(w.b)]).astype(np.uint8)
        book.append(n.astype(np.int32), kinds)
        for s in range(w.b):
            if n[s] == 0:
                continue
            meta = book.prefill_keys(s, int(n[s]))
            hid, cl = meta >> 1, meta & 1
            ln = meta.size
            q0 = ln - int(n[s])
            iq = np.arange(q0, ln)
            cnt = (iq + 1) - np.searchsorted(np.sort(hid), iq, side="left")
            pairs += int(np.where(cl[iq] == 1, 1, cnt).sum())
            never = hid == 0x3FFFFFFF
            listed = np.concatenate([[0], np.cumsum(never)])  # rows that no span hides before each row
            for lo in range(q0, ln, 128):
                b0 = lo
                while b0 > 0 and not never[b0 - 1] and hid[b0 - 1] >= lo:
                    b0 -= 1
                own = int(listed[b0]) + lo - b0
                if 128 % kt == 0:
                    own = -(-own // kt) * kt
                keys += -(-(own + min(lo + 128, ln) - lo) // kt) * kt
        seq, cl_, cr_ = [], [], []
        for s in range(w.b):
            for a, c in book.pending_spans(s):
                seq.append(s)
                cl_.append(a)
                cr_.append(c)
        if seq:
            book.compress(seq, cl_, cr_)
        start = start + n
    return 4 * w.d * pairs * w.H, 4 * w.d * 128 * keys * w.H


def time_prompt_prefill(w, steps_total, dev, block: int):
    """Prompt ingestion with masked prefill attention of every layer (tensor cores), one go
    (block 0) or block by block with the closed spans freed in between; reports the prefill kernel's
    TFLOP/s (algorithmic: visible pairs only) against the measured dense 16-bit peak."""
    import torch

    import harness

    run = harness.Runner(w, steps_total, device=dev)
    ev = []
    run.prefill_prompt(block=block, events=ev)
    torch.cuda.synchronize()
    ms = [a.elapsed_time(b) for a, b in ev]
    status = run.cache.device_status()
    del run
    torch.cuda.empty_cache()
    alg, executed = prefill_work(w, block)
    total_s = sum(ms) / 1e3
    n_blocks = max(1, len(ms) // w.M)
    peak, kind = measured_tensor_peak()
    achieved = alg * w.M / total_s / 1e12
    return {"kernel": "prefill_kernel (tcgen05.mma, TMEM accumulators, TMA-swizzled K/V)",
            "mode": "one go" if block <= 0 else f"blocks of {block} tokens", "launches": len(ms),
            "ms_total": sum(ms), "ms_per_layer": sum(ms) / w.M, "blocks": n_blocks,
            "tflop_per_layer_algorithmic": alg / 1e12, "tflop_per_layer_executed": executed / 1e12,
            "achieved": achieved, "executed_tflops": executed * w.M / total_s / 1e12, "peak": peak,
            "unit": "TFLOP/s", "frac": achieved / peak, "peak_kind": kind, "device_status": status}


def run_capacity_sweep(args):
    """Largest batch whose compressed KV cache fits a memory cap, and its decode-step throughput, for
    several compression ratios: a synthetic restatement of the paper's throughput-vs-VRAM experiment
    (Sec. 4.3, Fig. 2 bottom right) and memory experiment (App. C, Fig. 4).  The cap covers the KV
    cache only (no model weights: this path has none).  Prompts are ingested with write-time freeing,
    so a sequence holds only its kept rows plus the generated ones."""
    import torch

    import harness
    import paper_2310_08152_gb300 as kvc
    from synth import workloads as wl

    torch.cuda.set_device(0)
    caps_gb = [float(x) for x in args.caps.split(",")]
    ratios = [float(x) for x in args.ratios.split(",")]
    steps = args.steps
    for cap_gb in caps_gb:
        for r in ratios:
            probe = wl.throughput_3b(r, b=1, steps=steps)
            kept = int(probe.prompt_len[0]) - sum(c - a for a, c in probe.prompt_spans[0])  # paper policy
            per_seq = probe.M * 2 * probe.H * probe.d * 2 * (kept + args.warmup + steps)
            b = int(cap_gb * 1e9 // per_seq)
            b = max(1, min(b, 4096))
            w = wl.throughput_3b(r, b=b, steps=steps)
            # capacity: only what a sequence stores (kept prompt rows + generated rows)
            run = harness.Runner(w, args.warmup + steps, capacity=np.full(b, kept + args.warmup + steps))
            run.load_prompt(mode="free")
            # every generated token is a normal token: one step's inputs serve every step (the values
            # read from the cache, not these, set the work)
            inp = run.make_step_inputs(0)
            out = torch.empty(w.M, w.b, w.H, w.d, dtype=torch.float32, device="cuda")
            for g in range(args.warmup):
                run.step(inp, out)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for g in range(args.warmup, args.warmup + steps):
                run.step(inp, out)
            e1.record()
            torch.cuda.synchronize()
            sec = e0.elapsed_time(e1) / 1e3
            kv_gb = run.cache.sizes["k"] * 2 / 1e9
            print(json.dumps({"sweep": "capacity", "kv_cap_gb": cap_gb, "ratio": r, "batch": b,
                              "kept_prompt_rows": kept, "kv_allocated_gb": kv_gb, "tokens_per_s": w.b * steps / sec,
                              "ms_per_step": sec / steps * 1e3, "status": run.cache.device_status()}), flush=True)
            del run, inp, out
            torch.cuda.empty_cache()


def timed_decode_steps(run, w, inputs, warmup: int, steps: int, world: int = 1, clocks=None):
    """Warm-up steps through the harness, then `steps` timed decode steps in a lean loop: device
    pointers are computed up front and the entry points are called directly, so the host enqueues
    faster than the GPU drains.  Each step: append the token (all layers), decode every layer in one
    kvc_decode_attention_layers call (one launch when the segments are balanced, else one per layer),
    free the span a <CR> closed.  An event pair around each step's decode call times the decode."""
    import torch
    import torch.distributed as dist

    import paper_2310_08152_gb300 as kvc

    dev = run.device
    out = torch.empty(w.M, w.b, w.H, w.d, dtype=torch.float32, device=dev)
    torch.cuda.synchronize()
    for g in range(warmup):
        run.step(inputs[g], out)
    dec = kvc.lib().kvc_decode_attention_layers
    stream_h = torch.cuda.current_stream().cuda_stream
    handle = run.cache.handle
    n = w.b * w.H * w.d
    q_ptrs = [inputs[g].q.data_ptr() for g in range(warmup + steps)]
    out_ptr = out.data_ptr()
    ones = np.ones(w.b, np.int32)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    bytes_per_step, dec_launches = [], 0
    plans = collections.Counter()  # the plan each step's decode used (mode, warps, tile rows, stages)
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    launches0 = run.cache.launch_count
    if clocks is not None:
        clocks.start()
    t_start.record()
    for k in range(steps):
        g = warmup + k
        inp = inputs[g]
        run.cache.append(inp.kv_k, inp.kv_v, ones, inp.kinds)
        # decode bytes of this step are fixed once the token is appended: computed from the host lengths
        bytes_per_step.append(run.decode_bytes() * w.M)
        l0 = run.cache.launch_count
        ev[k][0].record()
        rc = dec(handle, 0, w.M, q_ptrs[g], n, w.scale, out_ptr, n, stream_h)
        ev[k][1].record()
        if rc:
            raise kvc.KvcError(rc, kvc.lib().kvc_last_error().decode())
        dec_launches += run.cache.launch_count - l0
        plans[tuple(run.cache.last_decode_plan.values())] += 1
        seq, cl, cr = run.step_spans(inp.kinds)
        run.g += 1
        if seq:
            run.cache.compress_spans(seq, cl, cr)
    t_end.record()
    torch.cuda.synchronize()
    clk = clocks.stop() if clocks is not None else None
    launches = run.cache.launch_count - launches0
    elapsed = t_start.elapsed_time(t_end) / 1e3
    dec_us = [e0.elapsed_time(e1) * 1e3 for e0, e1 in ev]
    dec_total_s = sum(dec_us) / 1e6
    achieved = sum(bytes_per_step) / dec_total_s / 1e9
    peak, peak_kind = measured_hbm_peak()
    common, n_common = plans.most_common(1)[0]
    plan = dict(zip(("mode", "workers", "tile_rows", "stages"), common))
    plan["share_of_steps"] = n_common / steps
    return {"elapsed": elapsed, "tokens": w.b * steps, "launches": launches, "dec_launches": dec_launches,
            "dec_total_s": dec_total_s, "dec_us": dec_us, "bytes": sum(bytes_per_step), "achieved": achieved,
            "peak": peak, "peak_kind": peak_kind, "plan": plan, "clocks": clk}


PLAN_NAMES = ["one unbalanced layer: CTA or cluster per segment, or stream-K", "CTA or cluster per segment, or several per CTA",
              "warp per segment", "whole segments, several per warp",
              "unbalanced layers: CTA per segment, or whole segments per warp cut by rows"]


def plan_record(plan, launches_per_step: float):
    return {"mode": PLAN_NAMES[plan["mode"]] if plan["mode"] >= 0 else None, "warps": plan["workers"],
            "tile_rows": plan["tile_rows"], "stages": plan["stages"], "launches_per_step": launches_per_step,
            "share_of_steps": plan.get("share_of_steps")}


def measure_workload(name: str, dev, steps: int, warmup: int = 3):
    """Decode and compaction roofline fractions of one more workload, measured the way the headline is
    (a shorter timed window): prompt appended, freed in one compaction (timed), then timed steps."""
    import torch

    import harness
    from synth import workloads as wl

    w = wl.by_name(name)
    run = harness.Runner(w, warmup + steps, device=dev)
    run.load_prompt(compress=False)
    comp = time_prompt_compaction(run, w)
    inputs = [run.make_step_inputs(g) for g in range(warmup + steps)]
    r = timed_decode_steps(run, w, inputs, warmup, steps)
    status = run.cache.device_status()
    del inputs, run
    torch.cuda.empty_cache()
    n_launch = max(1, r["dec_launches"])
    return {"workload": name, "tokens_per_s": r["tokens"] / r["elapsed"], "steps": steps,
            "decode_attention_tokens_per_s": r["tokens"] / r["dec_total_s"],
            "decode": {"achieved": r["achieved"], "peak": r["peak"], "unit": "GB/s",
                       "frac": r["achieved"] / r["peak"], "frac_of_8tbs": r["achieved"] / 8000.0,
                       "peak_kind": r["peak_kind"], "bytes_per_launch_mean": r["bytes"] / n_launch,
                       "launch_us_mean": r["dec_total_s"] / n_launch * 1e6,
                       "plan": plan_record(r["plan"], r["dec_launches"] / steps)},
            "compaction": {k: comp[k] for k in ("bytes", "ms", "scan_ms", "move_ms", "call_ms", "achieved", "frac",
                                                "frac_of_8tbs", "move_frac")},
            "device_status": status}


def run_kvc(args, w):
    import torch
    import torch.distributed as dist

    import harness

    rank, world, local = dist_setup(args.gpus)
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    steps_total = args.warmup + args.steps
    dev = torch.device("cuda", local)

    # ---------------- device-resident run ----------------
    run = harness.Runner(w, steps_total, device=dev)
    append_ev = []
    run.load_prompt(compress=False, timer=append_ev)
    compaction = time_prompt_compaction(run, w)
    torch.cuda.synchronize()
    compaction["prompt_append_ms"] = sum(a.elapsed_time(b) for a, b in append_ev)
    prompt_free = time_prompt_write_time_freeing(w, steps_total, dev)
    if w.extra.get("policy") == "local":
        # the local-attention cache keeps a window, not the sentinel structure the prefill mask reads
        prefill = "not defined for the local-attention cache"
    else:
        prefill = [time_prompt_prefill(w, steps_total, dev, blk) for blk in (0, 512)]
    inputs = [run.make_step_inputs(g) for g in range(steps_total)]
    r = timed_decode_steps(run, w, inputs, args.warmup, args.steps, world, ClockSampler(local))
    tokens, elapsed = aggregate(r["tokens"], r["elapsed"], dev)
    value = tokens / elapsed
    n_launch = max(1, r["dec_launches"])
    status = run.cache.device_status()
    del inputs, run
    torch.cuda.empty_cache()

    # ---------------- end to end through the C ABI with host buffers ----------------
    e2e = None
    if not args.no_e2e:
        e2e = run_e2e(args, w, dev, world)

    # ---------------- the other workloads' roofline fractions (rank 0) ----------------
    per_workload = []
    if rank == 0 and args.per_workload:
        for name in [x for x in args.per_workload.split(",") if x and x != w.name]:
            per_workload.append(measure_workload(name, dev, args.per_workload_steps))

    if rank == 0:
        dec_us = sorted(r["dec_us"])
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": elapsed / args.steps * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": w.dtype,
            "data": "synthetic (seeded counter-based generator; no dataset or weights)",
            "config": workload_config(w),
            "roofline": {"bound": "hbm", "achieved": r["achieved"], "peak": r["peak"], "unit": "GB/s",
                         "frac": r["achieved"] / r["peak"], "frac_of_8tbs": r["achieved"] / 8000.0,
                         "peak_kind": r["peak_kind"],
                         "kernel": "decode_cta_kernel / decode_kernel (single-query attention over the kept rows: whole segments per CTA, cluster or warp, or split-K, with a log-sum-exp combine)",
                         "traffic": recorded_traffic(w.name, r["bytes"] / n_launch),
                         "bytes_per_launch_mean": r["bytes"] / n_launch,
                         "launch_us_mean": r["dec_total_s"] / n_launch * 1e6},
            "decode_plan": plan_record(r["plan"], r["dec_launches"] / args.steps),
            "decode_us_per_step": {"min": dec_us[0], "median": statistics.median(dec_us), "max": dec_us[-1]},
            "decode_share_of_step": r["dec_total_s"] / r["elapsed"],
            # b / (decode kernel time per step), the decode-attention rate alone; `value` is per whole step
            "decode_attention_tokens_per_s": r["tokens"] / r["dec_total_s"],
            "compaction": compaction,
            "prompt_write_time_freeing": prompt_free,
            "prefill": prefill,
            "per_workload": per_workload,
            "gpu_launches": r["launches"],
            "device_status": status,
            "clocks": r["clocks"],
            "e2e": e2e,
        }
        if not args.no_cpu_baseline:
            line["cpu_baseline"] = cpu_baseline(w, steps_total, args.cpu_seconds)
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_e2e(args, w, dev, world):
    """The same steps through the public API with inputs in host memory: each step stages its token's
    K/V and the queries into a pinned buffer, copies them host->device and reads the outputs back
    device->host.  The timed region runs `--e2e-reps` times, each on a fresh cache built from the
    same prompt, and the median is reported with every sample: on a shared host a window's copies
    can stall."""
    vals, clocks = [], []
    h2d = d2h = 0
    for _ in range(max(1, args.e2e_reps)):
        tokens, elapsed, clk, h2d, d2h = _e2e_once(args, w, dev, world)
        vals.append(tokens / elapsed)
        if clk:
            clocks.append(clk)
    merged = None
    if clocks:
        merged = {"sm_mhz": statistics.median(c["sm_mhz"] for c in clocks),
                  "sm_max_mhz": max(c["sm_max_mhz"] for c in clocks),
                  "reasons": sorted({r for c in clocks for r in c["reasons"]}),
                  "samples": sum(c["samples"] for c in clocks), "source": clocks[0]["source"]}
    return {"value": statistics.median(vals), "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
            "samples": vals, "clocks": merged}


def _e2e_once(args, w, dev, world):
    import torch
    import torch.distributed as dist

    import harness

    steps_total = args.warmup + args.steps
    run = harness.Runner(w, steps_total, device=dev)
    run.load_prompt()
    # every step's inputs in ordinary (pageable) host memory, as a caller would hold them
    host_in = []
    for g in range(steps_total):
        inp = run.make_step_inputs(g)
        host_in.append((inp.kinds, inp.kv_k.cpu(), inp.kv_v.cpu(), inp.q.cpu()))
    shape = (w.M, w.b, w.H, w.d)
    # Two pinned staging sets: each step's inputs are copied into one on the host, then uploaded from
    # it while the previous step computes; a set is refilled once its previous uploads have read it.
    # (Uploading from a distinct pinned buffer per step -- 5 GB of pinned memory for the ragged
    # workload -- made single 38 MB uploads take up to 9 ms and slowed the decodes they overlapped.)
    stage = [tuple(torch.empty(shape, dtype=run.tdt).pin_memory() for _ in range(3)) for _ in range(2)]
    # Two sets of device inputs and outputs: an upload stream copies the next step's inputs while
    # the current step runs, and a download stream reads each step's outputs back while the next one
    # runs (one stream per direction, so the two copy engines never wait on each other).  Every
    # step's copies happen inside the timed region; only their overlap with compute is new.
    dk = [torch.empty(shape, dtype=run.tdt, device=dev) for _ in range(2)]
    dv = [torch.empty_like(dk[0]) for _ in range(2)]
    dq = [torch.empty_like(dk[0]) for _ in range(2)]
    out = [torch.empty(shape, dtype=torch.float32, device=dev) for _ in range(2)]
    host_out = [torch.empty(shape, dtype=torch.float32).pin_memory() for _ in range(2)]
    h2d = 3 * dk[0].numel() * dk[0].element_size()
    d2h = host_out[0].numel() * 4
    comp = torch.cuda.current_stream(dev)
    up = torch.cuda.Stream(dev)
    down = torch.cuda.Stream(dev)
    ev_in = [torch.cuda.Event() for _ in range(2)]     # inputs of the set uploaded
    ev_done = [torch.cuda.Event() for _ in range(2)]   # the step using the set finished
    ev_out = [torch.cuda.Event() for _ in range(2)]    # its outputs read back

    def upload(g):
        i = g & 1
        kinds, hk, hv, hq = host_in[g]
        ev_in[i].synchronize()  # the staging set's previous uploads have read it
        for dst, src in zip(stage[i], (hk, hv, hq)):
            dst.copy_(src)
        with torch.cuda.stream(up):
            up.wait_event(ev_done[i])   # the step that last used this set is done with its inputs
            dk[i].copy_(stage[i][0], non_blocking=True)
            dv[i].copy_(stage[i][1], non_blocking=True)
            dq[i].copy_(stage[i][2], non_blocking=True)
            ev_in[i].record(up)

    def one(g, last):
        i = g & 1
        comp.wait_event(ev_in[i])
        comp.wait_event(ev_out[i])        # the outputs of the set's previous step have been read back
        if not last:
            upload(g + 1)
        run.step(harness.StepInputs(host_in[g][0], dk[i], dv[i], dq[i]), out[i], stream=comp)
        ev_done[i].record(comp)
        with torch.cuda.stream(down):
            down.wait_event(ev_done[i])
            host_out[i].copy_(out[i], non_blocking=True)
            ev_out[i].record(down)

    for i in range(2):
        ev_done[i].record(comp)
        ev_out[i].record(comp)
        ev_in[i].record(comp)
    upload(0)
    for g in range(args.warmup):
        one(g, g == args.warmup - 1)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = ClockSampler(dev.index)
    clocks.start()
    t0 = time.perf_counter()
    upload(args.warmup)  # every timed step's inputs are staged and uploaded inside the timed region
    for k in range(args.steps):
        one(args.warmup + k, k == args.steps - 1)
    torch.cuda.synchronize()
    elapsed = time.perf_counter() - t0
    clk = clocks.stop()
    tokens, elapsed = aggregate(w.b * args.steps, elapsed, dev)
    del run
    torch.cuda.empty_cache()
    return tokens, elapsed, clk, h2d, d2h


def main():
    args = parse()
    from synth import workloads as wl

    if args.capacity_sweep:
        run_capacity_sweep(args)
        return
    kw = {}
    if args.ragged_lengths:
        if args.workload != "ragged":
            raise SystemExit("--ragged-lengths applies to the ragged workload only")
        lmin, lmax = (int(x) for x in args.ragged_lengths.split(","))
        kw = {"lmin": lmin, "lmax": lmax}
    w = wl.by_name(args.workload, **kw)
    if args.ragged_lengths:
        w = dataclasses.replace(w, name=f"{w.name}-L{lmin}-{lmax}")
    if args.layers:
        w = dataclasses.replace(w, M=args.layers, name=f"{w.name}-M{args.layers}")
    if args.prefill_only:
        import torch

        torch.cuda.set_device(0)
        dev = torch.device("cuda", 0)
        blocks = (0, 512) if args.prefill_block < 0 else (args.prefill_block,)
        for blk in blocks:
            r = time_prompt_prefill(w, 1, dev, blk)
            r["workload"] = w.name
            print(json.dumps(r), flush=True)
        return
    if args.impl == "reference":
        run_reference(args, w)
    else:
        run_kvc(args, w)


if __name__ == "__main__":
    main()
