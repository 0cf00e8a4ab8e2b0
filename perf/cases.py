"""The work that a user of the sentinel-compressed KV cache has it do, as cases that can be timed and compared.

Five kinds of pass, each through the package's public calls:

  decode    one decode step's attention over a cache that holds its prompt: layer by layer, as a model calls it between
            its projections, or all layers in one call, as in the throughput setting
  prefill   the masked attention of a prompt's queries, whole prompts or the last block of longer ones
  ingest    a new cache is made for a batch, its prompts are appended and their spans freed (by compaction, or as written)
  blocks    a new cache takes its prompts block by block: append and prefill of every layer, then the closed spans' freeing
  generate  a new cache, short prompts, and a run of decode steps that opens, closes and frees spans

Sizes are those of the repository's workloads (OPT-1.3B-, OPT-2.7B- and 3B-rotary-shaped caches, the ragged batch, the
tiny one, the Local Attention ring), and generic ones.  K, V and q are standard normal in the cache type, made from the
seed on the GPU.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2310_08152_gb300 as kvc

DEVICE = "cuda:0"
NORMAL, CL, CR = kvc.NORMAL, kvc.CL, kvc.CR
_POLICY = {"paper": kvc.POLICY_PAPER, "keep_cl": kvc.POLICY_KEEP_CL, "local": kvc.POLICY_LOCAL}
_TORCH = {"f16": torch.float16, "bf16": torch.bfloat16}

# Fields that a case may leave out.
_DEFAULTS = {"dtype": "f16", "rot": 0, "spans": "periodic", "interior": 32, "policy": "paper", "ratio": 0.0, "open": False,
             "fused": False, "block": 0, "steps": 0, "free": False, "shape_seed": 0}


def listed():
    return [
        # The smallest call: one layer of two short sequences; latency and launch cost are all there is.
        {"name": "decode_tiny", "kind": "decode", "M": 1, "H": 4, "d": 64, "b": 2, "lmin": 512, "lmax": 512},
        # A serving step of an OPT-1.3B-shaped model: a call per layer, as its projections leave no other way.
        {"name": "decode_opt1.3b_by_layer", "kind": "decode", "M": 24, "H": 32, "d": 64, "b": 16, "lmin": 2048, "lmax": 2048},
        # The throughput setting with rotary positions: every layer's queries ready, one call; large and balanced.
        {"name": "decode_rope3b_fused", "kind": "decode", "M": 32, "H": 32, "d": 80, "rot": 80, "b": 64, "lmin": 2048, "lmax": 2048,
         "fused": True},
        # Serving of requests of very different lengths, layer by layer: unbalanced segments.
        {"name": "decode_ragged_by_layer", "kind": "decode", "M": 12, "H": 32, "d": 64, "b": 48, "lmin": 256, "lmax": 8192,
         "spans": "sampled", "shape_seed": 5},
        # The paper's throughput setting at a high ratio: many short segments (about a hundred rows), bf16.
        {"name": "decode_short_bf16", "kind": "decode", "M": 4, "H": 32, "d": 80, "dtype": "bf16", "b": 96, "lmin": 700, "lmax": 800,
         "interior": 57, "fused": True, "shape_seed": 2},
        # The Local Attention baseline's ring, odd length, a wide head.
        {"name": "decode_local_d128", "kind": "decode", "M": 8, "H": 16, "d": 128, "b": 7, "lmin": 3001, "lmax": 3001, "spans": "none",
         "policy": "local", "ratio": 0.5},
        # Masked prefill of whole prompts, the OPT-1.3B shape: hidden interiors still stored.
        {"name": "prefill_opt1.3b", "kind": "prefill", "M": 1, "H": 32, "d": 64, "b": 16, "lmin": 2048, "lmax": 2048},
        # The same with rotary positions, d_head 80, prompts of all lengths and sampled spans.
        {"name": "prefill_rope_ragged", "kind": "prefill", "M": 1, "H": 32, "d": 80, "rot": 80, "b": 24, "lmin": 256, "lmax": 4096,
         "spans": "sampled", "shape_seed": 3},
        # The last block of long prompts whose earlier blocks are compacted already (the for-loop over blocks), bf16.
        {"name": "prefill_block_opt2.7b", "kind": "prefill", "M": 1, "H": 32, "d": 80, "dtype": "bf16", "b": 32, "lmin": 4096, "lmax": 4096,
         "interior": 44, "block": 512},
        # A new batch, prompts appended and their spans freed in one go.
        {"name": "ingest_opt1.3b", "kind": "ingest", "M": 24, "H": 32, "d": 64, "b": 16, "lmin": 2048, "lmax": 2048},
        # A whole prompt ingestion in blocks, a few layers: append, prefill and freeing together, with their host work.
        {"name": "blocks_rope", "kind": "blocks", "M": 2, "H": 32, "d": 128, "dtype": "bf16", "rot": 128, "b": 6, "lmin": 900, "lmax": 1500,
         "block": 384, "shape_seed": 4},
        # Interactive generation, small batch: append, decode and freeing of single tokens.
        {"name": "generate_small", "kind": "generate", "M": 4, "H": 16, "d": 64, "b": 4, "lmin": 150, "lmax": 300, "steps": 40,
         "shape_seed": 6},
    ]


def draw(rng):
    while True:
        c = _draw_once(rng)
        if _fits(c):
            return c


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_once(rng):
    kind = rng.choices(["decode", "prefill", "ingest", "blocks", "generate"], [5, 4, 2, 1, 1])[0]
    d = rng.choice([64, 64, 80, 80, 96, 128])
    c = {"kind": kind, "d": d, "dtype": rng.choice(["f16", "f16", "bf16"]), "H": rng.choice([4, 8, 12, 16, 20, 32, 32, 40]),
         "rot": rng.choice([0, 0, d, d, 32]), "spans": rng.choice(["periodic", "periodic", "sampled", "sampled", "none"]),
         "interior": rng.randint(8, 57), "policy": rng.choice(["paper", "paper", "paper", "keep_cl"]), "shape_seed": rng.randrange(1 << 20)}
    if kind == "decode":
        c.update(M=_log_int(rng, 1, 32), b=_log_int(rng, 1, 96), lmax=_log_int(rng, 130, 8192), fused=rng.random() < 0.5,
                 open=rng.random() < 0.3)
        if rng.random() < 0.15:
            c.update(policy="local", spans="none", ratio=rng.choice([0.25, 0.5, 0.8]), open=False)
    elif kind == "prefill":
        c.update(M=rng.randint(1, 3), b=_log_int(rng, 1, 32), lmax=_log_int(rng, 130, 4096))
        if rng.random() < 0.4:
            c["block"] = rng.choice([64, 128, 200, 256, 512, 512])
    elif kind == "ingest":
        c.update(M=_log_int(rng, 1, 24), b=_log_int(rng, 1, 16), lmax=_log_int(rng, 130, 4096), free=rng.random() < 0.5)
    elif kind == "blocks":
        c.update(M=rng.randint(1, 4), b=_log_int(rng, 1, 12), lmax=_log_int(rng, 260, 2500), block=rng.choice([128, 200, 384, 512]))
    else:
        c.update(M=rng.randint(1, 6), b=_log_int(rng, 1, 12), lmax=_log_int(rng, 130, 700), steps=rng.randint(8, 48))
    c["lmin"] = c["lmax"] if rng.random() < 0.4 else max(65, int(c["lmax"] * rng.uniform(0.05, 0.9)))
    return c


def _fits(c):
    """No dearer than the largest listed case of the kind (host time counts for those that make a cache)."""
    w = work(c)
    most = {"decode": (2.2e10, 1e30), "prefill": (3e9, 5e11), "ingest": (1.6e10, 1e30), "blocks": (2e9, 2e11), "generate": (4e9, 1e30)}[c["kind"]]
    return 1e5 < w["bytes"] <= most[0] and w["flops"] <= most[1]


# ------------------------------------------------------------------------------------------
# What a case looks like: token kinds, spans and visibility (plain numpy, no package code)
# ------------------------------------------------------------------------------------------

class _Shape:
    def __init__(self, case):
        c = dict(_DEFAULTS, **case)
        for k, v in c.items():
            setattr(self, k, v)
        rng = random.Random(self.shape_seed)
        self.lens = [self.lmax if self.lmin == self.lmax else rng.randint(self.lmin, self.lmax) for _ in range(self.b)]
        if self.lmin != self.lmax:
            self.lens[0] = self.lmax
        self.kinds, self.closed = [], []
        for L in self.lens:
            k, sp = self._prompt(L, rng)
            self.kinds.append(k)
            self.closed.append(sp)
        self.N = sum(self.lens)
        self.torch_dtype = _TORCH[self.dtype]
        self.scale = 1.0 / math.sqrt(self.d)

    def _prompt(self, L, rng):
        k = np.zeros(L, np.uint8)
        spans = []
        if self.spans == "periodic":  # one span per 64 tokens
            off = 7 if self.interior <= 54 else 0
            at = [(64 * i + off, 64 * i + off + 1 + self.interior) for i in range(L // 64 + 1)]
        elif self.spans == "sampled":  # interiors U[8, 64], about half of the tokens enclosed
            at, t = [], rng.randint(0, 40)
            while t < L:
                n = rng.randint(8, 64)
                at.append((t, t + 1 + n))
                t += n + 2 + rng.randint(4, 60)
        else:
            at = []
        for cl, cr in at:
            if cr < L - 5:
                k[cl], k[cr] = CL, CR
                spans.append((cl, cr))
        if self.open:
            k[L - 4] = CL
        return k, spans

    def positions(self, k):
        """A normal token counts the normal tokens before it; a sentinel shares the position of the token before it."""
        return np.maximum(np.cumsum(k == NORMAL) - 1, 0).astype(np.int64)

    def hidden(self, k, spans):
        """Rows that the freeing of `spans` drops."""
        h = np.zeros(k.size, bool)
        for cl, cr in spans:
            h[cl if self.policy != "keep_cl" else cl + 1:cr] = True
        return h

    def window(self, T):
        return T - int(math.floor(T * float(np.float32(self.ratio))))

    def attended(self, s):
        """History indices that the query at the last prompt token attends to, closed spans freed."""
        k = self.kinds[s]
        if self.policy == "local":
            return np.arange(k.size - self.window(k.size), k.size)
        h = self.hidden(k, self.closed[s])
        if self.policy == "paper":
            h |= k == CL
        return np.flatnonzero(~h)

    def stored(self, s):
        """History indices that are stored once the closed spans are freed."""
        k = self.kinds[s]
        return self.attended(s) if self.policy == "local" else np.flatnonzero(~self.hidden(k, self.closed[s]))

    def n_queries(self, s):
        return min(self.block, self.lens[s]) if self.block else self.lens[s]

    def visible_counts(self, s):
        """Keys that each of the prompt's queries sees."""
        k, spans = self.kinds[s], self.closed[s]
        h = self.hidden(k, spans)
        if self.policy == "paper":
            h |= k == CL
        seen = np.cumsum(~h)
        for cl, cr in spans:
            seen[cl:cr] = seen[cl] + np.arange(cr - cl)
            seen[cr] = seen[cl] + cr - cl
        seen[k == CL] = 1
        return seen

    def visibility(self, s, n_q):
        """[n_q, T] of the last n_q prompt queries, as a GPU tensor."""
        k, T = self.kinds[s], self.lens[s]
        q = torch.arange(T - n_q, T, device=DEVICE)[:, None]
        j = torch.arange(T, device=DEVICE)[None, :]
        until = np.full(T, T)  # a row is visible to queries up to this one
        for cl, cr in self.closed[s]:
            until[cl + 1:cr] = cr
        kt = torch.from_numpy(k.astype(np.int64)).to(DEVICE)
        if self.policy == "paper":
            until[k == CL] = -1
        vis = (j <= q) & (q <= torch.from_numpy(until).to(DEVICE)[None, :])
        cl_q = (kt[T - n_q:] == CL)[:, None]
        return torch.where(cl_q, j == q, vis | (j == q))


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _normal(seed, what, layer, shape, dtype):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((int(seed) * 1000003 + what * 4099 + layer * 7 + 1) % (1 << 62))
    return torch.randn(shape, generator=g, device=DEVICE, dtype=dtype)


def _kv(sh, seed, layer):
    """K and V of every prompt token of a layer, sequence after sequence: [N][H][d]."""
    return [_normal(seed, what, layer, (sh.N, sh.H, sh.d), sh.torch_dtype) for what in (1, 2)]


def _cache(sh, capacity):
    return kvc.KVCache(sh.M, sh.H, sh.d, capacity, sh.dtype, sh.rot, 10000.0, _POLICY[sh.policy], device=DEVICE, local_ratio=sh.ratio)


def _span_lists(sh):
    t = [(s, cl, cr) for s in range(sh.b) for cl, cr in sh.closed[s]]
    return [np.array([x[i] for x in t], np.int64) for i in range(3)]


class _State:
    pass


def prepare(case, seed):
    sh = _Shape(case)
    st = _State()
    st.sh = sh
    st.n_new = np.array(sh.lens, np.int32)
    st.kinds = np.concatenate(sh.kinds)
    if sh.kind in ("decode", "prefill"):
        _prepare_attention(st, seed)
    elif sh.kind == "ingest":
        k, v = (torch.empty(sh.M, sh.N, sh.H, sh.d, dtype=sh.torch_dtype, device=DEVICE) for _ in range(2))
        for m in range(sh.M):
            k[m], v[m] = _kv(sh, seed, m)
        st.k, st.v = k, v
        st.spans = _span_lists(sh)
        st.kept = [sh.stored(s).size for s in range(sh.b)]
        st.cache = None
    elif sh.kind == "blocks":
        st.parts = []
        kv = [_kv(sh, seed, m) for m in range(sh.M)]
        q = [_normal(seed, 3, m, (sh.N, sh.H, sh.d), sh.torch_dtype) for m in range(sh.M)]
        for n, at in _block_parts(sh):
            ix = torch.from_numpy(at).to(DEVICE)
            st.parts.append((n, st.kinds[at], [(a[ix], b[ix], c[ix]) for (a, b), c in zip(kv, q)],
                             torch.empty(sh.M, at.size, sh.H, sh.d, device=DEVICE)))
        st.cache = None
    else:
        k, v = (torch.empty(sh.M, sh.N, sh.H, sh.d, dtype=sh.torch_dtype, device=DEVICE) for _ in range(2))
        for m in range(sh.M):
            k[m], v[m] = _kv(sh, seed, m)
        st.k, st.v = k, v
        st.tokens = _normal(seed, 4, 0, (sh.steps, 3, sh.M, sh.b, sh.H, sh.d), sh.torch_dtype)
        st.out = torch.empty(sh.steps, sh.M, sh.b, sh.H, sh.d, device=DEVICE)
        st.ones = np.ones(sh.b, np.int32)
        st.step_kinds = [np.full(sh.b, _step_kind(g), np.uint8) for g in range(sh.steps)]
        st.cache = None
    return st


def _prepare_attention(st, seed):
    sh = st.sh
    if sh.kind == "prefill" and sh.block:
        cap = [sh.stored(s).size + sh.n_queries(s) + 140 for s in range(sh.b)]
    elif sh.kind == "prefill":
        cap = sh.lens
    else:
        cap = [sh.stored(s).size + 64 for s in range(sh.b)]
    c = st.cache = _cache(sh, cap)
    head = np.array([L - sh.n_queries(s) for s, L in enumerate(sh.lens)], np.int32) if sh.kind == "prefill" else st.n_new
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])

    def rows(lo, hi):
        return np.concatenate([np.arange(off[s] + lo[s], off[s] + hi[s]) for s in range(sh.b)])

    zero = np.zeros(sh.b, np.int32)
    parts = [p for p in ((head, rows(zero, head), True), (st.n_new - head, rows(head, st.n_new), False)) if p[1].size]
    kv = None
    for n, at, free in parts:
        whole = at.size == sh.N
        ix = None if whole else torch.from_numpy(at).to(DEVICE)
        for m in range(sh.M):
            kv = _kv(sh, seed, m)
            k, v = kv if whole else (kv[0][ix], kv[1][ix])
            c.append(k, v, n, st.kinds[at], layer=m, free_closed=free and sh.policy != "local")
    if sh.kind == "decode":
        st.q = _normal(seed, 3, 0, (sh.M, sh.b, sh.H, sh.d), sh.torch_dtype)
        st.out = torch.empty(sh.M, sh.b, sh.H, sh.d, device=DEVICE)
    else:
        st.n_q = (st.n_new - head).astype(np.int32)
        n = int(st.n_q.sum())
        st.q = [_normal(seed, 3, m, (n, sh.H, sh.d), sh.torch_dtype) for m in range(sh.M)]
        st.out = [torch.empty(n, sh.H, sh.d, device=DEVICE) for _ in range(sh.M)]


def _block_parts(sh):
    """(tokens per sequence, their indices among all prompt tokens) of each block."""
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])
    lens = np.array(sh.lens)
    for t in range(0, max(sh.lens), sh.block):
        n = np.clip(lens - t, 0, sh.block).astype(np.int32)
        yield n, np.concatenate([np.arange(off[s] + t, off[s] + t + n[s]) for s in range(sh.b) if n[s] > 0])


def _step_kind(g):
    """A generated span every 24 tokens: opened at the 4th, closed at the 20th."""
    return CL if g % 24 == 3 else CR if g % 24 == 19 else NORMAL


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------

def run(st):
    return {"decode": _run_decode, "prefill": _run_prefill, "ingest": _run_ingest, "blocks": _run_blocks,
            "generate": _run_generate}[st.sh.kind](st)


def _run_decode(st):
    sh, c = st.sh, st.cache
    if sh.fused:
        return c.decode_attention_layers(st.q, sh.scale, out=st.out)
    stream = kvc.stream_handle()
    for m in range(sh.M):
        c.decode_attention(m, st.q[m], sh.scale, out=st.out[m], stream=stream)
    return st.out


def _run_prefill(st):
    sh, c = st.sh, st.cache
    for m in range(sh.M):
        c.prefill_attention(m, st.q[m], st.n_q, sh.scale, out=st.out[m])
    return st.out


def _run_ingest(st):
    sh = st.sh
    st.cache = None  # the last batch is done
    c = st.cache = _cache(sh, st.kept if sh.free else sh.lens)
    c.append(st.k, st.v, st.n_new, st.kinds, free_closed=sh.free)
    if sh.free or not st.spans[0].size:
        return {"k": c.k, "v": c.v, "pos": c.pos[:c.C], "orig": c.orig[:c.C]}
    c.compress_spans(*st.spans)
    out = {}
    for s in range(sh.b):  # the kept rows of each sequence (views)
        lo, n = int(c.offsets[s]), st.kept[s]
        for name, buf in (("k", c.k), ("v", c.v)):
            rows = buf.view(sh.M, sh.H * c.C, sh.d)[:, sh.H * lo:sh.H * (lo + sh.lens[s])]
            out["%s%d" % (name, s)] = rows.unflatten(1, (sh.H, sh.lens[s]))[:, :, :n]
        out["pos%d" % s], out["orig%d" % s] = c.pos[lo:lo + n], c.orig[lo:lo + n]
    return out


def _run_blocks(st):
    sh = st.sh
    st.cache = None
    c = st.cache = _cache(sh, sh.lens)
    for n, kinds, layers, out in st.parts:
        for m, (k, v, q) in enumerate(layers):
            c.append(k, v, n, kinds, layer=m)
            c.prefill_attention(m, q, n, sh.scale, out=out[m])
        spans = [(s, cl, cr) for s in range(sh.b) for cl, cr in c.pending_spans(s)]
        if spans:
            c.compress_spans(*zip(*spans))
    return [p[3] for p in st.parts]


def _run_generate(st):
    sh = st.sh
    st.cache = None
    c = st.cache = _cache(sh, [L + sh.steps for L in sh.lens])
    c.append(st.k, st.v, st.n_new, st.kinds, free_closed=True)
    stream = kvc.stream_handle()
    opened = 0
    for g in range(sh.steps):
        k, v, q = st.tokens[g]
        c.append(k, v, st.ones, st.step_kinds[g], stream=stream)
        for m in range(sh.M):
            c.decode_attention(m, q[m], sh.scale, out=st.out[g, m], stream=stream)
        kind = _step_kind(g)
        if kind == CL:
            opened = g
        elif kind == CR:
            c.compress_spans(np.arange(sh.b), st.n_new + opened, st.n_new + g, stream=stream)
    return st.out


# ------------------------------------------------------------------------------------------
# What a pass cannot do without, and how far results may be off
# ------------------------------------------------------------------------------------------

def work(case):
    sh = _Shape(case)
    row = sh.H * sh.d  # elements of one token's K (or V) in one layer
    stored = [sh.stored(s).size for s in range(sh.b)]
    if sh.kind == "decode":
        seen = sum(sh.attended(s).size for s in range(sh.b))
        return {"bytes": sh.M * row * (4 * seen + 6 * sh.b), "flops": 4 * sh.M * row * seen}
    if sh.kind == "ingest":
        if sh.free:
            return {"bytes": 8 * sh.M * row * sum(stored), "flops": 0}
        moved = sum(n - sh.closed[s][0][0] for s, n in enumerate(stored) if sh.closed[s])
        return {"bytes": 8 * sh.M * row * (sh.N + max(0, moved)), "flops": 0}
    if sh.kind == "generate":
        seen = sh.steps * sum(stored) + sh.b * sh.steps * sh.steps // 4
        return {"bytes": sh.M * row * (8 * sum(stored) + 4 * seen + 14 * sh.b * sh.steps), "flops": 4 * sh.M * row * seen}
    pairs, rows, nq = 0, 0, 0
    for s in range(sh.b):
        n = sh.n_queries(s) if sh.kind == "prefill" else sh.lens[s]
        pairs += int(sh.visible_counts(s)[sh.lens[s] - n:].sum())
        nq += n
        rows += min(stored[s], sh.lens[s] - n) + n
    move = 8 * nq + 4 * rows * 2 if sh.kind == "blocks" else 0
    return {"bytes": sh.M * row * (4 * rows + 6 * nq + move), "flops": 4 * sh.M * row * pairs}


def tolerance(case):
    """About four times the largest error against exact() that was measured for each group."""
    c = dict(_DEFAULTS, **case)
    rotary, half = c["rot"] > 0, c["dtype"] == "f16"
    if c["kind"] == "ingest":
        # rows are copied; of rotated ones a few values may round the other way (by one unit in the last place)
        return {"rel": 1e-4 if half else 8e-4, "max": 2e-3 if half else 1.6e-2} if rotary else {"rel": 0.0, "max": 0.0}
    if c["kind"] in ("decode", "generate"):
        # 32-bit sums over 16-bit rows (measured 3e-7); rotated keys are stored rounded, where single values may round
        # the other way (measured 1e-5 f16)
        return {"rel": (4e-5 if half else 3e-4), "max": 4e-3} if rotary else {"rel": 2e-6, "max": 5e-5}
    if half:  # weights in one f16 part (measured 1.1e-4, with rotary positions 1.7e-4)
        return {"rel": 7e-4, "max": 2e-2}
    # bf16: weights in two parts (measured 1.3e-6; with rotary positions, 2.8e-5)
    return {"rel": 1.2e-4 if rotary else 6e-6, "max": 5e-3 if rotary else 2e-4}


# ------------------------------------------------------------------------------------------
# The same in 64 bits, by torch alone
# ------------------------------------------------------------------------------------------

def _rotate(x, pos, rot):
    """Rotate-half rotary embedding of x [n][H][d] (64 bits) at pos [n]."""
    if not rot:
        return x
    inv = 10000.0 ** (-2.0 * torch.arange(rot // 2, device=DEVICE, dtype=torch.float64) / rot)
    a = torch.as_tensor(pos, device=DEVICE, dtype=torch.float64)[:, None] * inv
    c, s = a.cos()[:, None, :], a.sin()[:, None, :]
    u, w = x[..., :rot // 2], x[..., rot // 2:rot]
    return torch.cat([u * c - w * s, w * c + u * s, x[..., rot:]], -1)


def _keys(sh, k, pos):
    """Stored keys: rotated at their positions and rounded to the cache type."""
    k = k.double()
    return _rotate(k, pos, sh.rot).to(sh.torch_dtype).double() if sh.rot else k


def _attend(sh, q, k, v, mask=None):
    """softmax(scale q k^T) v: q [n][H][d], k and v [m][H][d], mask [n][m]."""
    out = torch.empty_like(q)
    for h in range(0, sh.H, 4):
        z = torch.matmul(q[:, h:h + 4].transpose(0, 1), k[:, h:h + 4].permute(1, 2, 0)) * sh.scale
        if mask is not None:
            z = z.masked_fill(~mask, -math.inf)
        out[:, h:h + 4] = torch.matmul(torch.softmax(z, -1), v[:, h:h + 4].transpose(0, 1)).transpose(0, 1)
    return out


def _attend_one(sh, q, k, v):
    """The same for one query [H][d]."""
    p = torch.softmax(torch.einsum("hd,mhd->hm", q, k) * sh.scale, -1)
    return torch.einsum("hm,mhd->hd", p, v)


def exact(case, seed):
    sh = _Shape(case)
    return {"decode": _exact_decode, "prefill": _exact_prefill, "ingest": _exact_ingest, "blocks": _exact_blocks,
            "generate": _exact_generate}[sh.kind](sh, seed)


def _exact_decode(sh, seed):
    q = _normal(seed, 3, 0, (sh.M, sh.b, sh.H, sh.d), sh.torch_dtype).double()
    out = torch.empty_like(q)
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])
    rows = [sh.attended(s) for s in range(sh.b)]
    pos = [sh.positions(k) for k in sh.kinds]
    at = [torch.from_numpy(off[s] + rows[s]).to(DEVICE) for s in range(sh.b)]
    for m in range(sh.M):
        k, v = _kv(sh, seed, m)
        for s in range(sh.b):
            qs = _rotate(q[m, s][None], pos[s][-1:], sh.rot)[0]
            out[m, s] = _attend_one(sh, qs, _keys(sh, k[at[s]], pos[s][rows[s]]), v[at[s]].double())
    return out


def _exact_prefill(sh, seed):
    out = []
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])
    nq = [sh.n_queries(s) for s in range(sh.b)]
    for m in range(sh.M):
        k, v = _kv(sh, seed, m)
        q = _normal(seed, 3, m, (sum(nq), sh.H, sh.d), sh.torch_dtype).double()
        t = 0
        for s in range(sh.b):
            lo, hi = off[s], off[s] + sh.lens[s]
            pos = sh.positions(sh.kinds[s])
            qs = _rotate(q[t:t + nq[s]], pos[-nq[s]:], sh.rot)
            q[t:t + nq[s]] = _attend(sh, qs, _keys(sh, k[lo:hi], pos), v[lo:hi].double(), sh.visibility(s, nq[s]))
            t += nq[s]
        out.append(q)
    return out


def _exact_ingest(sh, seed):
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])
    kept = [sh.stored(s) for s in range(sh.b)]
    pos = [sh.positions(k) for k in sh.kinds]
    per = [[[], []] for _ in range(sh.b)]
    for m in range(sh.M):
        k, v = _kv(sh, seed, m)
        for s in range(sh.b):
            at = torch.from_numpy(off[s] + kept[s]).to(DEVICE)
            per[s][0].append(_rotate(k[at].double(), pos[s][kept[s]], sh.rot).transpose(0, 1) if sh.rot else k[at].transpose(0, 1))
            per[s][1].append(v[at].transpose(0, 1))
    if sh.free or not any(sh.closed):
        flat = [torch.cat([torch.cat([per[s][i][m].reshape(-1) for s in range(sh.b)]) for m in range(sh.M)]) for i in range(2)]
        return {"k": flat[0], "v": flat[1], "pos": None, "orig": None}
    out = {}
    for s in range(sh.b):
        out["k%d" % s], out["v%d" % s], out["pos%d" % s], out["orig%d" % s] = torch.stack(per[s][0]), torch.stack(per[s][1]), None, None
    return out


def _exact_blocks(sh, seed):
    whole = _Shape({"kind": "prefill", **{k: getattr(sh, k) for k in ("M", "H", "d", "dtype", "rot", "b", "lmin", "lmax", "spans", "interior",
                                                                      "policy", "shape_seed")}})
    out = torch.stack(_exact_prefill(whole, seed))
    return [out[:, torch.from_numpy(at).to(DEVICE)] for _, at in _block_parts(sh)]


def _exact_generate(sh, seed):
    tokens = _normal(seed, 4, 0, (sh.steps, 3, sh.M, sh.b, sh.H, sh.d), sh.torch_dtype).double()
    out = torch.empty(sh.steps, sh.M, sh.b, sh.H, sh.d, device=DEVICE, dtype=torch.float64)
    off = np.concatenate([[0], np.cumsum(sh.lens)[:-1]])
    gen = np.array([_step_kind(g) for g in range(sh.steps)], np.uint8)
    prompt = [_kv(sh, seed, m) for m in range(sh.M)]
    for s in range(sh.b):
        L = sh.lens[s]
        kinds = np.concatenate([sh.kinds[s], gen])
        pos = sh.positions(kinds)
        lo, hi = off[s], off[s] + L
        full = []
        for m in range(sh.M):
            k = torch.cat([prompt[m][0][lo:hi].double(), tokens[:, 0, m, s]])
            full.append((_keys(sh, k, pos), torch.cat([prompt[m][1][lo:hi].double(), tokens[:, 1, m, s]])))
        for g in range(sh.steps):
            T = L + g + 1
            cls = L + np.flatnonzero(gen[:g + 1] == CL)
            crs = L + np.flatnonzero(gen[:g + 1] == CR)
            spans = sh.closed[s] + [(a, c) for a, c in zip(cls, crs) if c < T - 1]
            h = sh.hidden(kinds[:T], spans)
            if sh.policy == "paper":
                h |= kinds[:T] == CL
            rows = np.array([T - 1]) if gen[g] == CL else np.flatnonzero(~h)
            at = torch.from_numpy(rows).to(DEVICE)
            for m in range(sh.M):
                qs = _rotate(tokens[g, 2, m, s][None], pos[T - 1:T], sh.rot)[0]
                out[g, m, s] = _attend_one(sh, qs, full[m][0][at], full[m][1][at])
    return out
