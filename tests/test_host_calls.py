"""The host side of a call: spans listed past the binding's first buffer, appends at tied positions in one
call, and uploads staged in the caller's pinned memory."""
import numpy as np
import pytest
import torch

import paper_2310_08152_gb300 as kvc


@pytest.mark.parametrize("n", [0, 1, 64, 65, 200])
def test_pending_spans_of_any_number(n):
    book = kvc.Book(2, [4 * n + 8] * 2)
    kinds = np.array([0] + [kvc.CL, 0, kvc.CR] * n, np.uint8)
    book.append([0, kinds.size], kinds)
    assert book.pending_spans(1) == [(1 + 3 * i, 3 + 3 * i) for i in range(n)]
    assert book.pending_spans(0) == []


@pytest.mark.parametrize("shape", [(2,), (1, 2), (2, 1)])
def test_token_counts_of_any_shape(monkeypatch, shape):
    """Token counts per sequence come as an array of any shape: only their order counts."""
    c = object.__new__(kvc.KVCache)
    c.__dict__.update(M=3, H=4, d=64, b=2, torch_dtype=torch.float16, handle=None)
    seen = []
    monkeypatch.setattr(kvc, "_dev", lambda t, name, dtype, n: seen.append(n))
    monkeypatch.setattr(kvc, "kvc_append_tied", lambda handle, layer, k, v, n_new, *a: seen.append(n_new.ravel().tolist()))
    monkeypatch.setattr(kvc, "kvc_prefill_attention", lambda handle, layer, q, n_q, *a: seen.append(np.ravel(n_q).tolist()))
    n = np.array([3, 4]).reshape(shape)
    assert c.append(None, None, n, [0] * 7).size == 7
    c.prefill_attention(0, None, n, 0.125, out=torch.empty(0))
    assert seen == [3 * 7 * 256, 3 * 7 * 256, [3, 4], 7 * 256, 7 * 256, [3, 4]]


def _tokens(M, H, d, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(M, n, H, d, device="cuda", generator=g).half() for _ in range(2)]


@pytest.mark.gpu
@pytest.mark.parametrize("free_closed", [False, True])
def test_append_at_tied_positions_and_own_staging(free_closed):
    """KVCache.append without positions (one call, staging from torch's pinned pool) stores what next_positions
    and an append with them store in a cache whose ring the library allocates."""
    M, H, d = 2, 4, 64
    n_new = np.array([7, 0, 5], np.int32)
    kinds = np.array([0, kvc.CL, 0, 0, kvc.CR, 0, kvc.CL, 0, 0, kvc.CL, 0, kvc.CR], np.uint8)
    a, b = (kvc.KVCache(M, H, d, [16] * 3) for _ in range(2))
    kvc._check(kvc.lib().kvc_set_staging(b.handle, None, 0))
    for x in (a.k, a.v, a.pos, a.orig, b.k, b.v, b.pos, b.orig):
        x.zero_()
    k, v = _tokens(M, H, d, 12, 1)
    pos = a.append(k, v, n_new, kinds, free_closed=free_closed)
    assert np.array_equal(pos, b.book.next_positions(n_new, kinds))
    b.append(k, v, n_new, kinds, pos=pos, free_closed=free_closed)
    torch.cuda.synchronize()
    for x, y in ((a.k, b.k), (a.v, b.v), (a.pos, b.pos), (a.orig, b.orig)):
        assert torch.equal(x, y)
    # what was refused stays refused, with the kinds' errors before the tensors'
    with pytest.raises(kvc.KvcError) as e:
        a.append(k[:, :1], v, [0, 0, 1], [kvc.CR])
    assert e.value.status == 4
    with pytest.raises(ValueError):
        a.append(k, v, [1, 0, 0], [0])
    with pytest.raises(kvc.KvcError) as e:
        kvc.kvc_append_tied(a.handle, 1, k, v, n_new, kinds, np.empty(12, np.int32), False)
    assert e.value.status == 1
    # staging memory: before the first append only, large enough, aligned
    with pytest.raises(kvc.KvcError) as e:
        kvc.kvc_set_staging(a.handle, a.staging)
    assert e.value.status == 5
    c = kvc.KVCache(M, H, d, [16] * 3)
    for bad in (c.staging[:-1], torch.empty(c.staging.numel() + 16, dtype=torch.uint8)[1:]):
        with pytest.raises(kvc.KvcError) as e:
            kvc.kvc_set_staging(c.handle, bad)
        assert e.value.status == 1
    assert a.device_status() == 0 and b.device_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("own", [False, True])
def test_cache_that_ends_while_a_stream_captures(mode, own):
    """A cache's end waits for its upload on a busy stream, before torch's pool gets the staging memory back, and
    leaves the capture on another stream alone; so does a cache whose ring the library allocates."""
    c = kvc.KVCache(2, 4, 64, [600] * 2)
    if own:
        kvc._check(kvc.lib().kvc_set_staging(c.handle, None, 0))
    n = np.array([250, 250], np.int32)
    k, v = _tokens(2, 4, 64, 500, 2)
    kinds = np.zeros(500, np.uint8)
    c.append(k, v, n, kinds)
    x, side, uploaded = torch.ones(4, device="cuda"), torch.cuda.Stream(), torch.cuda.Event()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode=mode):
        x += 1
        with torch.cuda.stream(side):
            torch.cuda._sleep(400_000_000)  # 0.2 s
            c.append(k, v, n, kinds)
            uploaded.record()
        c.close()
        x += 1
    assert uploaded.query()
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [3.0] * 4


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("beside", [False, True])
def test_cache_that_is_made_while_a_stream_captures(mode, beside):
    """Made on the capturing stream or beside it (where torch has device memory at hand), a cache leaves the capture
    alone and works after it."""
    x, capturing, side = torch.ones(4, device="cuda"), torch.cuda.Stream(), torch.cuda.Stream()
    k, v = _tokens(1, 4, 64, 300, 3)
    kinds = np.zeros(300, np.uint8)
    with torch.cuda.stream(side):
        held = [kvc.KVCache(1, 4, 64, [cap]) for cap in (300, 30000)]
        again = [torch.empty_like(t) for c in held for t in (c.k, c.v, c.pos, c.orig, c.workspace)]
    torch.cuda.synchronize()
    del again
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(capturing):
        graph.capture_begin(capture_error_mode=mode)
        x += 1
        with torch.cuda.stream(side if beside else capturing):
            made = [kvc.KVCache(1, 4, 64, [cap]) for cap in (300, 30000)]
        x += 1
        graph.capture_end()
    graph.replay()
    for c in made:
        c.append(k, v, [300], kinds)
        out = c.decode_attention(0, k[0, -1:], 0.125)
        p = torch.softmax(torch.einsum("hd,nhd->hn", k[0, -1].double(), k[0].double()) * 0.125, -1)
        assert (out[0].double() - torch.einsum("hn,nhd->hd", p, v[0].double())).abs().max().item() < 3e-4
        assert c.device_status() == 0
    assert x.tolist() == [3.0] * 4


@pytest.mark.gpu
def test_cache_that_ends_after_its_append_was_captured():
    """The event of a captured upload cannot be waited for; no error of that is left for the calls that follow."""
    c = kvc.KVCache(1, 4, 64, [900])
    k, v = _tokens(1, 4, 64, 300, 5)
    kinds = np.zeros(300, np.uint8)
    c.append(k, v, [300], kinds)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.append(k, v, [300], kinds)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(c.stream_rows(c.v_plane(0), 0, 0, 600)[300:], v[0, :, 0])
    c.close()
    assert torch.ones(8, device="cuda").sum().item() == 8.0
    d = kvc.KVCache(1, 4, 64, [900])
    d.append(k, v, [300], kinds)
    assert d.device_status() == 0
