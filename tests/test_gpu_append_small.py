"""Appends of a few tokens, whose upload is a kernel parameter, and of a few more, whose upload is staged: at the
parameter's size (49 sequences fit, 50 do not) and at the number of units that take the other kernels."""
import numpy as np
import pytest
import torch

import paper_2310_08152_gb300 as kvc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,M,by_layer", [(1, 1, False), (1, 1, True), (49, 3, False), (49, 3, True), (50, 3, False),
                                          (49, 4, False), (4, 38, False), (4, 37, False)])
def test_append_of_one_token_a_sequence(b, M, by_layer):
    """Three steps (a sequence sits out the second): stored rows, positions and history indices exactly, and the
    decode that reads the uploaded state.  Its scores err by at most d^2 2^-24 scale = 3e-5 for |q|, |k| < 4 in
    d = 64 terms, and the outputs, weighted means of |v| < 5, by less than 5 times twice that."""
    H, d, scale = 2, 64, 0.125
    g = torch.Generator(device="cuda").manual_seed(b * M)
    c = kvc.KVCache(M, H, d, [4] * b)
    rows = [[] for _ in range(b)]
    for step in range(3):
        n_new = np.ones(b, np.int32)
        if step == 1 and b > 1:
            n_new[b // 2] = 0
        n = int(n_new.sum())
        k, v = (torch.randn(M, n, H, d, device="cuda", generator=g).clamp(-4, 4).half() for _ in range(2))
        kinds = np.zeros(n, np.uint8)
        if by_layer:
            for m in range(M):
                c.append(k[m], v[m], n_new, kinds, layer=m)
        else:
            c.append(k, v, n_new, kinds)
        for i, s in enumerate(np.flatnonzero(n_new)):
            rows[s].append((k[:, i], v[:, i]))
    q = torch.randn(M, b, H, d, device="cuda", generator=g).clamp(-4, 4).half()
    out = c.decode_attention_layers(q, scale).double()
    assert c.lengths()[0].tolist() == [len(r) for r in rows]
    for s in {0, b // 2, b - 1}:
        K, V = (torch.stack([r[i] for r in rows[s]], 2) for i in range(2))  # [M][H][n][d]
        n = K.shape[2]
        for m in range(M):
            for h in range(H):
                assert torch.equal(c.stream_rows(c.k_plane(m), s, h, n), K[m, h])
                assert torch.equal(c.stream_rows(c.v_plane(m), s, h, n), V[m, h])
        lo = int(c.offsets[s])
        assert c.pos[lo:lo + n].tolist() == list(range(n)) == c.orig[lo:lo + n].tolist()
        p = torch.softmax(torch.einsum("mhd,mhnd->mhn", q[:, s].double(), K.double()) * scale, -1)
        ref = torch.einsum("mhn,mhnd->mhd", p, V.double())
        assert (out[:, s] - ref).abs().max().item() < 3e-4
    assert c.device_status() == 0
