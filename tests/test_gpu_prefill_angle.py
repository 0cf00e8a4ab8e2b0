"""The rotation of the prefill's queries at far positions, where the turns' rounding error has to be carried: softmax
weights, read through unit rows of V, against 64 bits."""
import numpy as np
import pytest
import torch

import paper_2310_08152_gb300 as kvc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 80, 96, 128])
@pytest.mark.parametrize("base", [0, 4000, 100003, 1 << 22])
def test_rotated_queries_at_far_positions(d, base):
    """bf16, head p with its p-th pair of dimensions alone, |q|, |k| <= 4 sqrt 2 of them.  A logit is off by the query's two
    parts (2^-17 of it), the sine's 2^-21, the angle's 1e-7 turns (6e-7) and the weight's two parts (2^-17), all told
    scale |q| |k| 2^-16 + 2^-16 = 1.4e-4 with |q| |k| <= 32, scale 1/4; without the turns' error 4e-4 at 4,000 and 1e-2 at
    100,003."""
    L, H, scale, half = 64, 4, 0.25, d // 2
    g = torch.Generator(device="cuda").manual_seed(d + base)
    q, k = (torch.zeros(L, H, d, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for p in range(H):
        for x in (q, k):
            x[:, p, [p, p + half]] = (torch.rand(L, 2, generator=g, device="cuda") * 8 - 4).bfloat16()
    v = torch.zeros(L, H, d, dtype=torch.bfloat16, device="cuda")
    v[torch.arange(L), :, torch.arange(L)] = 1
    pos = (base + 37 * np.arange(L)).astype(np.int32)
    c = kvc.KVCache(1, H, d, [L], "bf16", d)
    c.append(k, v, [L], np.zeros(L, np.uint8), pos=pos)
    w = c.prefill_attention(0, q, [L], scale).double()
    for p in range(H):
        a = torch.from_numpy(pos.astype(np.float64)).cuda() * 10000.0 ** (-2.0 * p / d)
        x, y = q[:, p, p].double(), q[:, p, p + half].double()
        x, y = x * a.cos() - y * a.sin(), y * a.cos() + x * a.sin()
        kr = c.stream_rows(c.k_plane(0), 0, p, L).double()  # as stored
        z = (x[:, None] * kr[None, :, p] + y[:, None] * kr[None, :, p + half]) * scale
        z = z.masked_fill(torch.triu(torch.ones_like(z), 1) > 0, -float("inf"))
        ref, got = torch.log_softmax(z, -1), w[:, p, :L].log()
        err = (got - ref)[torch.isfinite(ref)].abs().max().item()
        assert err < 2 * 1.4e-4, (p, err)  # of a logit against the others' mean
    assert c.device_status() == 0
