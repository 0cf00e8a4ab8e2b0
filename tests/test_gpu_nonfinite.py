"""Infinities and NaN in the stored rows: they reach exactly the queries that see them.  References are masked softmaxes
in 64 bits by torch."""
import numpy as np
import pytest
import torch

import paper_2310_08152_gb300 as kvc

pytestmark = pytest.mark.gpu

INF, NAN = float("inf"), float("nan")


def _rows(n, H, d, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, H, d, device="cuda", generator=g).clamp(-4, 4).to(dtype)


def _check(got, ref, tol):
    bad = ~torch.isfinite(ref)
    assert torch.equal(torch.isnan(got), bad)
    assert bad.any() and not bad.all()
    assert (got.double() - ref)[~bad].abs().max().item() < tol


@pytest.mark.parametrize("d,dtype", [(64, torch.float16), (64, torch.bfloat16), (80, torch.float16), (80, torch.bfloat16),
                                     (96, torch.float16), (128, torch.bfloat16)])
def test_prefill_of_keys_that_are_not_finite(d, dtype):
    """Three heads: NaN and infinite keys in a span's interior alone (hidden from the queries past its <CR>); an infinite
    key that every later query sees but the <CL> queries, in tiles without the per-key rule for those; a NaN one.
    Outputs are means of |v| < 4 with weights of 16 bits (f16: off by 2^-11 of each, 4 2^-11 = 2e-3) or two parts."""
    L, H, scale = 700, 3, 0.125
    spans = [(20, 60), (130, 170), (300, 340), (420, 460), (600, 630)]
    kinds = np.zeros(L, np.uint8)
    until = np.full(L, L)
    for cl, cr in spans:
        kinds[cl], kinds[cr] = kvc.CL, kvc.CR
        until[cl], until[cl + 1:cr] = cl, cr
    q, k, v = (_rows(L, H, d, dtype, s) for s in range(3))
    k[30, 0, 0], k[140, 0, 1], k[310, 0], k[455, 0, 3] = INF, -INF, NAN, INF
    k[70, 1, 0] = INF
    k[200, 2, 5] = NAN
    c = kvc.KVCache(1, H, d, [L], "f16" if dtype == torch.float16 else "bf16")
    c.append(k, v, [L], kinds)
    got = c.prefill_attention(0, q, [L], scale)
    i, j = torch.arange(L, device="cuda")[:, None], torch.arange(L, device="cuda")[None, :]
    is_cl = torch.from_numpy(kinds == kvc.CL).cuda()[:, None]
    seen = torch.where(is_cl, i == j, (j <= i) & (i <= torch.from_numpy(until).cuda()[None, :]))
    z = torch.einsum("qhd,khd->hqk", q.double(), k.double()) * scale
    p = torch.softmax(z.masked_fill(~seen, -INF), -1)
    _check(got, torch.einsum("hqk,khd->qhd", p, v.double()), 2e-3)
    assert torch.isfinite(got[[20, 130, 300, 420, 600]]).all()  # the <CL> queries
    assert c.device_status() == 0


@pytest.mark.parametrize("d", [64, 80, 96, 128])
def test_decode_by_cta_of_rows_that_are_not_finite(d):
    """A closed span that is not freed yet hides rows of a cluster's CTAs, keys and values of which are NaN and infinite;
    one head sees a NaN key, one an infinite value, one an infinite key."""
    L, H, scale = 1200, 4, 0.125
    kinds = np.zeros(L, np.uint8)
    kinds[500], kinds[900] = kvc.CL, kvc.CR
    k, v = (_rows(L, H, d, torch.float16, s) for s in range(2))
    k[520:700], v[600:880], k[800, :, 3], v[500] = NAN, INF, -INF, NAN
    k[5, 1, 0], v[1150, 2, 7], k[3, 3, 2] = NAN, INF, INF
    c = kvc.KVCache(1, H, d, [L])
    c.append(k, v, [L], kinds)
    q = _rows(1, H, d, torch.float16, 3)
    got = c.decode_attention(0, q, scale)
    assert c.last_decode_plan["workers"] > 4 * H  # clusters
    rows = torch.cat([torch.arange(500), torch.arange(900, L)]).cuda()
    p = torch.softmax(torch.einsum("hd,khd->hk", q[0].double(), k[rows].double()) * scale, -1)
    ref = torch.einsum("hk,khd->hd", p, v[rows].double())
    finite = torch.isfinite(ref)
    assert finite[0].all() and not finite[1].any() and finite[2].sum() == d - 1
    assert torch.equal(torch.isnan(got[0]), torch.isnan(ref)) and torch.equal(torch.isinf(got[0]), torch.isinf(ref))
    # 32-bit sums of d products and of the rows: 1e-5 of |v| < 4
    assert (got[0].double() - ref)[finite].abs().max().item() < 1e-4
    assert c.device_status() == 0
