"""Attention where its tiling can go wrong, against the fp64 softmax: prefill (tiles
of one and of two 128-row halves, halves that end on different pages or hold a
single row) within the error of the split operands; decode on the tensor cores
(one and several pages a block, one block and many a request) at fp32."""
import math

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
P = 64


@pytest.fixture(scope="module")
def L():
    need_gpu()
    from paper_2512_21835_gb300 import loip
    return loip


def paged(lens, Hkv, d, seed):
    """Keys and values of the requests in randomly placed pages; the rest of each
    last page is NaN (nothing may read it into a result)."""
    import torch
    gen = torch.Generator("cuda").manual_seed(seed)
    n = [-(-t // P) for t in lens]
    kv = torch.randn(sum(n), 2, Hkv, P, d, generator=gen, device="cuda").to(torch.bfloat16)
    order, at = np.random.default_rng(seed).permutation(sum(n)), 0
    table = np.zeros((len(lens), max(n)), dtype=np.int64)
    flat = []
    for b, t in enumerate(lens):
        table[b, :n[b]] = order[at:at + n[b]]
        at += n[b]
        if t % P:
            kv[table[b, n[b] - 1], :, :, t % P:] = float("nan")
        pages = kv[torch.from_numpy(table[b, :n[b]]).cuda()]
        flat.append([pages[:, i].permute(0, 2, 1, 3).reshape(-1, Hkv, d)[:t].double() for i in (0, 1)])
    page_bytes = 2 * Hkv * P * d * 2
    return kv, torch.from_numpy(table * page_bytes).cuda(), page_bytes, flat


def softmax_rows(q, k, v, pos):
    """q [T, Hq, d] at positions pos over k, v [S, Hkv, d]: outputs and the weights' sums of |v|."""
    import torch
    G = q.shape[1] // k.shape[1]
    out, mag = torch.empty_like(q), torch.empty_like(q)
    mask = torch.arange(k.shape[0], device="cuda")[None] > pos[:, None]
    for h in range(q.shape[1]):
        w = torch.softmax((q[:, h] @ k[:, h // G].T / math.sqrt(q.shape[2])).masked_fill(mask, -math.inf), -1)
        out[:, h], mag[:, h] = w @ v[:, h // G], w @ v[:, h // G].abs()
    return out, mag


# at G = 1 and 8 kv heads a half is 128 positions, and 19 tiles of a half or fewer
# stay single: (40 kv heads) 385 rows are past that, 300 are not
@pytest.mark.parametrize("Hq,Hkv,d,lens,first", [
    (40, 40, 128, (385,), (0,)), (40, 40, 128, (300,), (63,)), (64, 8, 128, (513, 17, 64), (0, 100, 63)),
    (32, 8, 128, (1025, 33), (0, 0)), (16, 8, 64, (129, 1500), (5, 0)), (8, 8, 64, (2560, 1), (0, 0))])
def test_prefill_halves(L, Hq, Hkv, d, lens, first):
    import torch
    total = [n + f for n, f in zip(lens, first)]
    kv, table, page_bytes, flat = paged(total, Hkv, d, 3)
    M = sum(lens)
    q = torch.randn(M, Hq * d, generator=torch.Generator("cuda").manual_seed(4), device="cuda")
    tiles = torch.empty((M + len(lens)) * 16, dtype=torch.uint8, device="cuda")
    o = torch.empty(2, M, Hq * d, dtype=torch.bfloat16, device="cuda")
    L.loip_k_prefill_attention(q, kv, table, table.shape[1], lens, first, Hq, Hkv, d, P, 0, page_bytes, tiles, o)
    assert L.loip_k_attention_tc_status() == 0
    got, at = (o[0].double() + o[1].double()).view(M, Hq, d), 0
    for b, n in enumerate(lens):
        want, mag = softmax_rows(q[at:at + n].double().view(n, Hq, d), *flat[b],
                                 torch.arange(first[b], total[b], device="cuda"))
        # scores are off by 2^-17 of their terms' sizes (|q| |k| / sqrt d ~ sqrt d, a few
        # times that at most), which scales the weights; weights and outputs by 2^-17
        tol = 2.0 ** -17 * (8 * math.sqrt(d) + 4) * mag + 1e-6
        assert bool(((got[at:at + n] - want).abs() <= tol).all())
        at += n


# max_ctx decides for the tensor cores (512 pages over all requests and kv heads,
# 1280 with fewer than four query heads each); the lengths for the pages per block
@pytest.mark.parametrize("Hq,Hkv,d,max_ctx,lens", [
    (64, 8, 128, 4096, (1,)), (64, 8, 128, 4096, (4096,)), (32, 8, 128, 16384, (16384, 17, 4033, 64)),
    (40, 40, 128, 4096, (65, 2111)), (16, 8, 64, 8192, (15, 16, 8191)), (8, 8, 64, 16384, (16321,)),
    (64, 8, 128, 1088, (1088, 63, 1, 640, 129, 1025, 48, 700))])
def test_decode_long(L, Hq, Hkv, d, max_ctx, lens):
    import torch
    kv, table, page_bytes, flat = paged(lens, Hkv, d, 5)
    B, pages = len(lens), max_ctx // P
    assert pages * Hkv * B >= (512 if Hq >= 4 * Hkv else 1280)
    pt = torch.zeros(B, pages, dtype=torch.int64, device="cuda")
    pt[:, :table.shape[1]] = table
    q = torch.randn(B, Hq * d, generator=torch.Generator("cuda").manual_seed(6), device="cuda")
    scratch = torch.empty(L.loip_k_attention_scratch_floats(B, Hq, d, max_ctx, P), device="cuda")
    o, again = torch.empty(B, Hq * d, device="cuda"), torch.empty(B, Hq * d, device="cuda")
    ctx = torch.tensor(lens, dtype=torch.int32, device="cuda")
    for out in (o, again):
        L.loip_k_attention(q, kv, pt, pages, ctx, Hq, Hkv, d, P, 0, page_bytes, max_ctx, scratch, out)
    assert torch.equal(o, again)
    for b, n in enumerate(lens):
        want, mag = softmax_rows(q[b:b + 1].double().view(1, Hq, d), *flat[b],
                                 torch.tensor([n - 1], device="cuda"))
        # scores: d-term fp32 sums of |q||k|/sqrt d ~ sqrt d, which scale the weights;
        # outputs: up to n/16 weighted adds per warp
        tol = 2.0 ** -24 * ((d + 16) * 4 + n / 16 + 64) * mag + 1e-9
        assert bool(((o[b].double().view(1, Hq, d) - want).abs() <= tol).all())


def test_decode_infinities(L):
    """As in plain fp32: an infinite value reaches the outputs of its dim only, an
    infinitely low score has weight zero, an infinitely high one gives NaN."""
    import torch
    Hq, Hkv, d, n, max_ctx = 8, 1, 128, 700, 16384
    page_bytes, pages, B = 2 * Hkv * P * d * 2, max_ctx // P, 2
    kv = torch.randn(11, 2, Hkv, P, d, generator=torch.Generator("cuda").manual_seed(7), device="cuda").to(torch.bfloat16)
    pt = torch.zeros(B, pages, dtype=torch.int64, device="cuda")
    pt[:, :11] = torch.arange(11, device="cuda") * page_bytes
    q = torch.randn(B, Hq * d, device="cuda").abs()
    q[1].neg_()  # request 1 scores the infinite key infinitely high
    kv[3, 1, 0, 20, 5] = float("inf")
    kv[6, 0, 0, 33, 9] = float("-inf")
    assert pages * Hkv * B >= 512
    scratch = torch.empty(L.loip_k_attention_scratch_floats(B, Hq, d, max_ctx, P), device="cuda")
    o = torch.empty(B, Hq * d, device="cuda")
    L.loip_k_attention(q, kv, pt, pages, torch.tensor([n, n], dtype=torch.int32, device="cuda"), Hq, Hkv, d, P, 0,
                       page_bytes, max_ctx, scratch, o)
    o = o.view(B, Hq, d)
    assert bool(torch.isinf(o[0, :, 5]).all()) and bool((o[0, :, 5] > 0).all())
    fine = torch.ones(d, dtype=torch.bool, device="cuda")
    fine[5] = False
    k, v = (kv[:, i].permute(0, 2, 1, 3).reshape(-1, d)[:n].double() for i in (0, 1))
    w = torch.softmax(q[0].double().view(Hq, d) @ k.T / math.sqrt(d), -1)
    assert torch.allclose(o[0][:, fine].double(), (w @ v)[:, fine], rtol=1e-4, atol=1e-5)
    assert bool(torch.isnan(o[1]).all())
