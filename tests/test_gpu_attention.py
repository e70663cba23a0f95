"""Prefill attention where its tiling can go wrong (tiles of one and of two
128-row halves, halves that end on different pages or hold a single row), against
the fp64 softmax within the error of the split operands."""
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
