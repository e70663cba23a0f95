"""The projections of 2 to 8 rows (three-part bf16 activations on the tensor
cores) and of one row (a ring of bulk copies) at the sizes where their tiling can
go wrong, against the oracle within the a-priori fp32 summation bound, and their
behaviour on infinities and NaN."""
import numpy as np
import pytest

from gpu_util import U, dev_bits, dev_f32, dot_bound, need_gpu
from paper_2512_21835_gb300 import inputs

pytestmark = pytest.mark.gpu
SEED = 0x10A1B


@pytest.fixture(scope="module")
def L():
    need_gpu()
    from paper_2512_21835_gb300 import loip
    return loip


# K: below, at and past the 512-column chunk, with and without a multiple of 64
# (tensor-map loads or 16-byte copies); N: fewer rows than a tile, uneven ranges
# per block, several passes of eight tiles (> 152 x 128 rows)
@pytest.mark.parametrize("B,N,K", [(2, 1, 8), (8, 17, 64), (3, 4096, 512), (8, 300, 520), (5, 2433, 576),
                                   (2, 1000, 1544), (8, 20000, 72), (4, 39000, 64),
                                   (1, 401, 10816), (1, 2433, 1984), (1, 66000, 64)])
def test_resid_tiles(L, orc, B, N, K):
    a = inputs.normal_f32(3 * K + N, (B, K), 0.7)
    x0 = inputs.normal_f32(N, (B, N), 1.0)
    W = orc.gen_tensor(SEED, 40, N * K, 0).reshape(N, K)
    x = dev_f32(x0)
    L.loip_k_down(dev_f32(a), dev_bits(W), x)
    got, W64 = x.cpu().numpy().astype(np.float64), orc.bf16_bits_to_f64(W)
    want = x0.astype(np.float64) + a.astype(np.float64) @ W64.T
    for b in range(B):
        tol = dot_bound(W64, a[b].astype(np.float64), K) + 4 * U * np.abs(want[b])
        assert np.all(np.abs(got[b] - want[b]) <= tol)
    assert L.loip_k_tc_status() == 0


# the query / key / value ranges of a block begin and end inside a head
@pytest.mark.parametrize("B,H,Hq,Hkv,d", [(2, 576, 40, 40, 128), (8, 200, 24, 3, 64), (5, 1024, 64, 8, 128),
                                          (1, 576, 40, 40, 128), (1, 448, 72, 72, 64)])
def test_qkv_ranges(L, orc, B, H, Hq, Hkv, d):
    import torch
    P, eps, theta = 64, 1e-5, 10000.0
    x = inputs.normal_f32(H, (B, H), 1.2)
    g = orc.gen_tensor(SEED, 30, H, 1)
    rows = (Hq + 2 * Hkv) * d
    W = orc.gen_tensor(SEED, 31, rows * H, 0).reshape(rows, H)
    pos = np.array([(7 * b) % P for b in range(B)], dtype=np.int32)
    page = 2 * Hkv * P * d * 2
    kv = torch.zeros(B * page, dtype=torch.uint8, device="cuda")
    q = torch.empty(B, Hq * d, device="cuda")
    L.loip_k_qkv_rope(dev_f32(x), dev_bits(g), dev_bits(W), Hq, Hkv, d, eps, theta, dev_f32(pos).int(), q, kv,
                      torch.arange(B, device="cuda", dtype=torch.int64) * page, 1, P, 0, page)
    W64 = orc.bf16_bits_to_f64(W)
    cache = kv.cpu().numpy().view(np.uint16).reshape(B, 2, Hkv, P, d)
    for b in range(B):
        y = orc.rmsnorm(x[b].astype(np.float64), g, eps)
        r = W64 @ y
        tol = dot_bound(W64, y, H) + 8 * U * np.abs(r)
        heads, ht = r.reshape(-1, d), tol.reshape(-1, d)
        rot = np.stack([orc.rope(h, int(pos[b]), theta) for h in heads[:Hq + Hkv]])
        # rotating mixes a pair's errors; cos and sin are good to a few ulp
        rt = np.tile(ht[:, :d // 2] + ht[:, d // 2:], 2)[:Hq + Hkv] + 8 * U * np.linalg.norm(rot, axis=1)[:, None]
        assert np.all(np.abs(q[b].cpu().numpy().reshape(Hq, d) - rot[:Hq]) <= rt[:Hq])
        for got, want, t in ((cache[b, 0, :, pos[b]], rot[Hq:], rt[Hq:]), (cache[b, 1, :, pos[b]], heads[Hq + Hkv:], ht[Hq + Hkv:])):
            got = orc.bf16_bits_to_f64(got)
            assert np.all(np.abs(got - want) <= t + 2.0 ** -8 * (np.abs(want) + t))  # stored as bf16


def test_infinities_and_nan(L, orc):
    """As in a plain fp32 product: an infinite weight or activation gives an
    infinite sum (or NaN against a zero), a NaN spoils its own row only."""
    B, N, K = 4, 40, 640
    a = inputs.normal_f32(1, (B, K), 1.0)
    a[0, 5], a[1, 7], a[2, 9], a[:, 11] = 1.0, np.inf, np.nan, 0.5
    W = (orc.gen_tensor(SEED, 40, N * K, 0).reshape(N, K)).copy()
    W[3, 11], W[4, 5], W[6, 11] = 0x7f80, 0xff80, 0x7fc0  # +inf, -inf, NaN
    W[8, 7] = 0
    x = dev_f32(np.zeros((B, N)))
    L.loip_k_down(dev_f32(a), dev_bits(W), x)
    got = x.cpu().numpy()
    with np.errstate(invalid="ignore"):
        want = (a.astype(np.float64) @ orc.bf16_bits_to_f64(W).T).astype(np.float32)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    fine = np.isfinite(want)
    assert np.allclose(got[fine], want[fine], rtol=1e-4, atol=1e-4)
