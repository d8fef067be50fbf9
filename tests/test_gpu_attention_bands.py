"""The attention kernel where its work split can go wrong: partial bands and tiles, query heads
that share a kv head packed into one tile, the key axis split over clusters of 2, 4 and 8 CTAs
(with shares of unequal length and a ragged last block), and a running maximum that has to be
raised late (so that O is rescaled).

Against float64 softmax(q k^T / sqrt(hd)) v on the same bf16 inputs.  Tolerance: P is rounded to
fp16 (2^-12 relative) and O to bf16 (2^-9), so an element is within 2^-9 |o| + 2^-11 max |v|
(probabilities sum to one); doubled for the fp32 sums and the approximate exp2."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ops():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as dcl
    ctx = dcl.Context(None, 1, 1)
    yield ctx
    ctx.close()


def _check(ops, qkv, B, T, H, G, hd, qr):
    out = torch.full((B * T, H * hd), float("nan"), dtype=torch.bfloat16, device="cuda")
    ops.op_attention(qkv, out, B, T, H, G, hd, qr)
    torch.cuda.synchronize()
    x = qkv.view(B, T, H + 2 * G, hd).double()
    q0 = T - qr if qr else 0
    o = out.view(B, T, H, hd)
    assert torch.isnan(o[:, :q0]).all()  # rows outside the query set untouched
    for b in range(B):
        k, v = (x[b, :, a:a + G].repeat_interleave(H // G, 1) for a in (H, H + G))
        p = torch.softmax(torch.einsum("thd,shd->hts", x[b, q0:, :H], k) / math.sqrt(hd), -1)
        ref = torch.einsum("hts,shd->thd", p, v)
        err = (o[b, q0:].double() - ref).abs()
        tol = 2 * (2.0 ** -9 * ref.abs() + 2.0 ** -11 * v.abs().max())
        assert (err <= tol).all(), (b, float((err / tol).max()))


@pytest.mark.parametrize("B,T,H,G,hd,qr", [
    (1, 1, 4, 4, 128, 0), (1, 33, 2, 2, 64, 0), (3, 129, 6, 2, 64, 0), (2, 160, 7, 1, 128, 0), (1, 257, 1, 1, 128, 0),
    (5, 896, 28, 4, 128, 32),   # seven heads of a group in one unit, split over the keys
    (1, 1000, 4, 1, 64, 64), (1, 1024, 2, 2, 128, 32), (1, 1153, 2, 1, 128, 96), (1, 2000, 1, 1, 128, 160),
    (1, 384, 32, 32, 128, 32), (16, 512, 8, 8, 64, 288)])
def test_bands(ops, B, T, H, G, hd, qr):
    g = torch.Generator(device="cuda").manual_seed(T * 31 + H)
    qkv = torch.randn(B * T, (H + 2 * G) * hd, generator=g, device="cuda").to(torch.bfloat16)
    _check(ops, qkv, B, T, H, G, hd, qr)


@pytest.mark.parametrize("qr", [0, 32])
def test_late_maximum(ops, qr):
    """Scores that grow along the keys: the reference maximum is raised in several blocks (by more
    than 2^8), in every part of a split."""
    B, T, H, G, hd = 1, 1100, 4, 2, 128
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(B * T, H + 2 * G, hd, generator=g, device="cuda")
    x[:, :H, 0] = 8.0
    x[:, H:H + G, 0] = (torch.arange(T, device="cuda") / 16)[:, None]  # adds up to 48 to a score
    _check(ops, x.view(B * T, -1).to(torch.bfloat16).contiguous(), B, T, H, G, hd, qr)


@pytest.mark.parametrize("base", [-2.0 ** 14, -2.0 ** 10, 2.0 ** 10, 2.0 ** 14])
@pytest.mark.parametrize("B,T,H,G,hd,qr", [(8, 300, 16, 16, 128, 0), (8, 300, 16, 16, 64, 0),  # whole
                                           (1, 1100, 4, 2, 128, 32), (1, 1100, 4, 2, 64, 32)])  # split
def test_large_scores(ops, B, T, H, G, hd, qr, base):
    """Scores near +-10^3 and +-10^4 that differ by a few within a block, and along the keys by up
    to 12 in 16 steps: the reference maximum has to follow them exactly, P being held in fp16.
    q and k are small integers and powers of two, so q k^T is exact in fp32 (integers below 2^18)
    and the tolerance that of small scores."""
    g = torch.Generator(device="cuda").manual_seed(11)
    q, k = (torch.randint(-2, 3, (B * T, n, hd), generator=g, device="cuda").float() for n in (H, G))
    root = 8.0  # q k^T / root: base + steps (sqrt(hd) for hd = 64; for 128 the scores are 0.71 of that)
    q[..., 0], k[..., 0] = base / 128, 128.0 * root           # every score: base
    q[..., 1], k[..., 1] = 1.0, 6.0 * ((torch.arange(B * T, device="cuda") * 16 // T) % 16)[:, None]
    v = torch.randn(B * T, G, hd, generator=g, device="cuda")
    _check(ops, torch.cat([q, k, v], 1).view(B * T, -1).to(torch.bfloat16).contiguous(), B, T, H, G, hd, qr)
