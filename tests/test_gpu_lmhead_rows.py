"""The LM head of few rows (of a large head up to 16 are padded to 32 in scratch): every output
against float64 at row counts around the padding's end, repeated so that scratch of the call before is reused, with
vocabularies that end inside a 256-column tile and inside a chunk of 32 columns, tied maxima
included.  p1, p2 and H: fp32 sums of d products of bf16 values and of V exponentials, within
1e-4 absolute (as the other LM-head tests use 1e-3)."""
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


@pytest.mark.parametrize("V,d", [(1000, 128), (4097, 256), (33, 64), (126464, 256)])
@pytest.mark.parametrize("R", [16, 1, 7, 17, 31, 129])
def test_rows(ops, R, V, d):
    g = torch.Generator(device="cuda").manual_seed(R * V + d)
    x = torch.randn(R, d, generator=g, device="cuda").to(torch.bfloat16)
    w = (0.3 * torch.randn(V, d, generator=g, device="cuda")).to(torch.bfloat16)
    if V > 40:
        w[37] = w[5]  # equal logits in two chunks of 32 columns: the lower id counts
    t1 = torch.full((R,), -1, dtype=torch.int32, device="cuda")
    p1, p2, h = (torch.zeros(R, device="cuda") for _ in range(3))
    ops.op_lmhead_top2(x, w, t1, p1, p2, entropy=h)
    torch.cuda.synchronize()
    logp = torch.log_softmax(x.double() @ w.double().T, 1)
    two, ids = logp.topk(2, 1)
    assert (p1.double() - two[:, 0].exp()).abs().max() <= 1e-4
    assert (p2.double() - two[:, 1].exp()).abs().max() <= 1e-4
    assert (h.double() + (logp.exp() * logp).sum(1)).abs().max() <= 1e-4 * max(1.0, float(h.max()))
    lowest = (logp == two[:, :1]).int().argmax(1)
    sure = two[:, 0] - two[:, 1] > 1e-4
    sure |= (lowest == 5)
    assert (t1.long() == lowest)[sure].all()


@pytest.mark.parametrize("R", [16, 1, 7, 17])
def test_rows_of_a_large_head(ops, R):
    """Where up to 16 rows are padded: column tiles for most of the SMs, the last one ragged."""
    test_rows(ops, R, 32003, 2048)


@pytest.mark.parametrize("V,d,padded", [(4097, 256, False), (32003, 2048, True), (32003, 1984, False)])
def test_only_large_heads_copy_their_rows(ops, V, d, padded):
    """The copy and the zeros of the padding, 4 to 5 us, are not paid where it gains nothing."""
    from torch.profiler import ProfilerActivity, profile
    x, w = (torch.zeros(n, d, dtype=torch.bfloat16, device="cuda") for n in (4, V))
    t1, p1, p2 = (torch.zeros(4, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32))
    for _ in range(2):  # (the first profile records nothing)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            ops.op_lmhead_top2(x, w, t1, p1, p2)
            torch.cuda.synchronize()
    names = [e.name for e in prof.events()]
    assert any("gemm_tc" in n for n in names)
    assert any("Memset" in n or "DtoD" in n for n in names) == padded, names
