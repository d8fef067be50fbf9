"""The few-row GEMM (at most 128 rows; weight rows on the MMA's M side) against an fp32
reference of the same bf16 operands, at the edges of its tiles: row counts around the 32-row
groups, output widths around the 128-row weight tiles, K from one 64-wide block to a depth at
which every weight tile is cut over the CTAs of a cluster.

Tolerances.  Both sides multiply the same bf16 values; a product is exact in fp32, so they
differ by fp32 rounding in K-term sums, at most K * 2^-24 * sum |a w| per element (taken as
4 sqrt(K) 2^-24 of the root of the summed squares times 8 for the largest of ~10^5 elements),
plus, for a bf16 output, half an ulp: 2^-8 of the value."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as pkg
    with pkg.Context() as c:
        yield c


def _operands(M, N, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    w = (0.05 * torch.randn(N, K, generator=g, device="cuda")).to(torch.bfloat16)
    ref = a.double() @ w.double().T
    scale = torch.sqrt(a.double().square() @ w.double().square().T)  # root of the summed squares
    return a, w, ref, 32 * K ** 0.5 * 2.0 ** -24 * scale


@pytest.mark.parametrize("M", [1, 31, 32, 33, 96, 127, 128])
@pytest.mark.parametrize("N,K", [(32, 64), (128, 64), (160, 192), (256, 4096), (4096, 4096), (3616, 1024), (512, 12288)])
def test_linear_matches_reference(ctx, M, N, K):
    a, w, ref, tol = _operands(M, N, K, M * 7919 + N + K)
    out = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    ctx.op_linear(a, w, out)
    assert ((out.double() - ref).abs() <= tol + 2.0 ** -8 * ref.abs()).all()
    res = torch.randn(M, N, device="cuda")
    acc = res.clone()
    ctx.op_linear(a, w, acc, mode=1)
    # (the residual's own fp32 addition rounds once more)
    assert ((acc.double() - res.double() - ref).abs() <= tol + 2.0 ** -23 * (ref.abs() + res.double().abs())).all()


def test_repeats_bit_for_bit(ctx):
    a, w, _, _ = _operands(96, 4096, 4096, 5)
    first = torch.empty(96, 4096, dtype=torch.bfloat16, device="cuda")
    ctx.op_linear(a, w, first)
    for _ in range(20):  # (a cut tile's sums are added in K order)
        out = torch.empty_like(first)
        ctx.op_linear(a, w, out)
        assert torch.equal(out.view(torch.int16), first.view(torch.int16))


# rows of the step after a refresh: (prompt, gen, sequences, cache, offset of p) -> rows
STEPS = [
    (3, 2, 1, 0, 0),      # 5 rows, full recompute, positions no multiple of 32 (v through the transpose launch)
    (32, 64, 1, 0, 10),   # 96 rows, full recompute
    (64, 64, 1, 0, 40),   # 128 rows
    (64, 128, 1, 2, 70),  # the dual cache's 32-row block
    (64, 128, 3, 2, 20),  # three blocks, 96 rows
    (64, 128, 1, 1, 40),  # suffix of 96 rows
    (64, 128, 1, 1, 5),   # suffix of 128 rows
    (32, 97, 1, 0, 3),    # 129 rows: a second token tile of one row
    (37, 90, 3, 0, 21),   # 381 rows of three ragged sequences
    (64, 128, 8, 1, 5),   # suffixes of 128 rows, 1024 in all, after a refresh of 1536
]
# heads of 64 and of 128 columns, grouped-query
MODELS = {64: dict(d=768, H=12, G=4, F=1024), 128: dict(d=512, H=4, G=2, F=1536)}


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("N,M,B,cache,offset", STEPS)
def test_step_matches_the_pair_gemms(ctx, monkeypatch, hd, N, M, B, cache, offset):
    """A forward with the few-row GEMMs against the same forward on the CTA-pair GEMMs (a tile
    override keeps a step on those).  Each lies within 3.5e-3 relative rms per row of the
    64-bit forward per block (the teacher-forced bound), so they differ by at most twice that
    per block."""
    import paper_2607_20467_gb300 as dcl
    import synthetic as syn
    m = MODELS[hd]
    shape = syn.ModelShape(2, m["d"], m["H"], m["G"], hd, m["F"], 4096, 4095, 1e4)
    x, p = syn.decode_state(3, syn.prompt_ids(3, B, N, 4095), M, offset, max(1, M // 2), 4095)
    cfg = dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M, kv_cache=cache)
    start = 0 if not cache else N + 32 * (offset // 32)
    end = min(start + 32, N + M) if cache == 2 else N + M
    rows = B * (end - start)
    got = []
    for override in ("", "qkv=pair:1"):
        monkeypatch.setenv("DCL_GEMM_TILES", override)
        with dcl.Context(shape, max_batch=B, max_seq=N + M) as c:
            c.init_random_weights(7, 0.02, 2.0, 0.1)
            c.set_prompt(x[:, :N], cfg)
            c.set_state(x, p)
            out = []
            for _ in range(2):  # with a cache: the refresh, then the suffix or the block
                c.step()
                h = torch.zeros(B * (N + M), m["d"], device="cuda")
                p1 = torch.zeros(B, M, device="cuda")
                c.forward_debug(p1=p1)
                c.debug_hidden(1, h)
                out += [h[:rows].clone(), p1]
            got.append(out)
    for a, b in zip(got[0], got[1]):
        a, b = a.double(), b.double()
        rel = (a - b).norm(dim=1) / b.norm(dim=1)
        assert rel.max() <= 2 * 2 * 3.5e-3, rel.max()


def test_a_finished_sequence_leaves_its_neighbour_alone(ctx):
    """Sequences of 127 positions: with the first finished the step
    computes the second's rows only, from other places of every buffer, to the same bits."""
    import paper_2607_20467_gb300 as dcl
    import synthetic as syn
    m = MODELS[64]
    shape = syn.ModelShape(2, m["d"], m["H"], m["G"], 64, m["F"], 4096, 4095, 1e4)
    N, M, B = 37, 90, 2
    x, p = syn.decode_state(3, syn.prompt_ids(3, B, N, 4095), M, 21, M // 2, 4095)
    with dcl.Context(shape, max_batch=B, max_seq=N + M) as c:
        c.init_random_weights(7, 0.02, 2.0, 0.1)
        c.set_prompt(x[:, :N], dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M))
        both, other, alone = (torch.zeros(B, M, device="cuda") for _ in range(3))
        c.set_state(x, p)
        c.forward_debug(p1=both)
        y = x.copy()
        y[1, N:N + 20] = 11
        c.set_state(y, p)
        c.forward_debug(p1=other)  # other contents everywhere
        x[0, N:], p[0] = 5, N + M
        c.set_state(x, p)
        c.forward_debug(p1=alone)
        assert torch.equal(both[1], alone[1])
        assert not torch.equal(both[1], other[1])
