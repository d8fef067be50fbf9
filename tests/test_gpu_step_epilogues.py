"""The fused epilogues of the step's GEMMs element by element: RoPE on q and k, v stored transposed,
SwiGLU, the residual add, in a step of one layer whose weights let each of them be read from the
residual stream (O projection = identity; down projection = a choice of columns).  Few-row, mid-row
and CTA-pair kernels, heads of 64 and 128 columns, grouped-query, ragged and cached rows; which
kernels a step took is checked by its launches.  Against float64 on the same bf16 weights.

Tolerances.  u = 2^-8 is the largest relative rounding of bf16, 0.4 u its rms.  The normed rows are
rounded to bf16 once, so a sum of their products with d weights is off by 0.4 u of its rms; eight
times that bounds the largest of 10^7 elements.  Each further rounding to bf16 adds u of the value."""
import math

import numpy as np
import pytest
import torch

import synthetic as syn

pytestmark = pytest.mark.gpu

U = 2.0 ** -8
VOCAB = 4096
GEMM_MLP = 12  # DCL_K_GEMM_MLP
MODELS = {("few", 64): dict(d=768, H=12, G=4, F=1024), ("few", 128): dict(d=512, H=4, G=2, F=1536),
          ("mid", 64): dict(d=3584, H=56, G=8, F=18944), ("mid", 128): dict(d=4096, H=32, G=32, F=12288)}
# kernels, prompt, gen, sequences, cache, offset of p
STEPS = [
    ("few", 3, 2, 1, 0, 0),      # 5 rows, ragged
    ("few", 32, 97, 1, 0, 3),    # 129 rows: a second token tile of one row
    ("few", 64, 128, 1, 2, 70),  # the dual cache's block of 32 rows
    ("few", 64, 128, 3, 1, 40),  # suffixes, 288 rows
    ("mid", 90, 181, 2, 0, 7),   # 542 ragged rows
    ("mid", 224, 544, 1, 1, 0),  # a suffix of 544 rows
]


class Model:
    def __init__(self, monkeypatch, override, kind, hd, N, M, B, cache, offset):
        import __graft_entry__
        __graft_entry__.build()
        import paper_2607_20467_gb300 as dcl
        m = MODELS[kind, hd]
        self.dcl, self.hd, self.d, self.H, self.G, self.F = dcl, hd, m["d"], m["H"], m["G"], m["F"]
        self.N, self.T, self.B, self.cache = N, N + M, B, cache
        monkeypatch.setenv("DCL_GEMM_TILES", override)
        shape = syn.ModelShape(1, self.d, self.H, self.G, hd, self.F, VOCAB, VOCAB - 1, 1e4)
        self.c = dcl.Context(shape, max_batch=B, max_seq=N + M)
        self.g = torch.Generator(device="cuda").manual_seed(hd + N + M)
        self.w = {}
        one = torch.ones(self.d, dtype=torch.bfloat16, device="cuda")
        for k in (dcl.DCL_W_ATTN_NORM, dcl.DCL_W_MLP_NORM, dcl.DCL_W_FINAL_NORM):
            self.c.set_weight(k, 0, one)
        self.put("embed", dcl.DCL_W_EMBED, self.normal(VOCAB, self.d, 1.0))
        self.put("head", dcl.DCL_W_LM_HEAD, self.normal(VOCAB, self.d, 0.02))
        r = np.random.default_rng(5)
        self.x = r.integers(0, VOCAB - 1, size=(B, self.T)).astype(np.int32)
        self.p = np.full(B, N + offset, np.int32)
        self.cfg = dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M, kv_cache=cache, max_window=1)
        start = 0 if not cache else N + 32 * (offset // 32)
        self.span = start, min(start + 32, self.T) if cache == 2 else self.T

    def normal(self, rows, cols, std):
        return (std * torch.randn(rows, cols, generator=self.g, device="cuda")).to(torch.bfloat16)

    def put(self, name, kind, w):
        self.w[name] = w
        self.c.set_weight(kind, 0, w)

    def step(self, pair):
        """What a step's layer adds to the rows it computes, [B][rows][d] float64, and the whole embedding."""
        dcl, c = self.dcl, self.c
        c.set_prompt(self.x[:, :self.N], self.cfg)
        c.set_profiling(True)
        c.set_state(self.x, self.p)
        for _ in range(2 if self.cache else 1):  # with a cache: the refresh, then the suffix or the block
            c.step(return_k=True)
        assert (GEMM_MLP in c.profile_last_step()[1]) == pair  # (one launch with the pair kernels only)
        h = [torch.zeros(self.B * self.T, self.d, device="cuda") for _ in range(2)]
        c.forward_debug()
        for layer in (-1, 0):
            c.debug_hidden(layer, h[layer + 1])
        rows = self.B * (self.span[1] - self.span[0])
        ids = self.x.copy()
        for b in range(self.B):
            ids[b, self.p[b]] = VOCAB - 1
        e = self.w["embed"][torch.from_numpy(ids.astype(np.int64)).cuda()].double()
        assert torch.equal(h[0][:rows].double(), e[:, self.span[0]:self.span[1]].reshape(rows, -1))
        return (h[1][:rows].double() - h[0][:rows].double()).view(self.B, -1, self.d), e

    def normed(self, e):
        return e * torch.rsqrt(e.square().mean(-1, keepdim=True) + 1e-5)

    def mul(self, x, name):
        return x @ self.w[name].double().T

    def rope(self, v):  # [B][T][heads][hd]
        ang = torch.arange(self.T, device="cuda", dtype=torch.float64)[:, None] * torch.tensor(
            [1e4 ** (-2.0 * j / self.hd) for j in range(self.hd // 2)], device="cuda", dtype=torch.float64)[None]
        cos, sin, h = ang.cos()[None, :, None], ang.sin()[None, :, None], self.hd // 2
        return torch.cat([v[..., :h] * cos - v[..., h:] * sin, v[..., h:] * cos + v[..., :h] * sin], -1)


@pytest.fixture(params=["", "qkv=pair:1"], ids=["chosen", "pair"])
def override(request):
    return request.param


def _attention_weights(m, q_std, same):
    dcl, d, hd, H, G = m.dcl, m.d, m.hd, m.H, m.G
    k = m.normal(G * hd, d, q_std / math.sqrt(d))
    q = k.view(G, 1, hd, d).expand(G, H // G, hd, d).reshape(H * hd, d).contiguous() if same else m.normal(H * hd, d, q_std / math.sqrt(d))
    m.put("q", dcl.DCL_W_Q, q)
    m.put("k", dcl.DCL_W_K, k)
    m.put("v", dcl.DCL_W_V, m.normal(G * hd, d, 1.0 / math.sqrt(d)))
    m.put("o", dcl.DCL_W_O, torch.eye(d, dtype=torch.bfloat16, device="cuda"))
    m.put("gate", dcl.DCL_W_GATE, m.normal(m.F, d, 0.02))
    m.put("up", dcl.DCL_W_UP, m.normal(m.F, d, 0.02))
    m.put("down", dcl.DCL_W_DOWN, torch.zeros(d, m.F, dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("kind,N,M,B,cache,offset", STEPS)
def test_values(monkeypatch, override, kind, hd, N, M, B, cache, offset):
    """q = k of a length at which every position attends to itself alone: the layer adds v, and an
    element of it is one element of the transposed store."""
    m = Model(monkeypatch, override, kind, hd, N, M, B, cache, offset)
    with m.c:
        _attention_weights(m, 3.0, True)
        got, e = m.step(override != "")
        v = m.mul(m.normed(e), "v")[:, m.span[0]:m.span[1]]
        ref = v.view(B, -1, m.G, 1, hd).expand(-1, -1, -1, m.H // m.G, -1).reshape(got.shape)
        tol = 8 * 0.4 * U * v.square().mean().sqrt() + 2 * U * ref.abs()  # (v and the attention's output are rounded)
        assert ((got - ref).abs() <= tol).all(), float(((got - ref).abs() / tol).max())


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("kind,N,M,B,cache,offset", STEPS)
def test_queries_and_keys(monkeypatch, override, kind, hd, N, M, B, cache, offset):
    """Scores of standard deviation 1.4: rounding (q and k twice each) moves one by 2^0.5 x 0.57 u x 1.4 =
    0.0045, and a head's output by that much of itself, 0.57 u for v and 0.4 u for its own rounding:
    0.0053 in all over the rows of a head, and some times that in a row that few keys dominate.  A
    component of q or k that is off by half moves scores by 0.06 and the head's output by 0.04."""
    m = Model(monkeypatch, override, kind, hd, N, M, B, cache, offset)
    with m.c:
        _attention_weights(m, 1.2, False)
        got, e = m.step(override != "")
        x = m.normed(e)
        q = m.rope(m.mul(x, "q").view(B, m.T, m.H, hd))[:, m.span[0]:m.span[1]]
        k = m.rope(m.mul(x, "k").view(B, m.T, m.G, hd)).repeat_interleave(m.H // m.G, 2)
        v = m.mul(x, "v").view(B, m.T, m.G, hd).repeat_interleave(m.H // m.G, 2)
        for b in range(B):
            a = torch.softmax(torch.einsum("thd,shd->hts", q[b], k[b]) / math.sqrt(hd), -1)
            ref = torch.einsum("hts,shd->thd", a, v[b])
            rel = (got[b].view(ref.shape) - ref).norm(dim=2) / ref.norm(dim=2)
            by_head = rel.square().mean(0).sqrt()
            assert by_head.max() <= 0.01 and rel.max() <= 0.05, (b, float(by_head.max()), float(rel.max()))


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("kind,N,M,B,cache,offset", STEPS)
def test_swiglu_and_residual(monkeypatch, override, kind, hd, N, M, B, cache, offset):
    """v = 0 and a down projection that takes d of the F columns: the layer adds silu(gate) up."""
    m = Model(monkeypatch, override, kind, hd, N, M, B, cache, offset)
    with m.c:
        _attention_weights(m, 1.0, False)
        m.put("v", m.dcl.DCL_W_V, torch.zeros(m.G * hd, m.d, dtype=torch.bfloat16, device="cuda"))
        m.put("gate", m.dcl.DCL_W_GATE, m.normal(m.F, m.d, 1.5 / math.sqrt(m.d)))
        m.put("up", m.dcl.DCL_W_UP, m.normal(m.F, m.d, 1.0 / math.sqrt(m.d)))
        for first in list(range(0, m.F - m.d, m.d)) + [m.F - m.d]:
            down = torch.zeros(m.d, m.F, dtype=torch.bfloat16, device="cuda")
            down[torch.arange(m.d), first + torch.arange(m.d)] = 1.0
            m.put("down", m.dcl.DCL_W_DOWN, down)
            got, e = m.step(override != "")
            x = m.normed(e[:, m.span[0]:m.span[1]])
            g, up = (x @ m.w[n][first:first + m.d].double().T for n in ("gate", "up"))
            s = torch.nn.functional.silu(g)
            # |silu'| <= 1.1; the last term where gate and up are both near 0
            near = 8 * 0.4 * U
            tol = near * (1.1 * up.abs() * 1.5 + s.abs()) + U * (s * up).abs() + 1.1 * 1.5 * near ** 2
            assert ((got - s * up).abs() <= tol).all(), (first, float(((got - s * up).abs() / tol).max()))
