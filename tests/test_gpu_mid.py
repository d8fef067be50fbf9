"""The mid-row GEMMs (weights on the MMA's M side, tiles of tokens on its N side) in a step: row
counts just past a multiple of 256, a last token tile of one row, sequences that are no multiple of
32, K split with ordered adds, heads of 64 and 128 columns, and cached suffixes.

Each step's rows are checked to be ones that the library takes to these kernels (the profiled
launches of an unfused MLP), and the forward is compared with the same on the CTA-pair GEMMs (a tile
override): each lies within 3.5e-3 relative rms per row of the 64-bit forward per block (the
teacher-forced bound), so they differ by at most twice that per block."""
import pytest
import torch

pytestmark = pytest.mark.gpu

MODELS = {64: dict(d=3584, H=56, G=8, F=18944), 128: dict(d=4096, H=32, G=32, F=12288)}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _forward(monkeypatch, override, hd, N, M, B, cache, offset):
    import paper_2607_20467_gb300 as dcl
    import synthetic as syn
    m = MODELS[hd]
    shape = syn.ModelShape(2, m["d"], m["H"], m["G"], hd, m["F"], 4096, 4095, 1e4)
    x, p = syn.decode_state(3, syn.prompt_ids(3, B, N, 4095), M, offset, max(1, M // 2), 4095)
    cfg = dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M, kv_cache=cache)
    monkeypatch.setenv("DCL_GEMM_TILES", override)
    with dcl.Context(shape, max_batch=B, max_seq=N + M) as c:
        c.init_random_weights(7, 0.02, 1.0, 0.1)
        c.set_prompt(x[:, :N], cfg)
        c.set_profiling(True)
        c.set_state(x, p)
        out = []
        for _ in range(2 if cache else 1):  # with a cache: the refresh, then the suffix
            c.step()
            h = torch.zeros(B * (N + M), m["d"], device="cuda")
            p1 = torch.zeros(B, M, device="cuda")
            c.forward_debug(p1=p1)
            c.debug_hidden(1, h)
            out += [h, p1]
        return out, len(c.profile_last_step()[1])


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("N,M,B,cache,offset", [
    (256, 257, 1, 0, 0),    # 513 rows: a last tile of few rows
    (160, 384, 1, 0, 100),  # 544
    (90, 181, 2, 0, 7),     # 542 rows of two ragged sequences
    (512, 544, 1, 0, 3),    # 1056
    (224, 544, 1, 1, 0),    # a refresh of 768, then a suffix of 544
])
def test_step_matches_the_pair_gemms(monkeypatch, hd, N, M, B, cache, offset):
    got, n_mid = _forward(monkeypatch, "", hd, N, M, B, cache, offset)
    want, n_pair = _forward(monkeypatch, "qkv=pair:1", hd, N, M, B, cache, offset)
    assert n_mid == n_pair + 2  # (two layers, the MLP in two launches)
    rows = B * (N + M) if not cache else M
    for i, (a, b) in enumerate(zip(got, want)):
        a, b = a.double(), b.double()
        if i % 2 == 0:
            a, b = a[:rows], b[:rows]
        rel = (a - b).norm(dim=1) / b.norm(dim=1)
        assert rel.max() <= 2 * 2 * 3.5e-3, (i, rel.max())


def test_repeats_bit_for_bit(monkeypatch):
    """Which CTA adds a K split's part varies, the order of the adds does not."""
    first, _ = _forward(monkeypatch, "", 128, 160, 384, 1, 0, 100)
    for _ in range(5):
        again, _ = _forward(monkeypatch, "", 128, 160, 384, 1, 0, 100)
        assert all(torch.equal(a, b) for a, b in zip(first, again))
