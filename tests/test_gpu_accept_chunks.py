"""The acceptance pass's statistics, taken in chunks of a row's 16-byte vectors, where the split
can go wrong: rows that are not 16-byte aligned, fewer columns than a vector, one vector more or
less than a chunk, whole chunks of -inf or of the type's lowest value, the maximum at a chunk's
edge or tied across chunks, with the most chunks (one block) and with one (many rows).

Every row's confidence is 0.99 or 0.3 by construction (the other columns share the rest), far
from the threshold 0.7, so that ids and run lengths are exact whatever the order of the sums."""
import numpy as np
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


def _logits(rng, rows, V, fill):
    """[rows][V] bf16 logits: 64 live columns, the rest `fill`; the top column, its share."""
    z = np.full((rows, V), fill, np.float32)
    top = np.empty(rows, np.int64)
    sure = rng.random(rows) < 0.6
    for r in range(rows):
        edge = rng.choice([0, V - 1, 7, 8, 2047, 2048, V // 2])
        top[r] = edge if edge < V else V - 1
        live = np.unique(np.append(rng.integers(0, V, size=min(64, V)), top[r]))
        n = len(live) - 1
        share = 0.99 if sure[r] else 0.3
        if n == 0:
            sure[r] = True
        z[r, live] = 0.0
        # the rest: n columns of weight 1 each; the top's weight n * share / (1 - share)
        z[r, top[r]] = np.log(max(n, 1) * share / (1 - share)) if n else 0.0
        if not sure[r] and z[r, top[r]] <= 0.5:  # (too few columns for a share below the threshold)
            z[r, top[r]], sure[r] = 12.0, True
    return torch.from_numpy(z).to(torch.bfloat16).cuda(), top, sure


@pytest.mark.parametrize("confidence", [0, 1])
@pytest.mark.parametrize("fill", [-np.inf, -3.3895e38])
@pytest.mark.parametrize("B,P,V", [(1, 7, 126464), (1, 5, 126461), (2, 9, 2048), (2, 9, 2055), (2, 9, 4103), (3, 4, 9),
                                   (1, 1, 2), (40, 33, 1003), (257, 3, 2051), (1300, 32, 129)])
def test_chunks(ops, B, P, V, fill, confidence):
    import paper_2607_20467_gb300 as dcl
    rng = np.random.default_rng(B * 7919 + V)
    z, top, sure = _logits(rng, B * P, V, fill)
    committed = rng.integers(0, P, size=B).astype(np.int32)
    x0 = rng.integers(0, V, size=(B, P)).astype(np.int32)
    x, k = torch.from_numpy(x0.copy()).cuda(), torch.full((B,), -1, dtype=torch.int32, device="cuda")
    # p1 = 0.99 has exp(-H) > 0.7 (H = -0.99 ln 0.99 - 0.01 ln(0.01 / n) < 0.11 for n <= 64), 0.3 has not
    cfg = dcl.decode_config(tau_commit=0.7, tau_draft=0.7, max_window=2, gen_len=P, min_commit=1, confidence=confidence)
    ops.accept(z.view(B, P, V), torch.from_numpy(committed).cuda(), x, cfg, k)
    torch.cuda.synchronize()
    top, sure = top.reshape(B, P), sure.reshape(B, P)
    for b in range(B):
        c = int(committed[b])
        w = min(2, P - c)
        run = next((i for i in range(w) if not sure[b, c + i]), w)
        K = max(run, 1)
        want = x0[b].copy()
        want[c:c + K] = top[b, c:c + K]
        for i in range(c + 2, P):
            if sure[b, i]:
                want[i] = top[b, i]
        assert int(k[b]) == K, b
        assert (x[b].cpu().numpy() == want).all(), b


def test_lowest_column_of_a_tie_over_chunks(ops):
    """The maximum in three chunks and twice in a vector: its lowest column."""
    import paper_2607_20467_gb300 as dcl
    P, V = 4, 126464
    z = torch.zeros(1, P, V, device="cuda")
    cols = [(5, 6, 70000), (2047, 2048, 126463), (126462, 126463), (8191, 64000, 64001)]
    for i, c in enumerate(cols):
        z[0, i, list(c)] = 20.0
    x, k = torch.zeros(1, P, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    cfg = dcl.decode_config(tau_commit=0.2, tau_draft=1.0, max_window=P, gen_len=P)
    ops.accept(z.to(torch.bfloat16), torch.zeros(1, dtype=torch.int32, device="cuda"), x, cfg, k)
    torch.cuda.synchronize()
    assert int(k[0]) == P and x[0].tolist() == [c[0] for c in cols]
