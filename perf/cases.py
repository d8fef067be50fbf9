"""The cases that performance work on this library is measured on: denoise steps (full
recompute, prefix cache, dual cache) of the LLaDA-8B, Dream-7B and small shapes, the
acceptance pass on given logits, the attention and the LM head on their own.

A step case runs `dcl_generate` for a fixed number of steps from a given state and then reads
the predictions of that state.  tau_commit = tau_draft = 1 with min_commit = 0 is the literal
rule at thresholds nothing passes: the steps run whole (re-mask, forward, confidence,
acceptance) and leave the state where it is, so their work does not depend on how a near tie
rounds.  Where a trajectory's steps differ (cache modes: one refresh, then the suffix or the
current block), the state's place in the trajectory (`offset` = p - N of the first sequence)
and the number of steps give the mix.
"""
import math

import numpy as np
import torch

import paper_2607_20467_gb300 as dcl

BLOCK = 32
EXACT_FLOPS = 1.2e13  # what a 64-bit restatement may cost (about a TFLOP/s)

# layers aside: the repository's model shapes, and a small grouped-query one (two q heads of 64
# columns per 128, four kv heads)
SHAPES = {
    "tiny": dict(d=256, heads=4, kv=4, hd=64, ffn=1024, vocab=4096, theta=1e4),
    "small-gqa": dict(d=768, heads=12, kv=4, hd=64, ffn=2048, vocab=8224, theta=1e4),
    "llada8b": dict(d=4096, heads=32, kv=32, hd=128, ffn=12288, vocab=126464, theta=5e5),
    "dream7b": dict(d=3584, heads=28, kv=4, hd=128, ffn=18944, vocab=152064, theta=1e6),
}


class Shape:
    """What `dcl.Context` reads of a model shape."""

    def __init__(self, name, layers):
        s = SHAPES[name]
        self.n_layers, self.d_model, self.n_heads, self.n_kv_heads = layers, s["d"], s["heads"], s["kv"]
        self.head_dim, self.ffn_dim, self.vocab, self.mask_id = s["hd"], s["ffn"], s["vocab"], s["vocab"] - 1
        self.rope_theta, self.rms_eps = s["theta"], 1e-5


def _steps(name, shape, layers, batch, prompt, gen, offset, steps, cache=0, confidence=0, lm_scale=1.0, logits=0):
    return dict(name=name, kind="steps", shape=shape, layers=layers, batch=batch, prompt=prompt, gen=gen,
                offset=offset, steps=steps, cache=cache, confidence=confidence, lm_scale=lm_scale, logits=logits)


def listed():
    return [
        # the 2-layer test model, prompt 32 + gen 64: a step is launches and latency
        _steps("tiny-b1", "tiny", 2, 1, 32, 64, 16, 8, lm_scale=4.0, logits=1),
        # a small grouped-query model on sequences of 127 positions (no multiple of a tile or of 32)
        _steps("small-gqa-ragged", "small-gqa", 4, 3, 37, 90, 21, 4, confidence=1, lm_scale=3.0, logits=1),
        # the whole 32-layer LLaDA-8B shape, prompt 256 + gen 256, full recompute
        _steps("llada8b-b1", "llada8b", 32, 1, 256, 256, 96, 2, lm_scale=0.5, logits=1),
        # the long generation (prompt 512 + gen 1024) at batch 8, full recompute: the largest step
        _steps("llada8b-long-b8", "llada8b", 2, 8, 512, 1024, 500, 1),
        # the long generation, batch 1, prefix cache, half way: a refresh, then 544-row suffixes
        _steps("llada8b-prefix-b1", "llada8b", 8, 1, 512, 1024, 500, 8, cache=1),
        # the same near its end: suffixes of 96 rows
        _steps("llada8b-prefix-late", "llada8b", 8, 1, 512, 1024, 930, 12, cache=1),
        # the long generation, batch 1, dual cache: 32-row blocks between refreshes
        _steps("llada8b-dual-b1", "llada8b", 8, 1, 512, 1024, 300, 16, cache=2),
        # a batch of 16 under the dual cache, grouped-query heads: 512 rows a step
        _steps("dream7b-dual-b16", "dream7b", 4, 16, 384, 512, 200, 8, cache=2, confidence=1),
        # the acceptance pass of 64 blocks of 32 positions
        dict(name="accept-b64", kind="accept", batch=64, positions=32, vocab=126464, window=16, confidence=0,
             acceptance=0),
        # one sequence's block, the entropy confidence: a latency-bound call
        dict(name="accept-b1-entropy", kind="accept", batch=1, positions=32, vocab=152064, window=16, confidence=1,
             acceptance=0),
        # attention on its own, grouped-query heads, 1000 positions (no multiple of a tile)
        dict(name="attention-ragged", kind="attention", batch=4, tokens=1000, heads=28, kv=4, hd=128, q_rows=0),
        # the LM head with its softmax statistics for one block of one sequence
        dict(name="lmhead-r32", kind="lmhead", rows=32, vocab=126464, d=4096, entropy=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "steps", "accept", "attention", "lmhead"])
    if kind == "accept":
        vocab = rng.choice([126464, 152064, 32000, _log(rng, 1000, 150000)])
        return dict(kind="accept", batch=_log(rng, 1, 64), positions=_log(rng, 4, 40), vocab=vocab,
                    window=rng.choice([0, 16, 32]), confidence=rng.randint(0, 1), acceptance=int(rng.random() < 0.25))
    if kind == "attention":
        heads, kv, hd = rng.choice([(32, 32, 128), (28, 4, 128), (4, 4, 64), (12, 4, 64)])
        tokens = _log(rng, 64, 1800)
        q_rows = 32 * rng.randint(1, tokens // 32) if rng.random() < 0.5 else 0
        return dict(kind="attention", batch=_log(rng, 1, 8), tokens=tokens, heads=heads, kv=kv, hd=hd, q_rows=q_rows)
    if kind == "lmhead":
        d, vocab = rng.choice([(4096, 126464), (3584, 152064), (256, 4096), (768, _log(rng, 1000, 60000))])
        return dict(kind="lmhead", rows=_log(rng, 1, 1024), vocab=vocab, d=d, entropy=rng.randint(0, 1))
    shape = rng.choice(["tiny", "small-gqa", "llada8b", "llada8b", "dream7b", "dream7b"])
    small = shape in ("tiny", "small-gqa")
    cache = rng.choice([0, 1, 2])
    layers = rng.randint(1, 4)
    batch = _log(rng, 1, 16)
    most = max(96, min(1536, (9000 if small else 12288 // layers) // batch))
    prompt, gen = _log(rng, 17, most // 2), _log(rng, 33, most // 2)
    if cache:
        prompt, gen = max(32, prompt // 32 * 32), max(32, gen // 32 * 32)
    return dict(kind="steps", shape=shape, layers=layers, batch=batch, prompt=prompt, gen=gen,
                offset=rng.randrange(gen), steps=rng.randint(2, 8) if cache else rng.randint(1, 3), cache=cache,
                confidence=rng.randint(0, 1), lm_scale={"tiny": 4.0, "small-gqa": 3.0}.get(shape, 1.0),
                logits=int(not cache and batch * gen <= 1024))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, n, std, mean=0.0):
    out = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    for a in range(0, n, 1 << 28):
        m = min(1 << 28, n - a)
        out[a:a + m] = torch.randn(m, generator=g, device="cuda").mul_(std).add_(mean)
    return out


def _weights(case, seed):
    """(kind, layer, bf16 tensor) of every weight, in the order a forward uses them."""
    s, g = Shape(case["shape"], case["layers"]), _gen(seed)
    yield dcl.DCL_W_EMBED, 0, _draw_weight(case, s, g, dcl.DCL_W_EMBED)
    for layer in range(s.n_layers):
        for kind in range(dcl.DCL_W_ATTN_NORM, dcl.DCL_W_DOWN + 1):
            yield kind, layer, _draw_weight(case, s, g, kind)
    for kind in (dcl.DCL_W_FINAL_NORM, dcl.DCL_W_LM_HEAD):
        yield kind, 0, _draw_weight(case, s, g, kind)


def _draw_weight(case, s, g, kind):
    n = dcl.weight_elements(s, kind)
    if kind in (dcl.DCL_W_ATTN_NORM, dcl.DCL_W_MLP_NORM, dcl.DCL_W_FINAL_NORM):
        return _normal(g, n, 0.1, 1.0)
    return _normal(g, n, 0.02 * (case["lm_scale"] if kind == dcl.DCL_W_LM_HEAD else 1.0))


def _offsets(case):
    """p - N of every sequence: a batch's sequences are at different places."""
    return [(case["offset"] + 37 * b) % case["gen"] for b in range(case["batch"])]


def _rows(case):
    """Positions [start, end) of every sequence that a step computes (after a refresh)."""
    N, T = case["prompt"], case["prompt"] + case["gen"]
    if not case["cache"]:
        return [(0, T)] * case["batch"]
    starts = [N + BLOCK * (o // BLOCK) for o in _offsets(case)]
    return [(a, T if case["cache"] == 1 else min(a + BLOCK, T)) for a in starts]


def _state(case, seed):
    """x and p: the prompt, committed ids up to p, MASK on the window, drafts on 0.4 of what follows."""
    r = np.random.default_rng(seed)
    N, M, B, mask = case["prompt"], case["gen"], case["batch"], SHAPES[case["shape"]]["vocab"] - 1
    x = r.integers(0, mask, size=(B, N + M)).astype(np.int32)
    p = np.array([N + o for o in _offsets(case)], np.int32)
    free = r.random((B, N + M)) >= 0.4
    for b in range(B):
        x[b, p[b]:][free[b, p[b]:]] = mask
        x[b, p[b]:p[b] + max(1, M // 2)] = mask
    return x, p


_OPS = []


def _ops():
    """The one ops context a program keeps for its single-kernel calls."""
    if not _OPS:
        _OPS.append(dcl.Context())
    return _OPS[0]


def _accept_inputs(case, seed):
    g, r = _gen(seed), np.random.default_rng(seed)
    B, P, V = case["batch"], case["positions"], case["vocab"]
    # top-1 probabilities: half in 0.65 .. 0.9, a quarter above, a quarter below
    comp = r.choice(3, size=(B, P), p=[0.5, 0.25, 0.25])
    q = np.array([0.65, 0.90, 0.05])[comp] + np.array([0.25, 0.0999, 0.60])[comp] * r.beta(2.0, 2.0, size=(B, P))
    lift = torch.from_numpy(np.log(q / (1.0 - q))).cuda()
    top = torch.from_numpy(r.integers(0, V, size=(B, P))).cuda()
    logits = torch.empty(B, P, V, dtype=torch.bfloat16, device="cuda")
    for b in range(B):
        z = torch.randn(P, V, generator=g, device="cuda")
        z.scatter_(1, top[b][:, None], -math.inf)
        rest = torch.logsumexp(z, 1).double()
        z.scatter_(1, top[b][:, None], (lift[b] + rest).float()[:, None])
        logits[b] = z
    committed = r.integers(0, P + 1, size=B) if B > 1 else np.zeros(1, np.int64)
    x = r.integers(0, V - 1, size=(B, P))
    x[(r.random((B, P)) < 0.5) & (np.arange(P)[None] >= committed[:, None])] = V - 1
    to = lambda a: torch.from_numpy(a.astype(np.int32)).cuda()  # noqa: E731
    return logits, to(committed), to(x)


def _attention_input(case, seed):
    n = case["batch"] * case["tokens"] * (case["heads"] + 2 * case["kv"]) * case["hd"]
    return _normal(_gen(seed), n, 1.0).view(case["batch"] * case["tokens"], -1)


def _lmhead_inputs(case, seed):
    g = _gen(seed)
    w = _normal(g, case["vocab"] * case["d"], 0.24 * math.sqrt(4096 / case["d"]) / 2).view(case["vocab"], -1)
    return _normal(g, case["rows"] * case["d"], 1.0).view(case["rows"], -1), w


def prepare(case, seed):
    out = lambda *s: torch.zeros(*s, device="cuda")  # noqa: E731
    if case["kind"] == "accept":
        logits, committed, x = _accept_inputs(case, seed)
        cfg = dcl.decode_config(max_window=case["window"], confidence=case["confidence"], acceptance=case["acceptance"])
        return dict(case=case, ctx=_ops(), logits=logits, committed=committed, x=x, cfg=cfg,
                    k=torch.zeros(case["batch"], dtype=torch.int32, device="cuda"))
    if case["kind"] == "attention":
        qkv = _attention_input(case, seed)
        return dict(case=case, ctx=_ops(), qkv=qkv, out=torch.zeros(
            len(qkv), case["heads"] * case["hd"], dtype=torch.bfloat16, device="cuda"))
    if case["kind"] == "lmhead":
        x, w = _lmhead_inputs(case, seed)
        R = case["rows"]
        return dict(case=case, ctx=_ops(), x=x, w=w, top1=torch.zeros(R, dtype=torch.int32, device="cuda"), p1=out(R),
                    p2=out(R), entropy=out(R) if case["entropy"] else None)
    shape = Shape(case["shape"], case["layers"])
    B, N, M = case["batch"], case["prompt"], case["gen"]
    ctx = dcl.Context(shape, max_batch=B, max_seq=N + M)
    for kind, layer, w in _weights(case, seed):
        ctx.set_weight(kind, layer, w)
    x, p = _state(case, seed)
    ctx.set_prompt(x[:, :N], dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, block_len=BLOCK, gen_len=M,
                                               kv_cache=case["cache"], confidence=case["confidence"]))
    return dict(case=case, ctx=ctx, x=x, p=p, hidden=out(B * (N + M), shape.d_model), p1=out(B, M), p2=out(B, M),
                conf=out(B, M), entropy=out(B, M),
                logits=torch.zeros(B, M, shape.vocab, dtype=torch.bfloat16, device="cuda") if case["logits"] else None)


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "accept":
        ctx.accept(state["logits"], state["committed"], state["x"], state["cfg"], state["k"])
        return dict(x=state["x"], k=state["k"])
    if case["kind"] == "attention":
        ctx.op_attention(state["qkv"], state["out"], case["batch"], case["tokens"], case["heads"], case["kv"], case["hd"],
                         case["q_rows"])
        return state["out"].view(case["batch"], case["tokens"], -1)[:, -case["q_rows"]:]
    if case["kind"] == "lmhead":
        ctx.op_lmhead_top2(state["x"], state["w"], state["top1"], state["p1"], state["p2"], entropy=state["entropy"])
        return {k: state[k] for k in ("top1", "p1", "p2", "entropy")}
    ctx.set_state(state["x"], state["p"])
    tokens, _, status = ctx.generate(max_steps=case["steps"], check=False)
    if status not in (dcl.DCL_OK, dcl.DCL_ERR_TIMEOUT):  # (a state that does not advance uses up its steps)
        raise RuntimeError(f"generate: status {status}")
    preds = {k: state[k] for k in ("p1", "p2", "conf", "entropy")}
    ctx.forward_debug(logits=state["logits"], **preds)
    ctx.debug_hidden(case["layers"] - 1, state["hidden"])
    computed = sum(b - a for a, b in _rows(case))
    return dict(tokens=tokens, hidden=state["hidden"][:computed], logits=state["logits"], **preds)


# ---------------------------------------------------------------- work and tolerance
def work(case):
    if case["kind"] == "accept":
        # (the committed counts are drawn: half of the positions are read, all of a single block's)
        n = case["positions"] * (case["batch"] / 2 if case["batch"] > 1 else 1)
        return dict(bytes=2.0 * n * case["vocab"], flops=0)
    if case["kind"] == "attention":
        T, rows = case["tokens"], case["q_rows"] or case["tokens"]
        per_token = (case["heads"] + 2 * case["kv"]) * case["hd"]
        return dict(bytes=2.0 * case["batch"] * (T * per_token + rows * case["heads"] * case["hd"]),
                    flops=4.0 * case["batch"] * case["heads"] * rows * T * case["hd"])
    if case["kind"] == "lmhead":
        return dict(bytes=2.0 * case["d"] * (case["vocab"] + case["rows"]),
                    flops=2.0 * case["rows"] * case["vocab"] * case["d"])
    s = Shape(case["shape"], case["layers"])
    N, T, B = case["prompt"], case["prompt"] + case["gen"], case["batch"]
    d, hd, H, G, F = s.d_model, s.head_dim, s.n_heads, s.n_kv_heads, s.ffn_dim
    layer = (H + 2 * G) * hd * d + H * hd * d + 3 * F * d
    nbytes = flops = 0.0
    for i in range(case["steps"] + 1):
        spans = _rows(case) if i or not case["cache"] else [(0, T)] * B
        rows = sum(b - a for a, b in spans)
        nbytes += 2.0 * (s.n_layers * layer + s.vocab * d) + 2.0 * rows * d
        flops += _forward_flops(s, spans, N, T)
        if rows < B * T:  # the stored keys and values
            nbytes += 4.0 * s.n_layers * B * T * G * hd
    nbytes += 8.0 * d * rows  # the residual stream that is read out
    if case["logits"]:
        nbytes += 2.0 * s.vocab * (d + B * case["gen"])
        flops += 2.0 * B * case["gen"] * s.vocab * d
    return dict(bytes=nbytes, flops=flops)


def _forward_flops(s, spans, N, T):
    """Of one forward over positions [a, b) of each sequence, LM head on those from N on."""
    d, hd, H, G, F = s.d_model, s.head_dim, s.n_heads, s.n_kv_heads, s.ffn_dim
    rows, lm = sum(b - a for a, b in spans), sum(b - max(a, N) for a, b in spans)
    layer = (H + 2 * G) * hd * d + H * hd * d + 3 * F * d
    return 2.0 * rows * s.n_layers * layer + 4.0 * rows * T * H * hd * s.n_layers + 2.0 * lm * s.vocab * d


def tolerance(case):
    if case["kind"] == "accept":
        return "exact"  # ids and run lengths: whole numbers
    if case["kind"] == "attention":
        return dict(rel=7e-3)  # bf16 output, probabilities in 16 bits
    if case["kind"] == "lmhead":
        return dict(rel=1e-4, differ=0.01)  # 32-bit sums of up to 4096 products, logits of a few tens
    # bf16 operands: a rounding that falls the other way in one layer travels through those that
    # follow, and a logit's change is a probability's relative change
    return dict(rel=3e-2, max=0.9)


# ---------------------------------------------------------------- the same in 64 bits
def _stats(z):
    """top-1 id, p1, p2 and the entropy of logits z (float64 [rows][vocab])."""
    logp = torch.log_softmax(z, 1)
    two, ids = logp.topk(2, 1)
    return ids[:, 0].to(torch.int32), two[:, 0].exp(), two[:, 1].exp(), -(logp.exp() * logp).sum(1)


def _exact_forward(case, seed):
    s = Shape(case["shape"], case["layers"])
    N, M, B = case["prompt"], case["gen"], case["batch"]
    T, d, hd, H, G, F, V = N + M, s.d_model, s.head_dim, s.n_heads, s.n_kv_heads, s.ffn_dim, s.vocab
    x, p = _state(case, seed)
    for b in range(B):
        x[b, p[b]:p[b] + max(1, M // 2)] = s.mask_id
    ids = torch.from_numpy(x.astype(np.int64)).cuda().view(-1)
    ang = torch.arange(T, device="cuda", dtype=torch.float64)[:, None] * torch.tensor(
        [s.rope_theta ** (-2.0 * j / hd) for j in range(hd // 2)], device="cuda", dtype=torch.float64)[None]
    cos, sin = ang.cos()[None, :, None], ang.sin()[None, :, None]

    def rope(v):
        a, b = v[..., :hd // 2], v[..., hd // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

    def norm(h, w):
        return h * torch.rsqrt(h.square().mean(1, keepdim=True) + s.rms_eps) * w.double()

    h, have, hidden = None, {}, None
    for kind, layer, w in _weights(case, seed):
        if kind == dcl.DCL_W_EMBED:
            h = w.view(V, d)[ids].double()
            continue
        if kind == dcl.DCL_W_FINAL_NORM:
            hidden, have["final"] = h, w
            continue
        if kind == dcl.DCL_W_LM_HEAD:
            hn = norm(h.view(B, T, d)[:, N:].reshape(B * M, d), have["final"])
            lm = w.view(V, d).double()
            z = torch.cat([hn[a:a + 512] @ lm.T for a in range(0, B * M, 512)])
            break
        have[kind] = w
        if kind != dcl.DCL_W_DOWN:
            continue
        mat = lambda k, rows: have[k].view(rows, -1).double().T  # noqa: E731
        hn = norm(h, have[dcl.DCL_W_ATTN_NORM])
        q = rope((hn @ mat(dcl.DCL_W_Q, H * hd)).view(B, T, H, hd))
        k = rope((hn @ mat(dcl.DCL_W_K, G * hd)).view(B, T, G, hd)).repeat_interleave(H // G, 2)
        v = (hn @ mat(dcl.DCL_W_V, G * hd)).view(B, T, G, hd).repeat_interleave(H // G, 2)
        att = torch.empty_like(q)
        for b in range(B):
            a = torch.softmax(torch.einsum("thd,shd->hts", q[b], k[b]) / math.sqrt(hd), -1)
            att[b] = torch.einsum("hts,shd->thd", a, v[b])
        h = h + att.reshape(B * T, H * hd) @ mat(dcl.DCL_W_O, d)
        hn = norm(h, have[dcl.DCL_W_MLP_NORM])
        gate, up = hn @ mat(dcl.DCL_W_GATE, F), hn @ mat(dcl.DCL_W_UP, F)
        h = h + (torch.nn.functional.silu(gate) * up) @ mat(dcl.DCL_W_DOWN, d)
    rows = torch.cat([torch.arange(b * T + a, b * T + e, device="cuda") for b, (a, e) in enumerate(_rows(case))])
    return x, hidden[rows], z.view(B, M, V)


def exact(case, seed):
    if case["kind"] == "accept":
        return None  # whole numbers
    if case["kind"] == "steps":
        T = case["prompt"] + case["gen"]
        flops = _forward_flops(Shape(case["shape"], case["layers"]), [(0, T)] * case["batch"], case["prompt"], T)
    else:
        flops = work(case)["flops"]
    if flops > EXACT_FLOPS:
        return None
    if case["kind"] == "attention":
        B, T, H, G, hd = (case[k] for k in ("batch", "tokens", "heads", "kv", "hd"))
        qkv = _attention_input(case, seed).view(B, T, H + 2 * G, hd)
        out = []
        for b in range(B):
            q, k, v = (qkv[b, :, i:j].double() for i, j in ((0, H), (H, H + G), (H + G, H + 2 * G)))
            k, v = k.repeat_interleave(H // G, 1), v.repeat_interleave(H // G, 1)
            a = torch.softmax(torch.einsum("thd,shd->hts", q[-case["q_rows"]:], k) / math.sqrt(hd), -1)
            out.append(torch.einsum("hts,shd->thd", a, v).reshape(-1, H * hd))
        return torch.stack(out)
    if case["kind"] == "lmhead":
        x, w = _lmhead_inputs(case, seed)
        w = w.double()
        parts = [_stats(x[a:a + 256].double() @ w.T) for a in range(0, case["rows"], 256)]
        top1, p1, p2, entropy = (torch.cat(t) for t in zip(*parts))
        return dict(top1=top1, p1=p1, p2=p2, entropy=entropy if case["entropy"] else None)
    x, hidden, z = _exact_forward(case, seed)
    B, M = case["batch"], case["gen"]
    _, p1, p2, entropy = (t.view(B, M) for t in _stats(z.view(B * M, -1)))
    conf = torch.exp(-entropy) if case["confidence"] else p1
    return dict(tokens=x[:, case["prompt"]:], hidden=hidden, logits=z if case["logits"] else None, p1=p1, p2=p2,
                conf=conf, entropy=entropy)
