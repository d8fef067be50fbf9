"""The attention's CTAs walk the units of the rows there are: at most one CTA per SM whatever a
launch may have to hold, and the same results as a forward that computes every row.

Batches of more than 32 sequences (the units are found 32 sequences at a time), under the dual cache
with the current block of each, some sequences finished, heads of 64 and of 128, grouped or not.  The
state does not change between the steps, so the keys and values that a block step reads from the
refresh are a full forward's: both lie within 3.5e-3 relative rms per row and block of the 64-bit
forward (the teacher-forced bound), and differ by at most twice that per block."""
import json
import os

import numpy as np
import pytest
import torch

import synthetic as syn

pytestmark = pytest.mark.gpu

MODELS = {64: dict(d=768, H=12, G=4, F=1024), 128: dict(d=512, H=4, G=4, F=1536)}


def _context(hd, B, T):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as dcl
    m = MODELS[hd]
    c = dcl.Context(syn.ModelShape(2, m["d"], m["H"], m["G"], hd, m["F"], 4096, 4095, 1e4), max_batch=B, max_seq=T)
    c.init_random_weights(7, 0.02, 2.0, 0.1)
    return dcl, c


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("B,N,M", [(40, 64, 256), (70, 32, 96)])
def test_block_steps_of_many_sequences(hd, B, N, M):
    x, p = syn.decode_state(3, syn.prompt_ids(3, B, N, 4095), M, 0, M // 2, 4095)
    p = (N + (37 * np.arange(B)) % M).astype(np.int32)
    done = np.arange(B) % 5 == 3
    p[done] = N + M
    blocks = [(b, N + 32 * ((int(p[b]) - N) // 32)) for b in range(B) if not done[b]]
    got = []
    for cache in (2, 0):
        dcl, c = _context(hd, B, N + M)
        with c:
            c.set_prompt(x[:, :N], dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M, kv_cache=cache))
            c.set_state(x, p)
            for _ in range(2 if cache else 1):  # the refresh, then the blocks
                c.step()
            h = torch.zeros(B * (N + M), MODELS[hd]["d"], device="cuda")
            c.forward_debug()
            c.debug_hidden(1, h)
            if cache:  # rows: the live sequences' blocks, in order
                got.append(h[:32 * len(blocks)])
            else:      # the live sequences, all their positions
                full = h[:len(blocks) * (N + M)].view(len(blocks), N + M, -1)
                got.append(torch.cat([full[i, s:s + 32] for i, (_, s) in enumerate(blocks)]))
    a, b = (t.double() for t in got)
    rel = (a - b).norm(dim=1) / b.norm(dim=1)
    assert rel.max() <= 2 * 2 * 3.5e-3, rel.max()


def test_no_empty_ctas(tmp_path):
    """The current blocks of eight sequences, laid out beside refreshes of all their rows."""
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):  # (the first one records nothing)
        torch.zeros(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    B, N, M = 8, 256, 512
    dcl, c = _context(128, B, N + M)
    with c:
        x, p = syn.decode_state(3, syn.prompt_ids(3, B, N, 4095), M, 70, M // 2, 4095)
        c.set_prompt(x[:, :N], dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M, kv_cache=2))
        c.set_state(x, p)
        c.step(return_k=True)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            c.forward_debug()
            torch.cuda.synchronize()
    path = os.path.join(tmp_path, "trace.json")
    prof.export_chrome_trace(path)
    with open(path) as f:
        grids = [e["args"]["grid"][0] for e in json.load(f)["traceEvents"]
                 if e.get("cat") == "kernel" and "attn_tc" in e["name"]]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert len(grids) == 2 and max(grids) <= sms, grids
