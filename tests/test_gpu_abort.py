"""A GEMM of the step whose ordered adds wait for a counter that nothing signals: the wait runs
out after its limit (2 s), every warp of every CTA leaves, the call returns DCL_ERR_TIMEOUT, and
the next step on the same context gives the bits of an undisturbed one.

The counters are set to -1000 through the context's allocator: dcl_set_prompt allocates the row
table, then the counters.  (With epilogue threads that each left their loop on their own wait, some
could be left at a barrier that the others never reach: this test must not be run on such code.)"""
import ctypes
import time

import numpy as np
import pytest
import torch

import synthetic as syn

pytestmark = pytest.mark.gpu


def _context(dcl, shape, batch, seq, blocks):
    """A dcl.Context whose device buffers are torch tensors, listed in `blocks` as allocated."""
    def alloc(n, _):
        blocks.append(torch.zeros(n, dtype=torch.uint8, device="cuda"))
        return blocks[-1].data_ptr()

    cbs = (ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(alloc),
           ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(lambda p, _: None))
    table = dcl.Allocator(*(ctypes.cast(f, ctypes.c_void_p) for f in cbs), None)
    cfg, out = dcl.model_config(shape), ctypes.c_void_p()
    assert dcl.lib().dcl_create(ctypes.byref(cfg), batch, seq, None, ctypes.byref(table), ctypes.byref(out)) == dcl.DCL_OK
    c = dcl.Context.__new__(dcl.Context)
    c._L, c.shape, c.stream, c.ptr, c._callbacks = dcl.lib(), shape, None, out.value, cbs
    return c


@pytest.mark.parametrize("override,N,M", [("", 160, 384),            # mid-row GEMMs: the down projection's K splits
                                          ("qkv=pair:1", 256, 256)])  # CTA-pair GEMMs: the fused MLP
def test_a_counter_that_nothing_signals(monkeypatch, override, N, M):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as dcl
    monkeypatch.setenv("DCL_GEMM_TILES", override)
    shape = syn.ModelShape(1, 4096, 32, 32, 128, 12288, 4096, 4095, 1e4)
    x, p = syn.decode_state(3, syn.prompt_ids(3, 1, N, 4095), M, 100, M // 2, 4095)
    blocks = []
    with _context(dcl, shape, 1, N + M, blocks) as c:
        c.init_random_weights(7, 0.02, 1.0, 0.1)
        n0 = len(blocks)
        c.set_prompt(x[:, :N], dcl.decode_config(tau_commit=1.0, tau_draft=1.0, min_commit=0, gen_len=M))
        counters = blocks[n0 + 1].view(torch.int32)

        def step():
            c.set_state(x, p)
            c.step(return_k=True)
            h, p1 = torch.zeros(N + M, 4096, device="cuda"), torch.zeros(1, M, device="cuda")
            c.forward_debug(p1=p1)
            c.debug_hidden(0, h)
            return h, p1

        want = step()
        assert int(counters.abs().max()) == 0  # (every launch leaves them so)
        counters.fill_(-1000)
        t = time.perf_counter()
        with pytest.raises(dcl.DcleapError) as e:
            c.set_state(x, p)
            c.step(return_k=True)
        assert e.value.status == dcl.DCL_ERR_TIMEOUT
        assert 1.5 < time.perf_counter() - t < 60
        assert all(torch.equal(a, b) for a, b in zip(step(), want))
        assert int(counters.abs().max()) == 0
