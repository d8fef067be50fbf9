"""Scratch of the single-kernel calls: up to 256 MB stays with the context, larger belongs to the
call, and what is kept gives way to an allocation that would fail beside it.  Seen through the
context's allocator; the results are compared with those of a context without one."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
MB = 1 << 20


class Pool:
    """Device blocks as torch tensors, at most `budget` bytes at a time."""

    def __init__(self, dcl, budget):
        self.blocks, self.budget = {}, budget
        self.callbacks = (ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(self.alloc),
                          ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(self.free))
        self.table = dcl.Allocator(*(ctypes.cast(f, ctypes.c_void_p) for f in self.callbacks), None)

    def held(self):
        return sum(t.numel() for t in self.blocks.values())

    def alloc(self, n, _):
        if self.held() + n > self.budget:
            return None
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        self.blocks[t.data_ptr()] = t
        return t.data_ptr()

    def free(self, ptr, _):
        del self.blocks[ptr]

    def context(self, dcl):
        out = ctypes.c_void_p()
        assert dcl.lib().dcl_create(None, 1, 1, None, ctypes.byref(self.table), ctypes.byref(out)) == dcl.DCL_OK
        c = dcl.Context.__new__(dcl.Context)
        c._L, c.shape, c.stream, c.ptr = dcl.lib(), None, None, out.value
        return c


def _attention(c, B, seed, heads=32, T=1000):
    """32 query rows of each of B sequences: B * 8 MB of scratch (v transposed)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    qkv = torch.randn(B * T, 3 * heads * 128, generator=g, device="cuda", dtype=torch.bfloat16)
    out = torch.zeros(B * T, heads * 128, dtype=torch.bfloat16, device="cuda")
    c.op_attention(qkv, out, B, T, heads, heads, 128, 32)
    return out


def test_kept_up_to_a_limit():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as dcl
    pool = Pool(dcl, 1 << 40)
    with pool.context(dcl) as c, dcl.Context() as plain:
        start = pool.held()
        for B, kept in ((2, 2), (4, 4), (3, 4), (36, 4), (1, 4)):  # (36: 281 MB, the call's own)
            assert torch.equal(_attention(c, B, B), _attention(plain, B, B))
            assert pool.held() - start == kept * 1000 * 32 * 128 * 2
    assert pool.held() == 0


def test_gives_way():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_20467_gb300 as dcl
    pool = Pool(dcl, 350 * MB)
    with pool.context(dcl) as c, dcl.Context() as plain:
        for B in (30, 36, 30):  # 234 MB kept, 281 MB not beside it, and again
            assert torch.equal(_attention(c, B, B), _attention(plain, B, B))
        with pytest.raises(dcl.DcleapError) as e:
            _attention(c, 50, 1)
        assert e.value.status == dcl.DCL_ERR_OOM
        assert torch.equal(_attention(c, 2, 2), _attention(plain, 2, 2))
    assert pool.held() == 0
