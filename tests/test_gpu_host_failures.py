"""Pinned host keys when a device allocation of the call fails: the call gives
either the sorted keys or an error with the keys as they were.  Every allocation
of one call fails in turn (on the host, before any CUDA call)."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n", [("int32", (3 << 24) + 5), ("int64", (3 << 23) + 7), ("int32", 300000),
                                     ("int64", 5000)])
def test_every_allocation_fails_once(dtype, n):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    from paper_2305_05245_gb300 import _lib
    import synth
    lib = _lib.load()
    src = synth.keys_torch(n, dtype, "uniform", seed=n)
    want = torch.sort(src)[0]
    h = torch.empty_like(src, device="cpu", pin_memory=True)
    errors = 0
    for skip in range(40):
        h.copy_(src)
        assert lib.ps_debug_fail_alloc_after(skip, 1) == 0
        try:
            ps.sort_host(h)
            ok = True
        except _lib.PsortError as e:
            assert e.status == -3
            ok = False
        finally:
            lib.ps_debug_fail_alloc(0)
        assert torch.equal(h.cuda(), want if ok else src), "allocation %d failed, call %s" % (skip, "ok" if ok else "failed")
        errors += not ok
        if ok and skip >= 12:
            break
    # the buffer, and where blocks are copied in groups the table and each of four blocks' workspaces
    assert errors >= (6 if n > (1 << 24) else 1)
