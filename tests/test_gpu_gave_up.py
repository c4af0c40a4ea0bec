"""A bounded wait of the radix sort that gives up: calls that wait for the device
report it.  The waits are told to give up at the first look that fails, so the
sorts they belong to lose keys; every access stays inside its buffers."""
from __future__ import annotations

import ctypes
import time

import pytest

import synth

pytestmark = pytest.mark.gpu
TIMEOUT = -6


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2305_05245_gb300 import _lib
    return _lib.load()


def stalled(lib):
    """Whether a wait gave up since the last look (and forget it)."""
    out, any_ = (ctypes.c_uint64 * 4)(), False
    while lib.ps_debug_violation(out) == 1:
        assert out[0] % 100 == 90, "site %d index %d bound %d cta %d" % tuple(out)  # a wait, not an index
        any_ = True
    return any_


@pytest.mark.parametrize("dtype,n,pinned", [("int32", 3000001, True), ("int64", 3000001, False), ("int32", (3 << 24) + 5, True),
                                            ("int64", (3 << 23) + 5, True)])
def test_host_keys(lib, dtype, n, pinned):
    import torch
    import paper_2305_05245_gb300 as ps
    from paper_2305_05245_gb300 import _lib
    src = synth.keys_torch(n, dtype, "uniform", seed=n)
    want = torch.sort(src)[0].cpu()
    h = torch.empty_like(src, device="cpu", pin_memory=pinned)
    seen = 0
    stalled(lib)
    assert lib.ps_debug_radix_spins(0) == 0
    try:
        for _ in range(6):
            h.copy_(src)
            try:
                ps.sort_host(h)
                status = 0
            except _lib.PsortError as e:
                status = e.status
            assert status == (TIMEOUT if stalled(lib) else 0)
            if status == 0:
                assert torch.equal(h, want)
            seen += status != 0
    finally:
        lib.ps_debug_radix_spins(-1)
    assert seen > 0
    h.copy_(src)
    ps.sort_host(h)
    assert torch.equal(h, want) and not stalled(lib)


def test_records_by_embedded_key(lib):
    """The records are gathered by positions that the sort may have lost."""
    import torch
    import paper_2305_05245_gb300 as ps
    n = 6000001
    src = synth.keys_torch(3 * n, "int64", "uniform", seed=9).view(n, 3)
    stalled(lib)
    assert lib.ps_debug_radix_spins(0) == 0
    try:
        for _ in range(6):
            x = src.clone()
            ps.sort_struct(x)
            torch.cuda.synchronize()
    finally:
        lib.ps_debug_radix_spins(-1)
    assert stalled(lib)
    x = src.clone()
    ps.sort_struct(x)
    torch.cuda.synchronize()
    key = x[:, 0] ^ torch.iinfo(torch.int64).min
    assert bool((key[1:] >= key[:-1]).all()) and not stalled(lib)


@pytest.mark.parametrize("dtype", ["int32", "int64"])
def test_server_requests(lib, dtype):
    import torch
    import paper_2305_05245_gb300 as ps
    src = synth.keys_torch(3000001, dtype, "uniform", seed=5)
    want = torch.sort(src)[0]
    stalled(lib)
    srv = ps.Server(budget_bytes=4 << 30)
    x, seen = src.clone(), 0

    def once():
        x.copy_(src)
        torch.cuda.synchronize()
        rid = srv.submit(x)
        t0 = time.time()
        while time.time() - t0 < 30:
            for r, status in srv.poll():
                assert r == rid
                return status
        raise AssertionError("the request did not finish")

    assert lib.ps_debug_radix_spins(0) == 0
    try:
        for _ in range(6):
            status = once()
            torch.cuda.synchronize()
            assert status == (TIMEOUT if stalled(lib) else 0)
            seen += status != 0
    finally:
        lib.ps_debug_radix_spins(-1)
    assert seen > 0
    assert once() == 0 and torch.equal(x, want) and not stalled(lib)
    srv.close()
