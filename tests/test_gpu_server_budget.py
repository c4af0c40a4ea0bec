"""The server's memory budget holds what its rounds take, not only the sum of what
their requests would take alone: with the device limited to the budget (an injected
limit on the library's allocations), every request completes."""
from __future__ import annotations

import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cost(ps, n, code, size):
    return n * size + ps.workspace_bytes(n, code)


@pytest.mark.parametrize("dtype,code,size,lens", [
    ("int64", 1, 8, [140000] + [8200] * 1000),             # short ones that join the radix run of a long one
    ("int64", 1, 8, [20000] * 100 + [10000] * 60 + [40000] * 40 + [70000] * 9),
    ("int32", 0, 4, [300000] + [8200] * 1000),
    ("float64", 3, 8, [150000, 140001, 200000, 1 << 20, 300001]),
    ("int32", 0, 4, [(1 << 18) + 1] * 12),
])
def test_rounds_stay_within_the_budget(dtype, code, size, lens):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    from paper_2305_05245_gb300 import _lib
    lib = _lib.load()
    rng = np.random.default_rng(len(lens))
    dt = getattr(torch, dtype)
    host = [torch.from_numpy(rng.integers(0, 1 << 30, n)).to(dt) for n in lens]
    work = [h.cuda() for h in host]
    slack = 4096 + 32 * len(lens)  # instance tables
    budget = sum(cost(ps, n, code, size) for n in lens) + slack
    # requests that fill the budget one by one, so that the others queue up behind them
    big = budget // (2 * size) * 9 // 10
    while cost(ps, big, code, size) > budget - slack:
        big = big * 9 // 10
    ahead = [torch.randint(0, 1 << 30, (big,), dtype=torch.int32, device="cuda").to(dt) for _ in range(30)]
    torch.cuda.synchronize()
    srv = ps.Server(budget_bytes=budget, max_inflight=1 << 20)
    assert lib.ps_debug_limit_alloc(budget) == 0
    try:
        left = {srv.submit(t) for t in ahead} | {srv.submit(t) for t in work}
        t0 = time.time()
        while left and time.time() - t0 < 60:
            for rid, status in srv.poll():
                assert status == 0, status
                left.discard(rid)
    finally:
        srv.close()
        lib.ps_debug_limit_alloc(0)
    assert not left
    torch.cuda.synchronize()
    for h, w in zip(host, work):
        assert torch.equal(w.cpu(), torch.sort(h)[0])
