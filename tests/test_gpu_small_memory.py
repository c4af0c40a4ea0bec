"""Sorts whose radix workspace does not fit the device while the merges' does: the
device is limited (on the host) to what the merges take."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    assert torch.cuda.is_available()
    return ps


def limited(limit, f):
    """Runs f under the limit; the names of its kernels, or None for no memory."""
    import torch
    from paper_2305_05245_gb300 import _lib
    lib = _lib.load()
    lib.ps_profile_reset()
    lib.ps_profile_enable(1)
    assert lib.ps_debug_limit_alloc(limit) == 0
    try:
        f()
        torch.cuda.synchronize()
        st, n = (_lib.PsKernelStat * 64)(), ctypes.c_int()
        assert lib.ps_profile_read(st, 64, ctypes.byref(n)) == 0
        return {st[i].name.decode() for i in range(n.value)}
    except _lib.PsortError as e:
        assert e.status == -3
        return None
    finally:
        lib.ps_debug_limit_alloc(0)
        lib.ps_profile_enable(0)
        lib.ps_profile_reset()


def bounds(ps, n, code):
    """Workspace of the merges and of the automatic sort."""
    nb, np_ = ps.resolve_params(n, code)
    return ps.workspace_bytes(n, code, nb, np_), ps.workspace_bytes(n, code)


@pytest.mark.parametrize("dtype,code,n", [("int32", 0, (1 << 22) + 5), ("float32", 2, 9000001), ("int64", 1, (1 << 21) + 5),
                                          ("float64", 3, (1 << 24) + 1)])
def test_keys(ps, ora, dtype, code, n):
    import torch
    host = synth.keys(n, dtype, "uniform", seed=n)
    merges, radix = bounds(ps, n, code)
    assert merges < radix
    x = torch.from_numpy(host.copy()).cuda()
    used = limited(merges, lambda: ps.sort(x))
    assert used is not None and "radix_pass" not in used
    assert x.cpu().numpy().tobytes() == ora.reference_sort(host).tobytes()
    x.copy_(torch.from_numpy(host))
    assert limited(host.nbytes, lambda: ps.sort(x)) is None  # every way needs tables besides a copy of the keys
    assert x.cpu().numpy().tobytes() == host.tobytes()
    assert "radix_pass" in limited(radix, lambda: ps.sort(x))


@pytest.mark.parametrize("n", [(1 << 20) + 1, (1 << 24) + 1])
def test_records(ps, n):
    import torch
    merges, radix = bounds(ps, n, -1)
    assert merges < radix
    z = synth.splitmix64(n, n)
    k, p = torch.from_numpy((z >> np.uint64(2)).view(np.int64)).cuda(), torch.arange(n, dtype=torch.int32, device="cuda")
    want, order = torch.sort(k, stable=True)
    used = limited(merges, lambda: ps.sort_pairs(k, p))
    assert used is not None and "radix_pass" not in used
    assert torch.equal(k, want) and torch.equal(p.long(), order)


@pytest.mark.parametrize("dtype", ["int32", "int64"])
def test_batch(ps, dtype):
    """From a limit that the radix run fits down to one that nothing does."""
    import torch
    lens = [600000, 500, 1 << 20, 300001, 9000, 20000]
    off = torch.tensor([0] + list(np.cumsum(lens)), device="cuda")
    src = synth.keys_torch(sum(lens), dtype, "uniform", seed=4)
    want = torch.cat([torch.sort(s)[0] for s in torch.split(src, lens)])
    full = src.numel() * src.element_size()
    ways = []
    for percent in range(160, 90, -1):
        x = src.clone()
        used = limited(full * percent // 100, lambda: ps.sort_batch(x, off))
        ways.append("no memory" if used is None else "radix" if "radix_pass" in used else "merges")
        if used is not None:
            assert torch.equal(x, want)
    order = [w for i, w in enumerate(ways) if i == 0 or w != ways[i - 1]]
    assert order == ["radix", "merges", "no memory"], order
