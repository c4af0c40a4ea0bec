"""Sorts on a device that cannot place clusters of 16 (or any) thread blocks: the
library is told so (ps_debug_max_cluster), and every call that would use them
still gives the plain definition's result."""
from __future__ import annotations

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


@pytest.fixture(params=[1, 4, 8, 16])
def cap(request, ps):
    from paper_2305_05245_gb300 import _lib
    lib = _lib.load()
    assert lib.ps_debug_max_cluster(request.param) == 0
    yield request.param
    assert lib.ps_debug_max_cluster(0) == 0


def kernels(f):
    """Names of the kernels one call launches."""
    import ctypes
    import torch
    from paper_2305_05245_gb300 import _lib
    lib = _lib.load()
    lib.ps_profile_reset()
    lib.ps_profile_enable(1)
    f()
    torch.cuda.synchronize()
    lib.ps_profile_enable(0)
    st, n = (_lib.PsKernelStat * 64)(), ctypes.c_int()
    assert lib.ps_profile_read(st, 64, ctypes.byref(n)) == 0
    lib.ps_profile_reset()
    return {st[i].name.decode() for i in range(n.value)}


@pytest.mark.parametrize("dtype", sorted(synth.DTYPES))
@pytest.mark.parametrize("n", [1000, 8192, 8193, 16384, 16385, 65536, 98304, 98305, 131072])
def test_keys(ps, ora, cap, dtype, n):
    import torch
    host = synth.keys(n, dtype, "uniform", seed=n)
    st = {"uint32": np.int32, "uint64": np.int64}.get(dtype, host.dtype)
    x = torch.from_numpy(host.view(st).copy()).cuda()
    used = kernels(lambda: ps.sort(x.view(getattr(torch, dtype))))
    assert x.cpu().numpy().tobytes() == ora.reference_sort(host).tobytes()
    if cap < 4 and n > 8192 or cap < 16 and n > 16384:
        assert "cluster_sort" not in used


@pytest.mark.parametrize("n", [8192, 8193, 16385, 65536])
def test_records(ps, cap, n):
    import torch
    z = synth.splitmix64(n, 2 * n)
    k, p = z[:n] >> np.uint64(8), (z[n:] >> np.uint64(32)).astype(np.uint32)
    tk, tp = torch.from_numpy(k.view(np.int64).copy()).cuda(), torch.from_numpy(p.view(np.int32).copy()).cuda()
    ps.sort_pairs(tk, tp)
    torch.cuda.synchronize()
    o = np.lexsort((p, k))
    assert tk.cpu().numpy().view(np.uint64).tobytes() == k[o].tobytes()
    assert tp.cpu().numpy().view(np.uint32).tobytes() == p[o].tobytes()


@pytest.mark.parametrize("dtype", ["int32", "float64"])
def test_other_calls(ps, ora, cap, dtype):
    """Given blocks, batches, pinned host keys, the allocation-free sort."""
    import torch
    host = synth.keys(90000, dtype, "uniform", seed=3)
    want = ora.reference_sort(host).tobytes()
    dev = torch.from_numpy(host.copy())
    for nb in (1, 2, 8, 40):
        x = dev.cuda()
        ps.sort(x, n_blocks=nb, n_parts=nb)
        assert x.cpu().numpy().tobytes() == want
    h = dev.pin_memory()
    ps.sort_host(h)
    assert h.numpy().tobytes() == want
    x = dev.cuda()
    ps.sort_noalloc(x)
    torch.cuda.synchronize()
    assert x.cpu().numpy().tobytes() == want
    lens = [9000, 20000, 500, 8193, 40000, 12307]
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    x = dev[:int(off[-1])].cuda()
    ps.sort_batch(x, torch.from_numpy(off).cuda())
    segs = [ora.reference_sort(host[a:b]) for a, b in zip(off[:-1], off[1:])]
    assert x.cpu().numpy().tobytes() == np.concatenate(segs).tobytes()
